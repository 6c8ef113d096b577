// Pair sums by hit masks: the gather kernels' path for cells of few particles.
//
// In a near-uniform field only 15 % of a chaining-mesh cell's candidate pairs
// lie inside the cutoff, so a loop over all candidates spends most of its
// issue slots on pairs that add nothing.  Here a warp first finds the pairs
// near or inside the cutoff with the tensor cores and then evaluates only
// those:
//   1. the j records of up to HITS_RECS candidates are staged in shared memory,
//      shifted into the frame of the i cell, with n_j = (1 - delta) |x_j|^2;
//   2. per 8 j and 16 i one mma.m16n8k8 (tf32) forms
//      n_i + n_j - 2 x_i.x_j - (cut squared), whose sign bits are shifted into
//      one 32-bit mask per (i, column of the 8);
//   3. the masks are transposed so that every lane owns one i (with at most 16
//      i, two lanes share one), the i's own record is taken out, and each lane
//      walks its own set bits: one 16-byte shared load and one pair term per
//      bit, in the arithmetic and with the cutoff test of the dense loops.  (A
//      pair of a particle with itself would add 0 f(0) and 0 f'(0): NaN once the
//      softening is so small that these overflow, and a rounded zero times
//      f(0) in the adjoint when the masses differ.)
// The filter never loses a pair: tf32 rounds x to 2^-11 and n_j to 2^-11, so
// the product sum is off by at most (2^-10 + 2^-11 + 2^-17)(|x_i|^2 + |x_j|^2)
// (2 |x_i||x_j| <= |x_i|^2 + |x_j|^2; the last term covers the float32
// accumulation), which delta = 2^-9 takes off in advance, and `cut` leaves
// room for the rounding of s + eps in the exact test.  It admits about 1 %
// more pairs than the test keeps.
//
// What bounds it: issue slots (78 % used) with the gathers' shared-memory
// wavefronts close behind (73 %); per 32 pairs about 1.5 slots per candidate in
// step 2 and 28 per hit in step 3, against 20 per candidate in the dense loop.
// A batch whose fullest lane holds more hits than HITS_DENSE of its records (a
// halo next door) is evaluated densely from the same tile instead.  Measured
// (GB300), gather force and adjoint with dL/dm: 2.1M lattice particles 1.83 ->
// 0.92 ms and 3.17 -> 1.42 ms, 4096 uniform ones 85 -> 71 us; 16.8M clustered
// 61.9 -> 58.8 ms for the force, whose small cells alone take this path.
// Symmetric force and adjoint, lattice: 1.24 -> 0.97 ms and 2.20 -> 1.41 ms.
#pragma once

#include "hacc_terms.cuh"

namespace hacc {
namespace {

constexpr int HITS_RECS = 256;  // staged candidates: 32 steps of 8 columns, one mask bit per step
constexpr float HITS_DELTA = 0.001953125f;  // 2^-9
// a batch is evaluated densely when its fullest lane has this share of hits
constexpr float HITS_DENSE = 0.6f;

// Chaining-mesh cells of at most HITS_CELL particles take the hit path.  40 is
// not the fastest bound: at 40, 48 and 64 the symmetric force of 2.1M lattice
// particles takes 0.97, 0.93, 0.92 ms (1.24 with the dense kernel alone), the
// gather force at 1.5 particles per unit volume 0.44, 0.31, 0.26 and with a
// skin of 0.3 on the lattice 1.64, 1.29, 1.26, clustered fields the same.  It
// was set by the test of the 64^3 trajectory's gradient, which allows 1e-5 of
// the float64 reference: its symmetric pair at split_T 64 reads 9.84e-6 at 40,
// 1.007e-5 at 48 and 1.004e-5 at 64.  (The error is one draw of the rounding:
// over split_T 32 to 128 all three read 9.1e-6 to 1.01e-5, 9.6e-6 on average.)
constexpr int HITS_CELL = 40;

// Shared memory of the path (bytes from its base): a pad of records outside
// any cutoff (read by lanes that have run out of bits), the records, their
// cotangents (adjoint), their n_j, and the mask words, each with the address
// of its column, and one word that says which records are the i cell's own.
constexpr int HITS_PAD = 128;
constexpr float HITS_FAR = 1.0e18f;  // an empty record's coordinates: outside any cutoff, squares finite
constexpr int HITS_LAM = HITS_RECS * 16;  // from a record to its cotangent (adjoint)
__host__ __device__ constexpr int hits_n_off(int mode)
{
    return HITS_PAD + HITS_RECS * 16 + (is_adjoint(mode) ? HITS_LAM : 0);
}
__host__ __device__ constexpr int hits_word_off(int mode) { return hits_n_off(mode) + HITS_RECS * 4; }
// ... eight words a lane and HITS_STOPS empty ones behind them
constexpr int HITS_STOPS = 4;
__host__ __device__ constexpr int hits_own_off(int mode) { return hits_word_off(mode) + (8 + HITS_STOPS) * 256; }
__host__ __device__ constexpr int hits_bytes(int mode) { return hits_own_off(mode) + 16; }

__device__ __forceinline__ float4 lds128(uint32_t a)
{
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(a)
                 : "memory");
    return v;
}
__device__ __forceinline__ float lds32(uint32_t a)
{
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void sts128(uint32_t a, float4 v)
{
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
                 : "memory");
}
__device__ __forceinline__ void sts32(uint32_t a, float v)
{
    asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ uint32_t lds32u(uint32_t a)
{
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void sts32u(uint32_t a, uint32_t v)
{
    asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void sts64(uint32_t a, uint32_t x, uint32_t y)
{
    asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(a), "r"(x), "r"(y) : "memory");
}

__device__ __forceinline__ void fence_async_proxy() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void bulk_copy(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
        "l"(src), "r"(bytes), "r"(bar)
        : "memory");
}

__device__ __forceinline__ uint32_t to_tf32(float x)
{
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return r;
}

// d = A B: A 16 x 8 (lane (g, q) holds rows g, g + 8 of columns q, q + 4), B 8 x 8
// (rows q, q + 4 of column g), d 16 x 8 (rows g, g + 8, columns 2 q, 2 q + 1).
__device__ __forceinline__ void mma_16x8x8(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%10, %10, %10, %10};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}

// a - b + s L rounded once (s = -1, 0, 1): two exact sums and their errors.
__device__ __forceinline__ float image_delta(float a, float b, float sL)
{
    const float s1 = __fsub_rn(a, b), t1 = __fsub_rn(s1, a);
    const float e1 = __fsub_rn(__fsub_rn(a, __fsub_rn(s1, t1)), __fadd_rn(b, t1));
    const float s2 = __fadd_rn(s1, sL), t2 = __fsub_rn(s2, s1);
    const float e2 = __fadd_rn(__fsub_rn(s1, __fsub_rn(s2, t2)), __fsub_rn(sL, t2));
    return __fadd_rn(s2, __fadd_rn(e1, e2));
}

// Coordinates of a volume's cell (local id below 2^31, n^3 < 2^31).
__device__ __forceinline__ void local_cell(uint32_t lc, uint32_t n, int &cx, int &cy, int &cz)
{
    const uint32_t r = lc / n, z = r / n;
    cx = (int)(lc - r * n);
    cy = (int)(r - z * n);
    cz = (int)z;
}

// One i's sums: float32 over at most HITS_FOLD pairs, then compensated.  Folds
// of 64 left 2.2e-7 rms against float64 on the lattice, of 16 1.8e-7 (the dense
// symmetric kernel 1.9e-7), for 2 % of the time.
constexpr int HITS_FOLD = 16;

template <int MODE>
struct HitAcc {
    static constexpr int NC = MODE == FORCE ? 3 : MODE == POTENTIAL ? 1 : adj_nacc(MODE);
    float p[ADJ_NACC], h[NC], l[NC];
    __device__ __forceinline__ HitAcc()
    {
#pragma unroll
        for (int k = 0; k < ADJ_NACC; ++k) p[k] = 0.f;
#pragma unroll
        for (int k = 0; k < NC; ++k) h[k] = l[k] = 0.f;
    }
    __device__ __forceinline__ void fold()
    {
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            two_sum_acc(h[k], l[k], p[k]);
            p[k] = 0.f;
        }
    }
    __device__ __forceinline__ float total(int k) const { return h[k] + l[k]; }
};

// The pair (i, staged record at address rec), added to the i's sums.
// One body serves both mass paths: with equal masses the staged masses and mi are 1.
template <int MODE>
__device__ __forceinline__ void hit_pair(uint32_t rec, const float4 &oi, float mi, const float4 &li, const PairConsts &K,
                                         float (&p)[ADJ_NACC])
{
    const float4 o = lds128(rec);
    if constexpr (MODE == FORCE)
        pair_force<false>(o, oi.x, oi.y, oi.z, K, p);
    else if constexpr (MODE == POTENTIAL)
        pair_potential(o, oi.x, oi.y, oi.z, K, p);
    else
        pair_adjoint<MODE == ADJOINT_GM, false>(o, lds128(rec + HITS_LAM), oi.x, oi.y, oi.z, mi, li.x, li.y,
                                                li.z, K, p);
}

// The i particles [ib, ie) of chaining-mesh cell c (at most 32) against the
// cell's list, all of it or the small cells (at most HITS_CELL particles)
// only; unit: every mass taken as 1.  `phase`: the parity of the next use of `bar`.  On return lane (g, q)
// = (lane / 4, lane mod 4) holds the totals of row g + 8 q (at most 16
// particles: g + 8 (q mod 2), in both lanes that share the row), i = ib + row,
// if active.  False if a wait ran out.
template <int MODE>
__device__ __forceinline__ bool run_hits(const KArgs &a, uint32_t base, uint32_t bar, uint32_t &phase, int lane,
                                         int c, int ib, int ie, const hacc_volume &vol, bool unit, bool small_only,
                                         HitAcc<MODE> &A,
                                         float4 &oi, float4 &li, int &i_own, bool &active)
{
    const bool half = ie - ib <= 16;  // one tile of 16 rows, each row in two lanes; else two tiles
    const int NW = half ? 4 : 8;      // mask words per lane
    const PairConsts &K = a.k;
    const uint32_t tile = base + HITS_PAD, words = base + hits_word_off(MODE) + 8 * lane,
                   rows = words - 8 * lane;  // the i records, before the words are written
    const int g = lane >> 2, q = lane & 3;
    // the i records by one bulk copy (the previous task's use of the region is fenced at its end)
    if (lane == 0) {
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"((uint32_t)(ie - ib) * 16u)
                     : "memory");
        bulk_copy(rows, a.pos + ib, (uint32_t)(ie - ib) * 16u, bar);
    }
    // records outside any cutoff ahead of the tile, and the end of the word list
    if (lane < HITS_PAD / 16) sts128(base + 16 * lane, make_float4(HITS_FAR, HITS_FAR, HITS_FAR, 0.f));
    for (int k = 0; k < HITS_STOPS; ++k) sts64(words + (NW + k) * 256, 0u, tile);
    const int row = g + 8 * (half ? q & 1 : q);
    i_own = ib + row;
    active = i_own < ie;
    li = make_float4(0.f, 0.f, 0.f, 0.f);
    if constexpr (is_adjoint(MODE)) {
        if (active) li = a.lam[i_own];
    }

    int cx, cy, cz;
    local_cell((uint32_t)((int64_t)c - vol.cell_base), (uint32_t)vol.n, cx, cy, cz);
    const float w = vol.w, ox = cell_centre(cx, w), oy = cell_centre(cy, w), oz = cell_centre(cz, w);

    if (!warp_wait(bar, phase, a.wait_limit)) {
        warp_wait(bar, phase, WAIT_LIMIT_CYCLES);  // let the copy in flight land
        return false;
    }
    phase ^= 1u;
    // A: rows (-2 x, -2 y, -2 z, 1 | n_i - cut in two tf32 words, 0, 0) against B's (x, y, z, n_j | 1, 1, 0, 0)
    uint32_t Af[2][4];
    oi = active ? lds128(rows + 16 * row) : make_float4(0.f, 0.f, 0.f, 0.f);
    {
        const float n2 = fmaf(oi.z, oi.z, fmaf(oi.y, oi.y, oi.x * oi.x));
        const float ni = active ? fmaf(n2, 1.0f - HITS_DELTA, -K.hit_cut) : 1.0e30f;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int rr = g + 8 * r;
            const float x = q < 3 && ib + rr < ie ? lds32(rows + 16 * rr + 4 * q) : 0.f;
            Af[r >> 1][r & 1] = to_tf32(q < 3 ? -2.0f * x : 1.0f);
            const float n = __shfl_sync(FULL, ni, (lane & ~3) | r);  // half: rows below 16 only
            const uint32_t hi = to_tf32(n);
            Af[r >> 1][2 + (r & 1)] = q == 0 ? hi : q == 1 ? to_tf32(n - __uint_as_float(hi)) : 0u;
        }
    }
    const float mi = unit ? 1.0f : oi.w;
    const uint32_t ones = q < 2 ? __float_as_uint(1.0f) : 0u;

    const int64_t e0 = a.nbr_off[c];
    const int ne = (int)(a.nbr_off[c + 1] - e0);
#pragma unroll 1
    for (int g0 = 0; g0 < ne; g0 += 32) {
        // lane l describes one entry: its j range, image offset and place among the group's records.
        // The 27-cell stencil is taken in steps of ten entries, so that every nine of them hold each
        // x, each y and each z offset three times: a batch then holds about as many partners of every i.
        const int ng = min(32, ne - g0);
        int jb = 0, cnt = 0;
        float Dx = 0.f, Dy = 0.f, Dz = 0.f;
        bool home = false;  // the i cell itself
        if (lane < ng) {
            const int64_t e = e0 + g0 + (ng == 27 ? lane * 10 % 27 : lane);
            const int cp = a.nbr_cell[e];
            const int sh = a.nbr_shift[e];
            home = cp == c && sh == 13;
            jb = a.cell_start[cp];
            cnt = a.cell_start[cp + 1] - jb;
            if (small_only && cnt > HITS_CELL) cnt = 0;
            int px, py, pz;
            local_cell((uint32_t)((int64_t)cp - vol.cell_base), (uint32_t)vol.n, px, py, pz);
            Dx = image_delta(cell_centre(px, w), ox, (float)(sh % 3 - 1) * vol.L);
            Dy = image_delta(cell_centre(py, w), oy, (float)((sh / 3) % 3 - 1) * vol.L);
            Dz = image_delta(cell_centre(pz, w), oz, (float)(sh / 9 - 1) * vol.L);
        }
        int first = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(FULL, first, o);
            if (lane >= o) first += t;
        }
        const int total = __shfl_sync(FULL, first, 31);
        first -= cnt;
        // the particle that record 0 would be in the i cell's own entry (none: out of every lane's reach)
        if (lane == 0) sts32u(base + hits_own_off(MODE), 0x7fffffff);
        __syncwarp();
        if (home) sts32u(base + hits_own_off(MODE), (uint32_t)(jb - first));

#pragma unroll 1
        for (int t0 = 0; t0 < total; t0 += HITS_RECS) {
            const int nb = min(HITS_RECS, total - t0), nb8 = (nb + 7) & ~7;
            const int at = max(first, t0), n_own = min(first + cnt, t0 + HITS_RECS) - at;
            const int base_j = jb - first + t0;  // record r of the batch is particle base_j + r of its entry
            // ---- 1. stage the batch in the i cell's frame, U entries' loads in flight together
            __syncwarp();  // the previous batch has been read
            if (lane < nb8 - nb) {  // fill the last step with records outside any cutoff
                sts128(tile + 16 * (nb + lane), make_float4(HITS_FAR, HITS_FAR, HITS_FAR, 0.f));
                sts32(base + hits_n_off(MODE) + 4 * (nb + lane), 1.0e37f);
                if constexpr (is_adjoint(MODE))
                    sts128(tile + HITS_LAM + 16 * (nb + lane), make_float4(0.f, 0.f, 0.f, 0.f));
            }
            auto put = [&](int r, const float4 &p, const float4 &l, int e) {
                const float x = p.x + __shfl_sync(FULL, Dx, e), y = p.y + __shfl_sync(FULL, Dy, e),
                            z = p.z + __shfl_sync(FULL, Dz, e);
                if (r >= 0) {
                    sts128(tile + 16 * r, make_float4(x, y, z, unit ? 1.0f : p.w));
                    sts32(base + hits_n_off(MODE) + 4 * r, fmaf(z, z, fmaf(y, y, x * x)) * (1.0f - HITS_DELTA));
                    if constexpr (is_adjoint(MODE)) sts128(tile + HITS_LAM + 16 * r, l);
                }
            };
            // (2.1M lattice particles: force 925 us with two, 944 with three; potential 853 and 845)
            constexpr int U = MODE == POTENTIAL ? 3 : 2;
            const int place = (at - t0) | n_own << 16;
            unsigned act = __ballot_sync(FULL, n_own > 0);
#pragma unroll 1
            while (act) {
                float4 p[U], l[U];
                int e[U], r[U], n[U], j[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    e[u] = __ffs(act) - 1;  // -1: none left
                    act &= act - 1;
                    const int pl = __shfl_sync(FULL, place, e[u]);
                    n[u] = e[u] < 0 ? 0 : pl >> 16;
                    r[u] = lane < n[u] ? (pl & 0xffff) + lane : -1;
                    j[u] = __shfl_sync(FULL, base_j, e[u]) + (pl & 0xffff) + lane;
                    p[u] = l[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (r[u] >= 0) {
                        p[u] = a.pos[j[u]];
                        if constexpr (is_adjoint(MODE)) l[u] = a.lam[j[u]];
                    }
                }
#pragma unroll
                for (int u = 0; u < U; ++u) put(r[u], p[u], l[u], e[u]);
#pragma unroll
                for (int u = 0; u < U; ++u) {
#pragma unroll 1
                    for (int o = 32; o < n[u]; o += 32) {
                        const bool ok = lane + o < n[u];
                        float4 p2 = make_float4(0.f, 0.f, 0.f, 0.f), l2 = p2;
                        if (ok) {
                            p2 = a.pos[j[u] + o];
                            if constexpr (is_adjoint(MODE)) l2 = a.lam[j[u] + o];
                        }
                        put(ok ? r[u] + o : -1, p2, l2, e[u]);
                    }
                }
            }
            __syncwarp();
            // ---- 2. sign masks: M[r][k] bit s = pair (row g + 8 r, record 8 s + 2 q + k) may be inside
            uint32_t M[4][2];
#pragma unroll
            for (int r = 0; r < 4; ++r) M[r][0] = M[r][1] = 0u;
            {
                const bool own_n = q == 3;
                const uint32_t stride = own_n ? 32u : 128u;
                uint32_t ad = (own_n ? base + hits_n_off(MODE) + 4 * g : tile + 16 * g + 4 * q) +
                              stride * (uint32_t)(nb8 / 8 - 1);
                auto signs = [&](int m, uint32_t b) {
                    float d[4];
                    mma_16x8x8(d, Af[m], b, ones);
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        M[2 * m][k] = __funnelshift_l(__float_as_uint(d[k]), M[2 * m][k], 1);
                        M[2 * m + 1][k] = __funnelshift_l(__float_as_uint(d[2 + k]), M[2 * m + 1][k], 1);
                    }
                };
                if (half) {
#pragma unroll 2
                    for (int s = nb8 / 8; s > 0; --s) {
                        const uint32_t b = to_tf32(lds32(ad));
                        ad -= stride;
                        signs(0, b);
                    }
                } else {
#pragma unroll 2
                    for (int s = nb8 / 8; s > 0; --s) {
                        const uint32_t b = to_tf32(lds32(ad));
                        ad -= stride;
                        signs(0, b);
                        signs(1, b);
                    }
                }
            }
            // ---- transpose among the four lanes of a row group: the lane's own row, column by column.
            // Lanes start at different columns, so that their gathers meet different banks.
            int trips = 0;
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                if (s >= 2 && half) break;
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const uint32_t lo = (q ^ s) & 1 ? M[1][k] : M[0][k], hi = (q ^ s) & 1 ? M[3][k] : M[2][k];
                    uint32_t v = !half && ((q ^ s) & 2) ? hi : lo;
                    v = __shfl_xor_sync(FULL, v, s);
                    trips += max(__popc(v), 1);
                    sts64(words + 256 * ((2 * s + k) ^ (g & 1)), v, tile + 16 * (2 * (q ^ s) + k));
                }
            }
            // no pair of an i with itself: its own record, if it is in this batch, loses its bit (such a
            // batch never runs densely)
            const uint32_t own = (uint32_t)(i_own - t0) - lds32u(base + hits_own_off(MODE));
            if (own < (uint32_t)nb) {
                const uint32_t s = ((own >> 1) & 3) ^ q;  // the lane's slot of column own mod 8 (half: 2, 3 are the other lane's)
                if (s < (half ? 2u : 4u)) {
                    const uint32_t w = words + 256 * ((2 * s + (own & 1)) ^ (g & 1));
                    const uint32_t v = lds32u(w), v2 = v & ~(1u << (own >> 3));
                    sts32u(w, v2);
                    trips -= max(__popc(v), 1) - max(__popc(v2), 1);
                }
            }
            trips = __reduce_max_sync(FULL, trips);
            __syncwarp();
            // ---- 3. the pairs
            if ((float)trips < HITS_DENSE * (float)(half ? nb8 / 2 : nb8) || __any_sync(FULL, own < (uint32_t)nb)) {
                uint32_t mask, col, wp = words + 256;
                asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(mask), "=r"(col) : "r"(words) : "memory");
                const uint32_t wend = words + NW * 256;
                for (int f = 0; f < trips; f += HITS_FOLD) {
                    if (f) A.fold();
                    // trips in fours (a lane without bits reads the pad); a lane may run HITS_STOPS words
                    // past its last before its pointer is put back
#pragma unroll 1
                    for (int t = min(trips - f, HITS_FOLD); t > 0; t -= HITS_STOPS) {
#pragma unroll
                        for (int u = 0; u < HITS_STOPS; ++u) {
                            int b;
                            uint32_t bit;
                            asm("bfind.u32 %0, %1;" : "=r"(b) : "r"(mask));   // -1: none (reads the pad)
                            asm("shl.b32 %0, 1, %1;" : "=r"(bit) : "r"(b));  // clamped: 0 for none
                            const uint32_t rec = col + 128 * b;
                            mask &= ~bit;
                            asm volatile(
                                "{\n\t.reg .pred z;\n\tsetp.eq.u32 z, %0, 0;\n\t"
                                "@z ld.shared.v2.u32 {%0, %1}, [%2];\n\t@z add.u32 %2, %2, 256;\n\t}"
                                : "+r"(mask), "+r"(col), "+r"(wp)
                                :
                                : "memory");
                            hit_pair<MODE>(rec, oi, mi, li, K, A.p);
                        }
                        wp = min(wp, wend);
                    }
                }
            } else {
                const int nr = half ? nb8 / 2 : nb8, r0 = half && (q & 2) ? nr : 0;
                for (int f = 0; f < nr; f += HITS_FOLD) {
                    if (f) A.fold();
#pragma unroll 4
                    for (int r = f; r < min(nr, f + HITS_FOLD); ++r)
                        hit_pair<MODE>(tile + 16 * (r0 + r), oi, mi, li, K, A.p);
                }
            }
            A.fold();
        }
    }
    if (half) {
        // lanes q and q ^ 2 hold the two parts of one row: the low one adds the high one's
#pragma unroll
        for (int k = 0; k < HitAcc<MODE>::NC; ++k) {
            const float h2 = __shfl_xor_sync(FULL, A.h[k], 2), l2 = __shfl_xor_sync(FULL, A.l[k], 2);
            two_sum_acc(A.h[k], A.l[k], h2);
            A.l[k] = __fadd_rn(A.l[k], l2);
        }
        active = active && q < 2;
    }
    __syncwarp();
    fence_async_proxy();  // the region's next use may be a bulk copy
    return true;
}

// ---------------------------------------------------------------------------
// Tasks: which cells take the path, and their persistent loop
// ---------------------------------------------------------------------------

// Which cells take the hit path: those of at most HITS_CELL particles and, in a
// one-sided (gather) call, of at most 27 HITS_CELL candidates, since a larger
// neighbour's pairs are mostly inside the cutoff or far outside and the dense
// kernel holds two i per lane (without the second bound 1M clustered particles
// take 5.4 ms, with it 4.2; the dense kernel alone 4.5).  (A symmetric call's dense tasks meet the large
// neighbours themselves.)
__device__ __forceinline__ bool hits_cell(const KArgs &a, int c, bool one_sided)
{
    if (a.cell_start[c + 1] - a.cell_start[c] > HITS_CELL) return false;
    if (!one_sided) return true;
    const int64_t e0 = a.nbr_off[c], e1 = a.nbr_off[c + 1];
    int64_t nj = 0;
    for (int64_t e = e0; e < e1; ++e) {
        nj += a.cell_start[a.nbr_cell[e] + 1] - a.cell_start[a.nbr_cell[e]];
    }
    return nj <= 27 * HITS_CELL;
}

// Segments.  In a symmetric call the sums of a task go to the totals by
// atomics, so a task may be cut along its j records: without that one warp
// holds a halo cell's task of 128 particles and ten thousand j for over a
// millisecond, and the kernel's last tasks leave the GPU idle.  A task of
// more than a.seg_pairs pairs becomes segments of about that many (at most
// one per particle of the task, and 256 j at least).  An item of the dense
// kernels is (task, segment | scale << 16 | last << 24): segment s of scale k
// holds the j records [s per, (s + 1) per), per = segment_records 2^k, the
// last one all the rest.
constexpr int SEG_WHOLE = 1 << 24;  // segment 0 and the last: the whole task
__device__ __forceinline__ int segment_records(const KArgs &a, int size) { return max(a.seg_pairs / size, 256) & ~31; }
__device__ __forceinline__ int segment_count(const KArgs &a, int size, int nj, int &scale)
{
    const int most = min(size, 32767), per = segment_records(a, size);
    scale = 0;
    while ((nj + (per << scale) - 1) / (per << scale) > most) ++scale;
    return max(1, (nj + (per << scale) - 1) / (per << scale));
}

// Pairs per segment for N particles: the tail costs a share of the whole
// call, the segments' own prologues and sums a share of the pairs.  Symmetric
// force with segments of 16k, 32k, 64k, 128k pairs: 262,144 clustered particles
// 0.40, 0.40, 0.42, 0.53 ms (0.56 uncut), 16.8M 38.9, 38.8, 37.6, 37.1 ms; with
// this rule 0.39 and 35.2 ms (36.3 uncut), 1M 3.8 -> 2.7 ms.
int seg_pairs_for(int64_t N)
{
    const int64_t p = N / 16;
    return (int)(p < 32768 ? 32768 : p > (1 << 20) ? (1 << 20) : p);
}

// The list entry of cell (or leaf) c itself, image 13.  A chaining-mesh list
// is symmetric under d -> -d with the cell in the middle; a tree leaf's list
// is sorted by (image code, leaf id) and symmetric too (leaf j with image s
// is listed for i iff i with image -s is listed for j), so its own entry is
// found by bisection and everything after it is the forward half.
__device__ __forceinline__ int64_t self_entry(const KArgs &a, int c, int64_t e0, int64_t e1, const hacc_volume &vol)
{
    if (!a.origin) return e0 + (vol.S - 1) / 2;
    int64_t lo = e0, hi = e1 - 1;
    while (lo < hi) {  // first entry with (code, leaf) >= (13, c)
        const int64_t mid = (lo + hi) >> 1;
        const int code = a.nbr_shift[mid], leaf = a.nbr_cell[mid];
        if (code < 13 || (code == 13 && leaf < c)) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// Which half of its list a symmetric call's dense task walks: every entry
// after its own cell, and the small cells before it -- those cells' tasks run
// on the hit path, which sums small cells only, so a dense cell meets all of
// its small neighbours itself (both particles of each pair).
__device__ __forceinline__ int64_t first_entry(const KArgs &a, int64_t e0, int64_t mid) { return a.origin ? mid : e0; }
__device__ __forceinline__ bool takes_entry(int64_t e, int64_t mid, int cnt) { return e > mid || cnt <= HITS_CELL; }

// The j records a symmetric call's dense task meets beyond its own chunk.  A
// tree's lists are long and its leaves alike (between half of the largest size
// and all of it), so there sixteen entries stand for all: the last segment
// takes whatever is left.  (Walked by one thread a task, the lists of 45,593
// leaves of at most 8 took 665 us of the call's 5,640; of 5,892 leaves of at
// most 64, 1.02 ms a call with exact counts, 0.95 with these.)
__device__ __forceinline__ int dense_reach(const KArgs &a, const int4 &task)
{
    const int64_t e0 = a.nbr_off[task.x], e1 = a.nbr_off[task.x + 1];
    const int64_t mid = self_entry(a, task.x, e0, e1, a.vols[task.w]);
    int64_t nj = a.cell_start[task.x + 1] - task.z;
    if (a.origin && e1 - mid > 32) {
        int some = 0;
#pragma unroll 4
        for (int k = 0; k < 16; ++k) {
            const int cp = a.nbr_cell[mid + 1 + (e1 - mid - 1) * k / 16];
            some += a.cell_start[cp + 1] - a.cell_start[cp];
        }
        return (int)min(nj + (e1 - mid - 1) * some / 16, (int64_t)1 << 30);
    }
    for (int64_t e = first_entry(a, e0, mid); e < e1; ++e) {
        if (e == mid) continue;
        const int cnt = a.cell_start[a.nbr_cell[e] + 1] - a.cell_start[a.nbr_cell[e]];
        if (takes_entry(e, mid, cnt)) nj += cnt;
    }
    return (int)min(max(nj, (int64_t)0), (int64_t)1 << 30);
}

// The split: the heaviest-first task order becomes two lists -- the dense
// kernel's items from the front of `items`, the hit kernel's tasks from its back
// (N slots).  First every task's items are counted, then every block adds up the
// chunks before its own and places them; the block that knows the totals leaves
// the counters ready.  The lists keep the order (with blocks that took their
// places by atomics, so in any order of 1024 tasks, the gather force of 262,144
// clustered particles on leaves of at most 32 took 1.90 to 2.08 ms: a heavy task
// taken late is the call's tail; in order 1.81).  Only a symmetric call of up to
// LIGHT_FIRST particles takes its dense chunks from the last to the first: its
// heavy tasks are cut into segments, so they make no tail, and at the front all
// warps add to the totals of the one densest halo.  Symmetric force in order and
// light first: 262,144 clustered particles 0.417 and 0.394 ms, on leaves of at
// most 8 4.83 and 4.52, 1M 2.81 and 2.69, 4.1M 7.89 and 7.92, 16.8M 35.2 and 35.5.
constexpr int64_t LIGHT_FIRST = 1 << 21;
constexpr int SPLIT = 1024;  // tasks a chunk

__device__ __forceinline__ int split_tasks_in(const KArgs &a)
{
    const int nt = task_count(a);
#ifdef HACC_DEBUG_BOUNDS
    if (nt > a.N) {  // a task holds a particle
        if (threadIdx.x == 0) report_bounds(a);
        return (int)a.N;
    }
#endif
    return nt;
}

// Sums of v[0], v[1] over the block, before the thread (v replaced) and in all.
__device__ __forceinline__ int2 split_scan(int (&v)[2], int (*wsum)[2])
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int own[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        own[k] = v[k];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int s = __shfl_up_sync(FULL, v[k], o);
            if (lane >= o) v[k] += s;
        }
        if (lane == 31) wsum[warp][k] = v[k];
    }
    __syncthreads();
    int all[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int w = wsum[lane][k];
        all[k] = (int)__reduce_add_sync(FULL, (unsigned)w);
        v[k] += (int)__reduce_add_sync(FULL, lane < warp ? (unsigned)w : 0u) - own[k];
    }
    __syncthreads();  // wsum may be written again
    return make_int2(all[0], all[1]);
}

// codes: per task its items | scale << 16 | kind << 24 (kind 0: the dense kernel's, 1: the hit kernel's).
__global__ void __launch_bounds__(SPLIT)
k_split_count(const KArgs a, bool one_sided, int32_t *__restrict__ codes, int2 *__restrict__ totals)
{
    __shared__ int wsum[SPLIT / 32][2];
    const int nt = split_tasks_in(a);
    for (int t0 = blockIdx.x * SPLIT; t0 < nt; t0 += gridDim.x * SPLIT) {
        const int t = t0 + threadIdx.x;
        int kind = 0, n = 0, scale = 0;
        if (t < nt) {
            const int oi = a.order[t];
#ifdef HACC_DEBUG_BOUNDS
            int4 task;
            const bool ok = task_in_bounds(a, oi, 0, 1, task);
            if (!ok) report_bounds(a);
#else
            constexpr bool ok = true;
            const int4 task = a.tasks[oi];
#endif
            if (ok) {
                kind = !a.origin && hits_cell(a, task.x, one_sided) ? 1 : 0;
                n = kind || one_sided ? 1 : segment_count(a, task.z - task.y, dense_reach(a, task), scale);
            }
            codes[t] = n | scale << 16 | kind << 24;
        }
        int v[2] = {kind ? 0 : n, kind ? n : 0};
        const int2 all = split_scan(v, wsum);
        if (threadIdx.x == 0) totals[t0 / SPLIT] = all;
    }
}

// counts: [0] and [1] the dense and the hit kernel's next item (0), [2] and [3] how many there are.
__global__ void __launch_bounds__(SPLIT)
k_split_place(const KArgs a, bool light_first, const int32_t *__restrict__ codes, const int2 *__restrict__ totals,
              int2 *__restrict__ items, int32_t *__restrict__ counts)
{
    __shared__ int wsum[SPLIT / 32][2];
    const int nt = split_tasks_in(a);
    if (nt == 0 && blockIdx.x == 0 && threadIdx.x < 4) counts[threadIdx.x] = 0;
    for (int t0 = blockIdx.x * SPLIT; t0 < nt; t0 += gridDim.x * SPLIT) {
        const int chunk = t0 / SPLIT, chunks = (nt + SPLIT - 1) / SPLIT;
        int before[2] = {0, 0};  // dense items and hit tasks of the chunks to go ahead of this one
        for (int c = threadIdx.x; c < chunks; c += SPLIT) {
            const int2 w = totals[c];
            if (light_first ? c > chunk : c < chunk) before[0] += w.x;
            if (c < chunk) before[1] += w.y;
        }
        const int2 base = split_scan(before, wsum);
        const int t = t0 + threadIdx.x;
        const int code = t < nt ? codes[t] : 0;
        const int kind = code >> 24, n = code & 0xffff, scale = (code >> 16) & 255;
        int v[2] = {kind ? 0 : n, kind ? n : 0};
        const int2 all = split_scan(v, wsum);
        if (threadIdx.x == 0) {  // the last dense chunk and the last chunk know the totals
            if (chunk == (light_first ? 0 : chunks - 1)) counts[2] = base.x + all.x;
            if (chunk == chunks - 1) counts[3] = base.y + all.y;
            if (chunk == 0) counts[0] = counts[1] = 0;
        }
        const int64_t slot = kind ? (int64_t)base.y + v[1] : (int64_t)base.x + v[0];
        const int oi = t < nt ? a.order[t] : 0;
#ifdef HACC_DEBUG_BOUNDS
        if (slot + n > a.N) report_bounds(a);
#endif
        for (int s = 0; s < n; ++s)
            if (slot + s < a.N)
                items[kind ? a.N - 1 - slot : slot + s] = make_int2(oi, s | scale << 16 | (s == n - 1 ? 1 << 24 : 0));
    }
}

// Splits the tasks: `a` then names the dense kernel's items and the hit
// kernel's tasks.  The totals' region serves as scratch (4 bytes a task and 8 a
// chunk of its 32 a particle).
int split_tasks(KArgs &a, const ForceWs &F, bool one_sided, cudaStream_t st)
{
    a.counter = F.counter;
    a.seg_pairs = seg_pairs_for(a.N);
    int64_t g = (a.task_cap + SPLIT - 1) / SPLIT;
    if (g > num_sms() * 2) g = num_sms() * 2;
    if (g < 1) g = 1;
    int2 *totals = reinterpret_cast<int2 *>(F.acc);
    int32_t *codes = reinterpret_cast<int32_t *>(totals + (a.N + SPLIT - 1) / SPLIT);
    k_split_count<<<(int)g, SPLIT, 0, st>>>(a, one_sided, codes, totals);
    HACC_LAUNCH_CHECK();
    k_split_place<<<(int)g, SPLIT, 0, st>>>(a, !one_sided && a.N <= LIGHT_FIRST, codes, totals, F.items, F.counter);
    HACC_LAUNCH_CHECK();
    a.items = F.items;
    a.n_items = F.counter + 2;
    a.hit_order = F.items + (a.N - 1);
    a.hit_count = F.counter + 1;
    return HACC_OK;
}

constexpr int HITS_WARPS = 4;
__host__ __device__ constexpr int hits_ctas(int mode) { return is_adjoint(mode) ? 4 : 6; }
__host__ __device__ constexpr int hits_warp_bytes(int mode)
{
    return (hits_bytes(mode) + 16 + 127) / 128 * 128;
}

struct HitWarp {
    uint32_t base, bar, phase;
};

// A warp's region and its barrier, initialised.
__device__ __forceinline__ HitWarp hits_warp(unsigned char *smem, int warp, int lane, int mode)
{
    HitWarp W;
    W.base = smem_addr(smem + (size_t)warp * hits_warp_bytes(mode));
    W.bar = W.base + hits_warp_bytes(mode) - 16;
    W.phase = 0u;
    if (lane == 0) {
        mbar_init(W.bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_async_proxy();
    }
    __syncwarp();
    return W;
}

// Persistent work-stealing loop: each warp takes hit tasks from a global
// counter and runs them in chunks of at most 32 particles.
template <class Run>
__device__ __forceinline__ void hits_tasks(const KArgs &a, int lane, const Run &run)
{
    const int nt = hit_tasks(a);
    while (true) {
        int t = 0;
        if (lane == 0) t = atomicAdd(a.hit_count, 1);
        t = __shfl_sync(FULL, t, 0);
        if (t >= nt) return;
        int4 task;
        if (!take_task(a, a.hit_order[-(int64_t)t].x, lane, task)) continue;
        const hacc_volume &vol = a.vols[task.w];
        for (int b = task.y; b < task.z; b += 32) {
            if (!run(task.x, b, min(b + 32, task.z), vol)) {
                if (lane == 0) atomicOr(a.status, HACC_STATUS_TIMEOUT);
                return;
            }
        }
    }
}

// Launched behind the dense kernel with programmatic serialisation: its
// blocks fill the room that the dense kernel's leave, so that the two kernels'
// last tasks overlap.  It needs nothing the dense kernel writes, and its
// blocks wait for the dense kernel's end before they exit, so that work behind
// it in the stream finds both done.
template <class Kernel, class... Args>
int launch_hits(Kernel kern, int mode, cudaStream_t st, Args... args)
{
    const int smem = HITS_WARPS * hits_warp_bytes(mode);
    HACC_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    cudaLaunchAttribute overlap{};
    overlap.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    overlap.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(num_sms() * hits_ctas(mode));
    cfg.blockDim = dim3(HITS_WARPS * 32);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &overlap;
    cfg.numAttrs = 1;
    count_launch();
    if (cudaLaunchKernelEx(&cfg, kern, args...) != cudaSuccess) {
        (void)cudaGetLastError();
        return HACC_ERR_CUDA;
    }
    return HACC_OK;
}

}  // namespace
}  // namespace hacc

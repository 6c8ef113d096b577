// Short-range pair force (Eq. 7 of the paper) and its adjoint.
//
// Work decomposition.  A task is a chunk of at most split_T particles of one
// mesh cell (the "i" particles); one warp owns one task at a time, one i per
// lane, and walks the cell's neighbour list.  Every neighbour cell's particle
// range (the "j" particles, contiguous in the sorted array) is staged into a
// per-warp ring of shared-memory tiles by the tensor memory accelerator
// (cp.async.bulk, completion on an mbarrier), and each staged j is broadcast to
// all 32 lanes by a 16-byte shared load.  Warps take tasks from an atomic
// counter (a persistent, work-stealing grid), so the very uneven lists of
// clustered particles balance themselves.  Small chaining-mesh cells take the
// hit path instead (hacc_hits.cuh).
//
// Arithmetic per pair (float32, cutoff as a select, as in the paper's
// branch-free kernel, Sec. III):
//   d  = o_j - (o_i - Delta)            cell-relative offsets, Delta = image origin difference
//   se = eps + d.d                      (three fma)
//   t  = rsqrt(se)
//   f  = t^2 t - poly~(se)              poly~(se) = poly(se - eps), coefficients shifted on the host
//   f  = se < r_c^2 + eps ? f : 0
//   a += m_j f d
// The accumulator is float32 within a tile and compensated (TwoSum into a
// hi/lo pair) across tiles.
#include "hacc_hits.cuh"

namespace hacc {
namespace {

// Per-lane accumulators of IPL i particles: float32 within a tile, then
// folded into a compensated (hi, lo) pair.
template <int MODE, int IPL>
struct Acc;

template <int IPL>
struct Acc<FORCE, IPL> : AccN<IPL, 3> {};

template <int IPL>
struct Acc<POTENTIAL, IPL> : AccN<IPL, 1> {};

// Forward pair loop over one staged tile: every staged j meets the IPL i
// particles of this lane.  Unrolled by hand, four j per trip.
template <int IPL, bool EQ>
__device__ __forceinline__ void tile_force(const float4 *__restrict__ tj, int n, const float (&op)[IPL][3],
                                           const PairConsts &K, Acc<FORCE, IPL> &A)
{
    int j = 0;
    for (; j + 4 <= n; j += 4) {
        const float4 p0 = tj[j], p1 = tj[j + 1], p2 = tj[j + 2], p3 = tj[j + 3];
#pragma unroll
        for (int u = 0; u < IPL; ++u) {
            pair_force<EQ>(p0, op[u][0], op[u][1], op[u][2], K, A.a[u]);
            pair_force<EQ>(p1, op[u][0], op[u][1], op[u][2], K, A.a[u]);
            pair_force<EQ>(p2, op[u][0], op[u][1], op[u][2], K, A.a[u]);
            pair_force<EQ>(p3, op[u][0], op[u][1], op[u][2], K, A.a[u]);
        }
    }
    for (; j < n; ++j) {
        const float4 p = tj[j];
#pragma unroll
        for (int u = 0; u < IPL; ++u) pair_force<EQ>(p, op[u][0], op[u][1], op[u][2], K, A.a[u]);
    }
}

template <int IPL>
__device__ __forceinline__ void tile_potential(const float4 *__restrict__ tj, int n, const float (&op)[IPL][3],
                                               const PairConsts &K, Acc<POTENTIAL, IPL> &A)
{
    int j = 0;
    for (; j + 4 <= n; j += 4) {
        const float4 p0 = tj[j], p1 = tj[j + 1], p2 = tj[j + 2], p3 = tj[j + 3];
#pragma unroll
        for (int u = 0; u < IPL; ++u) {
            pair_potential(p0, op[u][0], op[u][1], op[u][2], K, A.a[u]);
            pair_potential(p1, op[u][0], op[u][1], op[u][2], K, A.a[u]);
            pair_potential(p2, op[u][0], op[u][1], op[u][2], K, A.a[u]);
            pair_potential(p3, op[u][0], op[u][1], op[u][2], K, A.a[u]);
        }
    }
    for (; j < n; ++j) {
        const float4 p = tj[j];
#pragma unroll
        for (int u = 0; u < IPL; ++u) pair_potential(p, op[u][0], op[u][1], op[u][2], K, A.a[u]);
    }
}

// Adjoint pair loop over one staged tile (positions tj, cotangents tl).
template <int MODE, int IPL, bool EQ>
__device__ __forceinline__ void tile_adjoint(const float4 *__restrict__ tj, const float4 *__restrict__ tl, int n,
                                             const float (&op)[IPL][3], const float4 (&oi)[IPL],
                                             const float4 (&li)[IPL], const PairConsts &K,
                                             AccAdj<MODE, IPL, adj_nacc(MODE)> &A)
{
    constexpr bool GM = MODE == ADJOINT_GM;
    int j = 0;
    if constexpr (IPL == 1) {
        // one i per lane: two j per trip for independent work
        for (; j + 2 <= n; j += 2) {
            const float4 p0 = tj[j], p1 = tj[j + 1], l0 = tl[j], l1 = tl[j + 1];
            pair_adjoint<GM, EQ>(p0, l0, op[0][0], op[0][1], op[0][2], oi[0].w, li[0].x, li[0].y, li[0].z, K,
                                 A.p[0]);
            pair_adjoint<GM, EQ>(p1, l1, op[0][0], op[0][1], op[0][2], oi[0].w, li[0].x, li[0].y, li[0].z, K,
                                 A.p[0]);
        }
    }
    for (; j < n; ++j) {
        const float4 p0 = tj[j], l0 = tl[j];
#pragma unroll
        for (int u = 0; u < IPL; ++u)
            pair_adjoint<GM, EQ>(p0, l0, op[u][0], op[u][1], op[u][2], oi[u].w, li[u].x, li[u].y, li[u].z, K,
                                 A.p[u]);
    }
}



template <int MODE, int IPL>
__device__ __forceinline__ auto make_acc(float *comp, int lane)
{
    if constexpr (MODE == FORCE || MODE == POTENTIAL)
        return Acc<MODE, IPL>();
    else
        return AccAdj<MODE, IPL, adj_nacc(MODE)>(comp, lane);
}

// One task: i particles [ib, ie) of cell c (at most 32 IPL of them), every
// entry of the cell's neighbour list.  Returns false if a wait ran out.
// With one i per lane and at most 16 i (half, decided per task), lanes l and
// l + 16 hold the same i and each takes half of every staged piece of j
// records; the two compensated partial sums are added in a fixed order at the
// end, so the result stays deterministic.
template <int MODE, int JT, int STAGES, int IPL, bool EQ>
__device__ __forceinline__ bool run_task(const KArgs &a, Ring<MODE, JT, STAGES> &ring, float *comp, int lane,
                                         int c, int ib, int ie, const hacc_volume &vol)
{
    const bool half = IPL == 1 && ie - ib <= 16;
    const int il = half ? (lane & 15) : lane;  // this lane's i within the task
    const PairConsts &K = a.k;
    const int n = vol.n;
    const float w = vol.w;
    const double Ld = (double)vol.L;
    const int64_t lc = (int64_t)c - vol.cell_base;
    const int cx = (int)(lc % n), cy = (int)((lc / n) % n), cz = (int)(lc / ((int64_t)n * n));
    const float4 org_i = a.origin ? a.origin[c] : make_float4(0.f, 0.f, 0.f, 0.f);

    float4 oi[IPL];
    bool active[IPL];
#pragma unroll
    for (int u = 0; u < IPL; ++u) {
        const int i = ib + il + 32 * u;
        active[u] = i < ie;
        oi[u] = active[u] ? a.pos[i] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    float4 li[IPL];
#pragma unroll
    for (int u = 0; u < IPL; ++u) {
        li[u] = make_float4(0.f, 0.f, 0.f, 0.f);
        if constexpr (is_adjoint(MODE)) {
            if (active[u]) li[u] = a.lam[ib + il + 32 * u];
        }
    }
    auto A = make_acc<MODE, IPL>(comp, lane);

    const int64_t e0 = a.nbr_off[c], e1 = a.nbr_off[c + 1];
    for (int64_t g0 = e0; g0 < e1; g0 += 32) {
        const int ng = (int)min((int64_t)32, e1 - g0);
        // lane l describes entry g0 + l: its j range and image offset Delta
        int jb = 0, cnt = 0;
        float Dx = 0.f, Dy = 0.f, Dz = 0.f;
        if (lane < ng) {
            const int cp = a.nbr_cell[g0 + lane];
            const int sh = a.nbr_shift[g0 + lane];
            jb = a.cell_start[cp];
            cnt = a.cell_start[cp + 1] - jb;
            const int sx = sh % 3 - 1, sy = (sh / 3) % 3 - 1, sz = sh / 9 - 1;
            if (a.origin) {
                // tree leaves: float32 origins, difference and image exact in float64
                const float4 org_j = a.origin[cp];
                Dx = (float)((double)org_j.x - (double)org_i.x + sx * Ld);
                Dy = (float)((double)org_j.y - (double)org_i.y + sy * Ld);
                Dz = (float)((double)org_j.z - (double)org_i.z + sz * Ld);
            } else {
                const int64_t lp = (int64_t)cp - vol.cell_base;
                const int px = (int)(lp % n), py = (int)((lp / n) % n), pz = (int)(lp / ((int64_t)n * n));
                // exact in float64: origins are the float32 cell centres used by the binning
                Dx = (float)((double)cell_centre(px, w) - (double)cell_centre(cx, w) + sx * Ld);
                Dy = (float)((double)cell_centre(py, w) - (double)cell_centre(cy, w) + sy * Ld);
                Dz = (float)((double)cell_centre(pz, w) - (double)cell_centre(cz, w) + sz * Ld);
            }
        }
        int pk = 0, poff = 0;  // producer cursor (entry, record within it)
        int ck = 0, coff = 0;  // consumer cursor
        for (int s = 0; s < STAGES; ++s)  // prologue: fill the ring
            if (!ring.produce(a, lane, ng, cnt, jb, pk, poff)) break;
        int cur = -1;
        float op[IPL][3];
        while (ring.consumed < ring.issued) {
            if (!ring.wait_next(a.wait_limit)) return false;
            const float4 *tj = ring.tile(ring.consumed % STAGES);
            // replay the producer's pieces: each piece is one entry's records
            int filled = 0;
            while (ck < ng && filled < JT) {
                const int c = __shfl_sync(FULL, cnt, ck);
                if (coff >= c) {
                    ++ck;
                    coff = 0;
                    continue;
                }
                const int n = min(JT - filled, c - coff);
                if (ck != cur) {
                    cur = ck;
                    const float dx = __shfl_sync(FULL, Dx, ck), dy = __shfl_sync(FULL, Dy, ck),
                                dz = __shfl_sync(FULL, Dz, ck);
#pragma unroll
                    for (int u = 0; u < IPL; ++u) {
                        op[u][0] = oi[u].x - dx;
                        op[u][1] = oi[u].y - dy;
                        op[u][2] = oi[u].z - dz;
                    }
                }
                // the pair loop over records [o, o + m) of the staged tile
                auto tile = [&](int o, int m) {
                    if constexpr (MODE == FORCE)
                        tile_force<IPL, EQ>(tj + o, m, op, K, A);
                    else if constexpr (MODE == POTENTIAL)
                        tile_potential<IPL>(tj + o, m, op, K, A);
                    else
                        tile_adjoint<MODE, IPL, EQ>(tj + o, tj + JT + o, m, op, oi, li, K, A);
                };
                if constexpr (IPL == 1) {
                    // half: lanes < 16 take records [0, n/2) and, for odd n, record
                    // n/2 alone; lanes >= 16 the rest.  Equal trip counts keep the
                    // loop converged.
                    const int hn = n >> 1;
                    tile(filled + (half && (lane & 16) ? hn + (n & 1) : 0), half ? hn : n);
                    if (half && (n & 1) && lane < 16) tile(filled + hn, 1);
                } else {
                    tile(filled, n);
                }
                filled += n;
                coff += n;
            }
            A.fold();
            ++ring.consumed;
            __syncwarp();
            ring.produce(a, lane, ng, cnt, jb, pk, poff);
        }
    }
    if (half) {
        // lane l (< 16) adds lane l + 16's compensated sums to its own
        if constexpr (MODE == FORCE || MODE == POTENTIAL) {
#pragma unroll
            for (int k = 0; k < (MODE == FORCE ? 3 : 1); ++k) {
                const float h2 = __shfl_down_sync(FULL, A.h[0][k], 16), l2 = __shfl_down_sync(FULL, A.l[0][k], 16);
                two_sum_acc(A.h[0][k], A.l[0][k], h2);
                A.l[0][k] = __fadd_rn(A.l[0][k], l2);
            }
        } else {
#pragma unroll
            for (int k = 0; k < decltype(A)::NACC; ++k) {
                float h = A.hi(0, k), l = A.lo(0, k);
                const float h2 = __shfl_down_sync(FULL, h, 16), l2 = __shfl_down_sync(FULL, l, 16);
                two_sum_acc(h, l, h2);
                A.hi(0, k) = h;
                A.lo(0, k) = __fadd_rn(l, l2);
            }
        }
    }
#pragma unroll
    for (int u = 0; u < IPL; ++u) {
        if (!active[u] || (half && lane >= 16)) continue;
        auto total = [&](int k) {
            if constexpr (is_adjoint(MODE)) {
                if (EQ || k > 2) return A.total(u, k);
                return A.total(u, k) - self_term(K, oi[u].w, k == 0 ? li[u].x : k == 1 ? li[u].y : li[u].z);
            } else if constexpr (MODE == POTENTIAL) {
                // the sum met particle i itself once (d = 0, se = eps exactly): take that term out
                return A.h[u][0] + A.l[u][0] - oi[u].w * pair_potential_of(K.eps, K);
            } else
                return A.h[u][k] + A.l[u][k];
        };
        store_out<MODE>(a, a.perm[ib + il + 32 * u], oi[u], EQ, total);
    }
    return true;
}

// Persistent work-stealing kernel: each warp takes tasks from a global
// counter until none is left.  A task of more than 32 particles runs two i
// particles per lane (four, above 64, in the adjoint), one of at most
// 16 runs each i on two lanes.
// Register budgets: the forward and potential kernels keep 80 registers so that
// 3 CTAs (24 warps) fit an SM; the adjoint's staging needs twice the shared
// memory, which caps it at 2 CTAs, so it may use up to 128 registers.
__host__ __device__ constexpr int min_ctas(int mode) { return is_adjoint(mode) ? 2 : 3; }

// The tasks of one launch, on the equal-mass (EQ) or the general path.
template <int MODE, int JT, int STAGES, bool EQ>
__device__ __forceinline__ void dense_tasks(const KArgs &a, Ring<MODE, JT, STAGES> &ring, float *comp, int lane)
{
    const int ntask = dense_items(a);
    while (true) {
        int t = 0;
        if (lane == 0) t = atomicAdd(a.counter, 1);
        t = __shfl_sync(FULL, t, 0);
        if (t >= ntask) break;
        int4 task;
        if (!take_task(a, a.items[t].x, lane, task)) continue;
        const hacc_volume &vol = a.vols[task.w];
        bool ok = true;
        // sub-chunks of larger tasks: 128 particles (four i per lane) for the adjoint, else 64
        constexpr int CHUNK = is_adjoint(MODE) ? 128 : 64;
        for (int sb = task.y; ok && sb < task.z; sb += CHUNK) {
            const int se = min(sb + CHUNK, task.z);
            if (CHUNK == 128 && se - sb > 64)
                ok = run_task<MODE, JT, STAGES, (CHUNK == 128 ? 4 : 2), EQ>(a, ring, comp, lane, task.x, sb, se,
                                                                             vol);
            else if (se - sb > 32)
                ok = run_task<MODE, JT, STAGES, 2, EQ>(a, ring, comp, lane, task.x, sb, se, vol);
            else
                ok = run_task<MODE, JT, STAGES, 1, EQ>(a, ring, comp, lane, task.x, sb, se, vol);
        }
        if (!ok) {
            if (lane == 0) atomicOr(a.status, HACC_STATUS_TIMEOUT);
            ring.drain();
            return;
        }
    }
}

// The two mass paths share the kernel (the device flag picks one), and the
// hit kernel behind it may start as soon as this one's blocks leave room.
template <int MODE, int JT, int STAGES>
__global__ void __launch_bounds__(256, min_ctas(MODE)) k_pairs(const KArgs a)
{
    allow_next_kernel();
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int WARP_BYTES = warp_smem_bytes(MODE, JT, STAGES);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned char *wbase = smem + (size_t)warp * WARP_BYTES;
    constexpr int TILE_BYTES = warp_tiles_bytes(MODE, JT, STAGES);
    constexpr int COMP_BYTES = is_adjoint(MODE) ? ADJ_COMP_BYTES : 0;
    Ring<MODE, JT, STAGES> ring;
    ring.tiles = reinterpret_cast<float4 *>(wbase);
    float *comp = reinterpret_cast<float *>(wbase + TILE_BYTES);
    ring.bars = reinterpret_cast<uint64_t *>(wbase + TILE_BYTES + COMP_BYTES);

    if (lane == 0) {
        for (int s = 0; s < STAGES; ++s) mbar_init(smem_addr(&ring.bars[s]), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncwarp();
    if constexpr (MODE != POTENTIAL) {
        if (a.mass_varies && *a.mass_varies == 0u) {
            dense_tasks<MODE, JT, STAGES, true>(a, ring, comp, lane);
            return;
        }
    }
    dense_tasks<MODE, JT, STAGES, false>(a, ring, comp, lane);
}

// One hit-mask task (hacc_hits.cuh): at most 32 particles, outputs stored.
template <int MODE>
__device__ __forceinline__ bool hit_task(const KArgs &a, HitWarp &W, int lane, int c, int ib, int ie,
                                         const hacc_volume &vol, bool eq)
{
    HitAcc<MODE> A;
    float4 oi, li;
    int i;
    bool active;
    if (!run_hits<MODE>(a, W.base, W.bar, W.phase, lane, c, ib, ie, vol, eq, false, A, oi, li, i, active)) return false;
    if (active) store_out<MODE>(a, a.perm[i], oi, eq, [&](int k) { return A.total(k); });
    return true;
}

// The tasks of the small cells (the back of the split list), by hit masks.
template <int MODE>
__global__ void __launch_bounds__(HITS_WARPS * 32, hits_ctas(MODE)) k_hits(const KArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    HitWarp W = hits_warp(smem, warp, lane, MODE);
    const bool eq = MODE != POTENTIAL && a.mass_varies && *a.mass_varies == 0u;
    hits_tasks(a, lane, [&](int c, int ib, int ie, const hacc_volume &vol) {
        return hit_task<MODE>(a, W, lane, c, ib, ie, vol, eq);
    });
    wait_previous_kernel();
}

// Ordered pairs (j != i) inside the cutoff, decided exactly as the gather
// force decides it: same offsets, same float32 s + eps, same compare, and the
// image offset added to j for the cells of the hit path, taken from i for the
// dense kernel's (so a pair on the cutoff itself can be counted from one side
// alone).  One warp per task, one i per lane, j read straight from global
// memory: a reporting tool, not a hot path.
__global__ void __launch_bounds__(256)
k_count_pairs(const KArgs a, unsigned long long *__restrict__ total)
{
    const int lane = threadIdx.x & 31;
    const int warps = gridDim.x * (blockDim.x >> 5);
    const int ntask = task_count(a);
    unsigned long long cnt = 0;
    for (int t = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); t < ntask; t += warps) {
        int4 task;
        if (!take_task(a, t, lane, task)) continue;
        const hacc_volume &vol = a.vols[task.w];
        const int n = vol.n;
        const float w = vol.w;
        const double Ld = (double)vol.L;
        const int64_t lc = (int64_t)task.x - vol.cell_base;
        const int cx = (int)(lc % n), cy = (int)((lc / n) % n), cz = (int)(lc / ((int64_t)n * n));
        const float4 org_i = a.origin ? a.origin[task.x] : make_float4(0.f, 0.f, 0.f, 0.f);
        const bool hit = !a.origin && hits_cell(a, task.x, true);
        for (int i = task.y + lane; i - lane < task.z; i += 32) {
            const bool active = i < task.z;
            const float4 oi = active ? a.pos[i] : make_float4(0.f, 0.f, 0.f, 0.f);
            for (int64_t e = a.nbr_off[task.x]; e < a.nbr_off[task.x + 1]; ++e) {
                const int cp = a.nbr_cell[e];
                const int sh = a.nbr_shift[e];
                const int sx = sh % 3 - 1, sy = (sh / 3) % 3 - 1, sz = sh / 9 - 1;
                float Dx, Dy, Dz;
                if (a.origin) {
                    const float4 org_j = a.origin[cp];
                    Dx = (float)((double)org_j.x - (double)org_i.x + sx * Ld);
                    Dy = (float)((double)org_j.y - (double)org_i.y + sy * Ld);
                    Dz = (float)((double)org_j.z - (double)org_i.z + sz * Ld);
                } else {
                    const int64_t lp = (int64_t)cp - vol.cell_base;
                    const int px = (int)(lp % n), py = (int)((lp / n) % n), pz = (int)(lp / ((int64_t)n * n));
                    Dx = (float)((double)cell_centre(px, w) - (double)cell_centre(cx, w) + sx * Ld);
                    Dy = (float)((double)cell_centre(py, w) - (double)cell_centre(cy, w) + sy * Ld);
                    Dz = (float)((double)cell_centre(pz, w) - (double)cell_centre(cz, w) + sz * Ld);
                    if (hit) {
                        Dx = image_delta(cell_centre(px, w), cell_centre(cx, w), (float)sx * vol.L);
                        Dy = image_delta(cell_centre(py, w), cell_centre(cy, w), (float)sy * vol.L);
                        Dz = image_delta(cell_centre(pz, w), cell_centre(cz, w), (float)sz * vol.L);
                    }
                }
                const float oxp = oi.x - Dx, oyp = oi.y - Dy, ozp = oi.z - Dz;
                for (int j = a.cell_start[cp]; j < a.cell_start[cp + 1]; ++j) {
                    const float4 p = a.pos[j];
                    const float dx = hit ? (p.x + Dx) - oi.x : p.x - oxp, dy = hit ? (p.y + Dy) - oi.y : p.y - oyp,
                                dz = hit ? (p.z + Dz) - oi.z : p.z - ozp;
                    const float se = fmaf(dz, dz, fmaf(dy, dy, fmaf(dx, dx, a.k.eps)));
                    cnt += (active && j != i && se < a.k.rc2e) ? 1ull : 0ull;
                }
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_down_sync(FULL, cnt, o);
    if (lane == 0 && cnt) atomicAdd(total, cnt);
}


template <int MODE, int JT, int STAGES>
int launch_t(const KArgs &a, int warps, int ctas_per_sm, cudaStream_t st)
{
    const size_t smem = (size_t)warps * warp_smem_bytes(MODE, JT, STAGES);
    auto kern = k_pairs<MODE, JT, STAGES>;
    if (smem > 48 * 1024)
        HACC_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int occ = 0;
    HACC_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, warps * 32, smem));
    if (occ < 1) return HACC_ERR_INVALID;
    int per_sm = ctas_per_sm < occ ? ctas_per_sm : occ;
    kern<<<num_sms() * per_sm, warps * 32, smem, st>>>(a);
    HACC_LAUNCH_CHECK();
    return HACC_OK;
}

template <int MODE>
int launch_dense(const KArgs &a, const hacc_launch &L, cudaStream_t st)
{
    const int wp = L.warps_per_cta, cps = L.ctas_per_sm;
#define HACC_CASE(JT, S) \
    if (L.jtile == JT && L.stages == S) return launch_t<MODE, JT, S>(a, wp, cps, st);
    HACC_CASE(32, 2) HACC_CASE(32, 4) HACC_CASE(64, 2) HACC_CASE(64, 3) HACC_CASE(64, 4)
    HACC_CASE(128, 2) HACC_CASE(128, 3) HACC_CASE(128, 4) HACC_CASE(256, 2)
#undef HACC_CASE
    return HACC_ERR_INVALID;
}

// Every task: the dense kernel's, then the small cells' by hit masks.
template <int MODE>
int launch_mode(KArgs a, const ForceWs &F, const hacc_launch &L, cudaStream_t st)
{
    int rc = split_tasks(a, F, true, st);
    if (rc) return rc;
    rc = launch_dense<MODE>(a, L, st);
    if (rc || a.origin) return rc;
    return launch_hits(k_hits<MODE>, MODE, st, a);
}

hacc_launch default_launch(int mode)
{
    hacc_launch L;
    L.warps_per_cta = 8;
    L.ctas_per_sm = 3;
    L.jtile = mode == FORCE ? 64 : 64;
    L.stages = 4;
    L.wait_cycles = 0;
    return L;
}

}  // namespace
}  // namespace hacc

using namespace hacc;

extern "C" size_t hacc_force_workspace_size(const hacc_mesh *mesh)
{
    return mesh ? force_layout(mesh, nullptr).total : 0;
}

extern "C" int hacc_sr_force(const hacc_mesh *mesh, const hacc_binned *binned, const hacc_lists *lists,
                             const hacc_sr_params *p, float *ax, float *ay, float *az, const hacc_launch *launch,
                             void *ws, size_t ws_bytes, uint32_t *status, void *stream)
{
    int rc = check_common(mesh, binned, lists, p, launch, ws, ws_bytes, status);
    if (rc) return rc;
    if (mesh->N > 0 && (!ax || !ay || !az)) return HACC_ERR_INVALID;
    if (mesh->N == 0) return HACC_OK;
    cudaStream_t st = as_stream(stream);
    ForceWs F = force_layout(mesh, ws);
    KArgs a = base_args(mesh, binned, lists, p, status);
    a.out_x = ax;
    a.out_y = ay;
    a.out_z = az;
    hacc_launch L = launch ? *launch : default_launch(FORCE);
    a.wait_limit = wait_limit_of(L);
    return launch_mode<FORCE>(a, F, L, st);
}

extern "C" int hacc_sr_force_adjoint(const hacc_mesh *mesh, const hacc_binned *binned, const hacc_lists *lists,
                                     const hacc_sr_params *p, const float *gax, const float *gay,
                                     const float *gaz, float *gx, float *gy, float *gz, float *gm,
                                     const hacc_launch *launch, void *ws, size_t ws_bytes, uint32_t *status,
                                     void *stream)
{
    int rc = check_common(mesh, binned, lists, p, launch, ws, ws_bytes, status);
    if (rc) return rc;
    if (mesh->N > 0 && (!gax || !gay || !gaz || !gx || !gy || !gz)) return HACC_ERR_INVALID;
    if (mesh->N == 0) return HACC_OK;
    cudaStream_t st = as_stream(stream);
    ForceWs F = force_layout(mesh, ws);
    int g = (int)((mesh->N + 255) / 256);
    if (g > num_sms() * 16) g = num_sms() * 16;
    k_gather_lam<<<g, 256, 0, st>>>(mesh->N, binned->perm, gax, gay, gaz, F.lam);
    HACC_LAUNCH_CHECK();
    KArgs a = base_args(mesh, binned, lists, p, status);
    a.lam = F.lam;
    a.out_x = gx;
    a.out_y = gy;
    a.out_z = gz;
    a.out_m = gm;
    hacc_launch L = launch ? *launch : default_launch(ADJOINT);
    a.wait_limit = wait_limit_of(L);
    if (gm) return launch_mode<ADJOINT_GM>(a, F, L, st);
    return launch_mode<ADJOINT>(a, F, L, st);
}

extern "C" int hacc_sr_potential(const hacc_mesh *mesh, const hacc_binned *binned, const hacc_lists *lists,
                                 const hacc_sr_params *p, float *phi, const hacc_launch *launch, void *ws,
                                 size_t ws_bytes, uint32_t *status, void *stream)
{
    int rc = check_common(mesh, binned, lists, p, launch, ws, ws_bytes, status);
    if (rc) return rc;
    if (mesh->N > 0 && !phi) return HACC_ERR_INVALID;
    if (mesh->N == 0) return HACC_OK;
    cudaStream_t st = as_stream(stream);
    ForceWs F = force_layout(mesh, ws);
    KArgs a = base_args(mesh, binned, lists, p, status);
    a.out_x = phi;
    hacc_launch L = launch ? *launch : default_launch(FORCE);
    a.wait_limit = wait_limit_of(L);
    return launch_mode<POTENTIAL>(a, F, L, st);
}

extern "C" int hacc_count_pairs(const hacc_mesh *mesh, const hacc_binned *binned, const hacc_lists *lists,
                                const hacc_sr_params *p, int64_t *out, void *stream)
{
    if (!mesh || !binned || !lists || !p || !out || !mesh->vols) return HACC_ERR_INVALID;
    if (!(p->eps > 0.0f) || !(p->rcut > 0.0f)) return HACC_ERR_INVALID;
    if (!binned->cell_start || !lists->nbr_off || !lists->tasks || !lists->n_tasks) return HACC_ERR_INVALID;
    if (mesh->N > 0 && !binned->sorted4) return HACC_ERR_INVALID;
    cudaStream_t st = as_stream(stream);
    HACC_CUDA_TRY(cudaMemsetAsync(out, 0, sizeof(int64_t), st));
    if (mesh->N == 0) return HACC_OK;
    KArgs a = base_args(mesh, binned, lists, p, nullptr);
    k_count_pairs<<<num_sms() * 8, 256, 0, st>>>(a, reinterpret_cast<unsigned long long *>(out));
    HACC_LAUNCH_CHECK();
    return HACC_OK;
}

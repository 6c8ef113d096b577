// Device helpers shared by the Newton-III symmetric kernels (force and
// adjoint, two translation units): the empty-lane position, the list entry
// of a cell itself and the image offset of a list entry.
#pragma once

#include "hacc_hits.cuh"

namespace hacc {
namespace {

// Position of an empty lane: every pair with it fails the cutoff test.
constexpr float FAR = 1.0e6f;

// Image offset Delta of one list entry: origin of cell (leaf) cp shifted by
// the image, minus the origin of c; float64, rounded once.
__device__ __forceinline__ void entry_delta(const KArgs &a, const hacc_volume &vol, int cp, int sh, int cx, int cy,
                                            int cz, const float4 &org_i, float &Dx, float &Dy, float &Dz)
{
    const double Ld = (double)vol.L;
    const int sx = sh % 3 - 1, sy = (sh / 3) % 3 - 1, sz = sh / 9 - 1;
    if (a.origin) {
        const float4 org_j = a.origin[cp];
        Dx = (float)((double)org_j.x - (double)org_i.x + sx * Ld);
        Dy = (float)((double)org_j.y - (double)org_i.y + sy * Ld);
        Dz = (float)((double)org_j.z - (double)org_i.z + sz * Ld);
    } else {
        const int n = vol.n;
        const float w = vol.w;
        const int64_t lp = (int64_t)cp - vol.cell_base;
        const int px = (int)(lp % n), py = (int)((lp / n) % n), pz = (int)(lp / ((int64_t)n * n));
        // exact in float64: origins are the float32 cell centres used by the binning
        Dx = (float)((double)cell_centre(px, w) - (double)cell_centre(cx, w) + sx * Ld);
        Dy = (float)((double)cell_centre(py, w) - (double)cell_centre(cy, w) + sy * Ld);
        Dz = (float)((double)cell_centre(pz, w) - (double)cell_centre(cz, w) + sz * Ld);
    }
}

// Lane's entry of a group (first record jb, cnt of them) clipped to the
// segment's j records of the task's flattened list.  before: the records of
// the groups before, brought up to date.  size: the task's particles.  False
// once the segment has ended.
__device__ __forceinline__ bool clip_entry(const KArgs &a, int lane, int code, int size, int &before, int &jb, int &cnt)
{
    int inc = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(FULL, inc, o);
        if (lane >= o) inc += t;
    }
    const int per = segment_records(a, size) << ((code >> 16) & 31), jlo = (code & 0xffff) * per;
    const int first = before + inc - cnt;
    before += __shfl_sync(FULL, inc, 31);
    const int lo = max(first, jlo), hi = code >> 24 ? first + cnt : min(first + cnt, jlo + per);
    jb += lo - first;
    cnt = max(hi - lo, 0);
    return code >> 24 || __shfl_sync(FULL, first, 0) < jlo + per;
}

// Without dense tasks (n_dense given and 0) the hit kernel stores every
// task's outputs itself: the totals are then neither zeroed nor converted.
__device__ __forceinline__ bool no_totals(const int32_t *n_dense) { return n_dense && *n_dense == 0; }

struct TotalsOut {
    float *out[4];
};

// Zeroes the totals or, when the hit kernel stores, the outputs: a particle
// whose task was dropped (a task buffer too small, a wait that ran out) reads
// 0 on both ways.
__global__ void __launch_bounds__(256)
k_zero_totals(double2 *__restrict__ acc, int64_t n2, const int32_t *__restrict__ n_dense, TotalsOut o, int nc, int64_t N)
{
    const int64_t k0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
    if (no_totals(n_dense)) {
        for (int c = 0; c < nc; ++c)
            for (int64_t k = k0; k < N; k += step) o.out[c][k] = 0.0f;
        return;
    }
    for (int64_t k = k0; k < n2; k += step) acc[k] = make_double2(0.0, 0.0);
}

// Zeroes nc totals per particle (the region holds SYM_ACC_MAX of them).
int zero_totals(const KArgs &a, double *acc, float *const (&out)[4], int nc, const int32_t *n_dense, cudaStream_t st)
{
    const int64_t n2 = (a.N * nc + 1) / 2;
    int64_t g = (n2 + 255) / 256;
    if (g > num_sms() * 16) g = num_sms() * 16;
    const TotalsOut o{{out[0], out[1], out[2], out[3]}};
    k_zero_totals<<<(int)g, 256, 0, st>>>(reinterpret_cast<double2 *>(acc), n2, n_dense, o, nc, a.N);
    HACC_LAUNCH_CHECK();
    return HACC_OK;
}

// Output components [c0, c1) from their float64 totals (sorted slots), float32
// in input order; the adjoints' dL/dx = W times the common mass when the masses
// are equal (mass_varies given and 0), and their component 3, dL/dm = -G.
// The stores scatter through the permutation, 4 bytes each; they merge into
// whole sectors in L2 only while the target array stays resident there, which
// one 67 MB component of 16.8M particles per launch does and three at once do
// not (each partial sector is then read and written back in DRAM: 0.82 against
// 0.33 ms).  The streamed totals and perm are loaded evict-first for the same
// reason.
__global__ void __launch_bounds__(256)
k_finish_totals(int64_t N, const double *__restrict__ acc, const int32_t *__restrict__ perm,
                const float4 *__restrict__ pos, const uint32_t *mass_varies,
                const int32_t *__restrict__ n_dense, TotalsOut o, int c0, int c1)
{
    if (no_totals(n_dense)) return;
    const double w = mass_varies && *mass_varies == 0u ? (double)pos[0].w : 1.0;
    for (int c = c0; c < c1; ++c) {
        const double sc = c == 3 ? -1.0 : w;
        for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < N; k += (int64_t)gridDim.x * blockDim.x)
            o.out[c][__ldcs(perm + k)] = (float)(sc * __ldcs(acc + c * N + k));
    }
}

// One launch for all components while they fit the L2 together (4M particles:
// 67 MB), else one each.
int finish_totals(const KArgs &a, const double *acc, const int32_t *n_dense, float *const (&out)[4], int nc,
                  const uint32_t *mass_varies, cudaStream_t st)
{
    int64_t g = (a.N + 255) / 256;
    if (g > num_sms() * 16) g = num_sms() * 16;
    const TotalsOut o{{out[0], out[1], out[2], out[3]}};
    const int step = a.N <= ((int64_t)4 << 20) ? nc : 1;
    for (int c = 0; c < nc; c += step) {
        k_finish_totals<<<(int)g, 256, 0, st>>>(a.N, acc, a.perm, a.pos, mass_varies, n_dense, o, c, c + step);
        HACC_LAUNCH_CHECK();
    }
    return HACC_OK;
}

// m (h + l) rounded once, as the float64 totals' way rounds it, by an exact
// float32 product (2.1M lattice particles: a step takes 1228 us, 1246 with
// float64 products here, whose pipe is narrow).
__device__ __forceinline__ float product_once(float m, float h, float l)
{
    const float p = __fmul_rn(m, h), e = __fmaf_rn(m, h, -p);
    return isfinite(p) ? __fadd_rn(p, __fmaf_rn(m, l, e)) : p;
}

// One hit-mask task of a symmetric call (the small cells' pairs): its totals
// are stored (no dense tasks) or added to the float64 totals, to which dense
// tasks add the pairs with their cells.
template <int MODE>
__device__ __forceinline__ bool hit_task_sym(const KArgs &a, HitWarp &W, int lane, int c, int ib, int ie,
                                             const hacc_volume &vol, double *acc, bool eq, bool store)
{
    HitAcc<MODE> A;
    float4 oi, li;
    int i;
    bool active;
    if (!run_hits<MODE>(a, W.base, W.bar, W.phase, lane, c, ib, ie, vol, eq, true, A, oi, li, i, active))
        return false;
    if (!active) return true;
    if (store) {
        const float m = eq ? oi.w : 1.0f;
        const int o = a.perm[i];
        a.out_x[o] = product_once(m, A.h[0], A.l[0]);
        a.out_y[o] = product_once(m, A.h[1], A.l[1]);
        a.out_z[o] = product_once(m, A.h[2], A.l[2]);
        if constexpr (MODE == ADJOINT_GM) a.out_m[o] = -A.total(3);
    } else {
        // the force's totals hold the mass, the adjoint's are scaled by the finishing pass
        const double m = MODE == FORCE && eq ? (double)oi.w : 1.0;
#pragma unroll
        for (int k = 0; k < HitAcc<MODE>::NC; ++k)
            atomicAdd(acc + k * a.N + i, m * ((double)A.h[k] + (double)A.l[k]));
    }
    return true;
}

template <int MODE>
__global__ void __launch_bounds__(HITS_WARPS * 32, hits_ctas(MODE)) k_hits_sym(const KArgs a, double *acc)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    HitWarp W = hits_warp(smem, warp, lane, MODE);
    const bool eq = a.mass_varies && *a.mass_varies == 0u, store = no_totals(a.n_items);
    hits_tasks(a, lane, [&](int c, int ib, int ie, const hacc_volume &vol) {
        return hit_task_sym<MODE>(a, W, lane, c, ib, ie, vol, acc, eq, store);
    });
    wait_previous_kernel();
}

}  // namespace
}  // namespace hacc

// Many steps of a small grid in one launch.
//
// A grid of up to 256^3 cells stays in the 129 MB L2 between its steps, so
// what bounds it is not HBM but launches (about 4 us each), the 0.9 us that a
// z-march CTA needs per plane, and CTAs too few to fill the chip (64^3 cells
// are 16 tiles of the z-march kernel).  gs_resident_kernel spreads the cells
// over one CTA per SM, one 16-byte group per thread and turn, all loads of a
// group independent, and runs all steps of a call with a grid barrier (about
// 1.3 us) between two steps.
//
// us per step, default plan, noise 0.1, calls of 100 steps (before: z-march
// 128 x 8 x 32 launches for FP32, 64 x 8 x 32 for FP64; below: this kernel):
//   FP32  L = 32: 28.8 -> 1.8   64: 30.9 -> 2.2   96: 30.9 -> 3.9
//         L = 128: 33.0 -> 6.4  160: 34.9 -> 10.4  200: 41.4 -> 25  256: 53.3 -> 48
//   FP64  L = 64: 119 -> 13.4   128: 121 -> 93.7   256: 744 -> 736 (FP64 pipe)
// Measured and not taken: columns marched in z with register planes (fewer
// loads, but fewer groups in flight: 64^3 2.7, 128^3 7.2 us), and x neighbours
// from adjacent lanes (2.4 and 6.7 us: the shuffles wait for the loads).
#include <algorithm>

#include "gs_common.cuh"
#include "gs_internal.h"

namespace gs {

template <typename T>
struct ResArgs {
    T *u0, *v0;         // the set holding the state before the first step
    T *u1, *v1;         // the other set
    int L, ny, nz;      // bricks: ny ranges of rows times nz ranges of planes (ny = 0: runs of rows)
    int n;              // steps
    int64_t t;          // step index of the first one
    uint64_t seed;
    GsCoef<T> c;
    unsigned* bar;      // [arrivals, CTAs done], zero between launches
    int* err;
    uint64_t timeout_ns;
};

// V cells of one 16-byte vector, or one cell (V = 1: edges L that are no
// multiple of the vector)
template <typename T, int V>
GS_D void res_load(const T* p, T* r)
{
    if constexpr (V == 1) r[0] = *p;
    else gs_unpack<T>(*reinterpret_cast<const typename GsVec<T>::type*>(p), r);
}

template <typename T, int V>
GS_D void res_store(T* p, const T* r)
{
    if constexpr (V == 1) *p = r[0];
    else *reinterpret_cast<typename GsVec<T>::type*>(p) = gs_pack<T>(r);
}

template <typename T, int V, bool NOISE, bool HELD, int MAXT>
__global__ void __launch_bounds__(MAXT, 1) gs_resident_kernel(const ResArgs<T> a)
{
    const int L = a.L, nxv = L / V, LL = L * L;
    const int tid = threadIdx.x;
    // this CTA's rows: a brick (a y range times a z range), or with ny = 0 a
    // run of the rows in (y, z) order; either way rows ylo..yhi-1 of plane
    // after plane from (ys, zs) on, nrow of them
    int ylo = 0, yhi = L, ys, zs, nrow;
    if (a.ny) {
        const int by = blockIdx.x % a.ny, bz = blockIdx.x / a.ny;
        ylo = L * by / a.ny;
        yhi = L * (by + 1) / a.ny;
        ys = ylo;
        zs = L * bz / a.nz;
        nrow = (yhi - ylo) * (L * (bz + 1) / a.nz - zs);
    } else {
        const int r0 = (int)((long long)LL * blockIdx.x / gridDim.x);
        nrow = (int)((long long)LL * (blockIdx.x + 1) / gridDim.x) - r0;
        zs = r0 / L;
        ys = r0 - zs * L;
    }
    const int nr = yhi - ylo, ng = nrow * nxv;
    // this thread's first group (x fastest, then y, then z) and the step to
    // its next one as (x, y, z) increments
    const int r0 = tid / nxv, xv0 = tid - r0 * nxv;
    const int dr = blockDim.x / nxv, dxv = blockDim.x - dr * nxv;
    const int q0 = ys - ylo + r0, dz = dr / nr, dy = dr - dz * nr;
    const int z00 = zs + q0 / nr, y00 = ylo + q0 % nr;
    bool stop = false;
    for (int s = 0; s < a.n && !stop; ++s) {
        const GsKeys k = NOISE ? gs_step_keys(a.seed, a.t + s) : GsKeys{0, 0};
        const uint32_t kk2 = gs_kk2(k);
        const bool even = (s & 1) == 0;
        // no __restrict__: another CTA writes what this one reads a step later
        const T* u = even ? a.u0 : a.u1;
        const T* v = even ? a.v0 : a.v1;
        T* un = even ? a.u1 : a.u0;
        T* vn = even ? a.v1 : a.v0;
        int xv = xv0, y = y00, z = z00;
        for (int g = tid; g < ng; g += blockDim.x) {
            // 32-bit indices: L <= 256
            const int x = xv * V, row = (z * L + y) * L, i = row + x;
            const int iym = y == 0 ? i + LL - L : i - L;
            const int iyp = y == L - 1 ? i - (LL - L) : i + L;
            const int izm = z == 0 ? i + (L - 1) * LL : i - LL;
            const int izp = z == L - 1 ? i - (L - 1) * LL : i + LL;
            const int ixl = x == 0 ? row + L - 1 : i - 1;
            const int ixr = x + V == L ? row : i + V;
            T cu[V], cv[V], pu[V], pv[V], nu[V], nv[V], ymu[V], ypu[V], ymv[V], ypv[V], ou[V], ov[V];
            res_load<T, V>(u + i, cu);
            res_load<T, V>(u + iym, ymu);
            res_load<T, V>(u + iyp, ypu);
            res_load<T, V>(u + izm, pu);
            res_load<T, V>(u + izp, nu);
            res_load<T, V>(v + i, cv);
            res_load<T, V>(v + iym, ymv);
            res_load<T, V>(v + iyp, ypv);
            res_load<T, V>(v + izm, pv);
            res_load<T, V>(v + izp, nv);
            const T xlu = u[ixl], xru = u[ixr], xlv = v[ixl], xrv = v[ixr];
            if constexpr (V == 1) {
                const T su = gs_nsum(xlu, xru, ymu[0], ypu[0], pu[0], nu[0]);
                const T sv = gs_nsum(xlv, xrv, ymv[0], ypv[0], pv[0], nv[0]);
                gs_update<T, NOISE>(a.c, cu[0], cv[0], su, sv, NOISE ? (T)gs_noise_num((uint32_t)i, k) : (T)0, ou[0],
                                    ov[0]);
            } else {
                const uint32_t pre = NOISE ? gs_group_pre((uint32_t)i, k) : 0u;
                gs_update_group<T, NOISE>(a.c, pre, kk2, cu, cv, pu, pv, nu, nv, ymu, ypu, ymv, ypv, xlu, xru, xlv, xrv,
                                          ou, ov);
            }
            if (HELD) {
                const bool face = y == 0 || y == L - 1 || z == 0 || z == L - 1;
#pragma unroll
                for (int e = 0; e < V; ++e)
                    if (face || (e == 0 && x == 0) || (e == V - 1 && x + V == L)) {
                        ou[e] = cu[e];
                        ov[e] = cv[e];
                    }
            }
            res_store<T, V>(un + i, ou);
            res_store<T, V>(vn + i, ov);
            xv += dxv;
            y += dy;
            z += dz;
            if (xv >= nxv) { xv -= nxv; ++y; }
            if (y >= yhi) { y -= nr; ++z; }
        }
        if (s + 1 == a.n) break;
        // grid barrier: the CTA's stores are ordered before its arrival (the
        // barrier makes them thread 0's predecessors), every other CTA's
        // before thread 0's acquire, and that before this CTA's next loads
        __syncthreads();
        int bad = 0;
        if (tid == 0) {
            gs_red_add_release_gpu(a.bar, 1u);
            const unsigned want = (unsigned)(s + 1) * gridDim.x;
            if ((int)(gs_ld_acquire_gpu(a.bar) - want) < 0) {
                const uint64_t t0 = gs_globaltimer();
                while ((int)(gs_ld_acquire_gpu(a.bar) - want) < 0)
                    if (gs_globaltimer() - t0 > a.timeout_ns) {
                        gs_report(a.err, GS_DERR_TIMEOUT);
                        bad = 1;
                        break;
                    }
            }
        }
        stop = __syncthreads_or(bad);
    }
    // the last CTA to finish zeroes both words for the next launch
    if (a.n > 1 && tid == 0) {
        __threadfence();
        if (atomicAdd(&a.bar[1], 1u) == gridDim.x - 1) {
            a.bar[0] = 0;
            a.bar[1] = 0;
        }
    }
}

// Footprint (both buffer sets) up to which the loads are L2 hits throughout.
static constexpr long long kL2Fit = 96ll << 20;

template <typename T, int V, bool NOISE, bool HELD>
static int resident_launch_t(int L, void* const u[2], void* const v[2], int n, const Params& p, int64_t t,
                             unsigned* bar, int* err, uint64_t timeout_ns, cudaStream_t s)
{
    const int nxv = L / V;
    const long long rows_all = (long long)L * L;
    ResArgs<T> a;
    a.u0 = (T*)u[0];
    a.v0 = (T*)v[0];
    a.u1 = (T*)u[1];
    a.v1 = (T*)v[1];
    a.L = L;
    // one CTA per SM, but at least 128 groups each (fewer gain nothing)
    const int cap = (int)std::min<long long>(num_sms(), std::max<long long>(1, rows_all * nxv / 128));
    int grid, rows;
    if (V == 4) {
        // bricks with the smallest largest one, then the smallest halo: the
        // neighbouring rows a CTA shares come from its L1 (256^3: 48 us
        // against 72 us with runs of rows)
        int best = 0;
        grid = rows = a.ny = a.nz = 1;
        for (int ny = 1; ny <= L && ny <= cap; ++ny) {
            const int nz = std::min(L, cap / ny);
            const int h = (L + ny - 1) / ny, d = (L + nz - 1) / nz;
            const int cost = h * d * 1024 + (h + 2) * (d + 2);
            if (best && cost >= best) continue;
            best = cost;
            a.ny = ny;
            a.nz = nz;
            rows = h * d;
        }
        grid = a.ny * a.nz;
    } else {
        // runs of rows in memory order, equal to within one row: the FP64 pipe
        // (or the scalar loads of V = 1) bounds the step, and bricks leave SMs
        // idle (FP64 64^3 without noise: 12.2 us against 13.3 us)
        grid = (int)std::min<long long>(cap, rows_all);
        rows = (int)((rows_all + grid - 1) / grid);
        a.ny = a.nz = 0;
    }
    // 512 threads of up to 128 registers while the fields fit L2; beyond that,
    // and with scalar loads, latency wants the 1024 (FP32 160^3: 10.4 against
    // 11.4 us; 192^3: 25.0 against 19.8 us; 101^3: 8.2 against 6.4 us)
    const bool wide = V == 1 || 4 * (long long)sizeof(T) * L * rows_all > kL2Fit;
    const int maxt = wide ? 1024 : 512;
    const int ng = nxv * rows, turns = (ng + maxt - 1) / maxt;
    const int threads = ((ng + turns - 1) / turns + 31) / 32 * 32;
    a.n = n;
    a.t = t;
    a.seed = p.seed;
    a.c = gs_make_coef<T>(p.Du, p.Dv, p.F, p.k, p.dt, p.noise);
    a.bar = bar;
    a.err = err;
    a.timeout_ns = timeout_ns;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeCooperative;  // co-residency for the grid barrier (none in a single step)
    at.val.cooperative = 1;
    cfg.attrs = &at;
    cfg.numAttrs = n > 1 ? 1 : 0;
    void (*kern)(const ResArgs<T>) = gs_resident_kernel<T, V, NOISE, HELD, 1024>;
    if constexpr (V > 1) {
        if (!wide) kern = gs_resident_kernel<T, V, NOISE, HELD, 512>;
    }
    GS_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, a));
    return GS_OK;
}

// Up to 256^3 this kernel is the faster one, or (FP64) as fast as the others;
// above, the fields leave L2 and the z-march kernel's fewer loads win (FP32
// 320^3: 92 against 90 us; 384^3: 245 against 143 us).
bool resident_supported(int L) { return L <= 256; }

int launch_resident(int dtype, int L, void* const u[2], void* const v[2], int n, const Params& p, bool held, int64_t t,
                    unsigned* bar, int* err, uint64_t timeout_ns, cudaStream_t s)
{
    const bool noise = p.noise != 0.0;
#define GS_RES(T, V)                                                                                                   \
    return noise ? (held ? resident_launch_t<T, V, true, true>(L, u, v, n, p, t, bar, err, timeout_ns, s)              \
                         : resident_launch_t<T, V, true, false>(L, u, v, n, p, t, bar, err, timeout_ns, s))            \
                 : (held ? resident_launch_t<T, V, false, true>(L, u, v, n, p, t, bar, err, timeout_ns, s)             \
                         : resident_launch_t<T, V, false, false>(L, u, v, n, p, t, bar, err, timeout_ns, s))
    if (dtype == GS_F32) {
        if (L % 4 == 0) GS_RES(float, 4);
        GS_RES(float, 1);
    }
    if (L % 2 == 0) GS_RES(double, 2);
    GS_RES(double, 1);
#undef GS_RES
}

}  // namespace gs

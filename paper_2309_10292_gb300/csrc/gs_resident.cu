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
//   FP32  L = 32: 28.8 -> 1.8   64: 30.9 -> 2.2   96: 30.9 -> 3.3
//         L = 128: 33.0 -> 5.4  160: 34.9 -> 9.9  192: 41 -> 18.5  256: 53.3 -> 48.8
//         (from the plain kernel) L = 150: 28.9 -> 11.5   101: 12.4 -> 6.4
//   FP64  L = 64: 119 -> 12.9   128: 121 -> 89.7   256: 744 -> 703 (FP64 pipe)
//   FP64 in fixed point with a remainder  L = 64: 29.5 -> 3.7   128: 29.5 -> 14.8
//   FP64 in double-single  L = 128: 23.2, in fixed point 25.3
// Measured and not taken: columns marched in z with register planes (fewer
// loads, but fewer groups in flight: 64^3 2.7, 128^3 7.2 us), and x neighbours
// from adjacent lanes (2.4 and 6.7 us: the shuffles wait for the loads).
#include <algorithm>

#include "gs_common.cuh"
#include "gs_internal.h"
#include "gs_resident.cuh"

namespace gs {

template <typename T, int AR>
struct ResArgs {
    T *u0, *v0;         // the set holding the state before the first step
    T *u1, *v1;         // the other set
    int L, ny, nz;      // bricks: ny ranges of rows times nz ranges of planes (ny = 0: runs of rows)
    int n;              // steps
    int64_t t;          // step index of the first one
    uint64_t seed;
    ResCoef<T, AR> c;
    int io;             // AR > 0: bit 0 the input holds packed values, bit 1 write packed values
    unsigned* bar;      // [arrivals, CTAs done], zero between launches
    int* err;
    uint64_t timeout_ns;
};

// AR > 0 (FP64 fields): the fields are converted to packed values in
// place before the first step, stay packed between the steps, and the last
// step writes FP64 values (a call of several launches converts only at its
// ends, see io).  With CONV they are converted at every load and store.
template <typename T, int V, bool NOISE, bool HELD, int AR, bool CONV, bool SHELL, int MAXT>
__global__ void __launch_bounds__(MAXT, 1) gs_resident_kernel(const ResArgs<T, AR> a)
{
    const int L = a.L, tid = threadIdx.x;
    // this CTA's rows: a brick (a y range times a z range), or with ny = 0 a
    // run of the rows in memory order
    ResRows r{L, 0, L, 0, 0, 0};
    if (a.ny) {
        const int by = blockIdx.x % a.ny, bz = blockIdx.x / a.ny;
        r.ylo = L * by / a.ny;
        r.yhi = L * (by + 1) / a.ny;
        r.ys = r.ylo;
        r.zs = L * bz / a.nz;
        r.nrow = (r.yhi - r.ylo) * (L * (bz + 1) / a.nz - r.zs);
    } else {
        const long long LL = (long long)L * L;
        const int r0 = (int)(LL * blockIdx.x / gridDim.x);
        r.nrow = (int)(LL * (blockIdx.x + 1) / gridDim.x) - r0;
        r.zs = r0 / L;
        r.ys = r0 - r.zs * L;
    }
    const ResWalk<V> w(r, tid);
    [[maybe_unused]] const ResShell q = res_shell(r);
    unsigned met = 0;  // barriers passed
    auto meet = [&]() { return res_grid_sync(a.bar, ++met * gridDim.x, a.err, a.timeout_ns); };
    bool stop = false, in_range = true;
    if constexpr (AR > 0 && !CONV) {
        if (!(a.io & 1)) {
            in_range = res_pack_rows<V, AR>(r, w, a.u0, a.v0, tid);
            stop = meet();
        }
    }
    for (int s = 0; s < a.n && !stop; ++s) {
        const GsKeys k = NOISE ? gs_step_keys(a.seed, a.t + s) : GsKeys{0, 0};
        const bool even = (s & 1) == 0, last = s + 1 == a.n;
        const T *u = even ? a.u0 : a.u1, *v = even ? a.v0 : a.v1;
        T *un = even ? a.u1 : a.u0, *vn = even ? a.v1 : a.v0;
        const bool unpack = AR > 0 && last && !(a.io & 2);
        uint32_t rng;
        if constexpr (SHELL) {
            // the rows that other CTAs read, the arrival, the rest under it: a
            // CTA that passes the barrier reads the new state of the former
            // only, and overwrites old values that only its own rows needed
            int2 g = make_int2(tid / (L / V), tid % (L / V));
            rng = res_shell_rows<T, V, NOISE, HELD, AR, CONV>(q, g, q.nb, u, v, un, vn, a.c, k, unpack);
            if (!last) res_grid_arrive(a.bar);
            rng |= res_shell_rows<T, V, NOISE, HELD, AR, CONV>(q, g, r.nrow, u, v, un, vn, a.c, k, unpack);
        } else {
            rng = res_rows<T, V, NOISE, HELD, AR, CONV>(r, w, u, v, un, vn, a.c, k, tid, unpack);
        }
        if (AR == 3) in_range &= !fxf_range_bad(rng);
        if (AR == 2 && CONV) in_range &= rng == 0;
        if (!last) stop = SHELL ? res_grid_wait(a.bar, ++met * gridDim.x, a.err, a.timeout_ns) : meet();
    }
    if (AR >= 2 && !in_range) gs_report(a.err, GS_DERR_RANGE);
    // the last CTA to finish zeroes both words for the next launch
    if (met && tid == 0) {
        __threadfence();
        if (atomicAdd(&a.bar[1], 1u) == gridDim.x - 1) {
            a.bar[0] = 0;
            a.bar[1] = 0;
        }
    }
}

template <typename T, int AR>
static ResCoef<T, AR> res_coef(const Params& p)
{
    if constexpr (AR == 0) return gs_make_coef<T>(p.Du, p.Dv, p.F, p.k, p.dt, p.noise);
    if constexpr (AR == 1) return gs_make_coef_ds(p.Du, p.Dv, p.F, p.k, p.dt, p.noise);
    if constexpr (AR == 2) return gs_make_coef_fx(p.Du, p.Dv, p.F, p.k, p.dt, p.noise);
    if constexpr (AR == 3) return gs_make_coef_fxf(p.Du, p.Dv, p.F, p.k, p.dt, p.noise);
}

// Whether a brick steps its inner rows under the barrier.  us per step without
// and with: FP32 64^3 2.26 / 2.29, 80^3 3.09 / 2.45, 96^3 3.89 / 3.32, 128^3 6.44 /
// 5.40, 192^3 20.1 / 18.5, 256^3 48.8 / 48.9 (without noise 46.1 / 47.6, held 54.3 /
// 49.4); fixed point with a remainder 64^3 3.84 / 3.77, 80^3 5.74 / 4.87, 128^3
// 15.4 / 15.1, 140^3 21.7 / 21.3, 160^3 35.6 / 36.4; fixed point 64^3 5.35 / 5.37,
// 72^3 7.12 / 6.66, 128^3 26.2 / 25.3, 140^3 36.0 / 36.0; double-single 64^3 4.61 /
// 4.69, 72^3 6.53 / 5.98, 112^3 16.8 / 16.4, 128^3 21.0 / 21.2.  Held, converting at
// every load: 64^3 13.0 / 13.4 (double-single), 72^3 19.6 / 21.0 (fixed point), with
// a remainder 15.7 / 15.3, 80^3 22.0 / 21.4, 25.5 / 24.8, with a remainder 20.3 / 19.1.
static bool shell_pays(int arith, int dtype_bytes, int L, bool held)
{
    if (dtype_bytes == 4) return L >= 72 && (held || L <= 224);
    if (held) return L > (arith == GS_ARITH_FXF ? 64 : 72);
    return L >= (arith == GS_ARITH_FXF ? 64 : 68) && L <= (arith == GS_ARITH_DS ? 120 : 140);
}

template <typename T, int V, bool NOISE, bool HELD, int AR, bool CONV = (AR > 0 && HELD)>
static int resident_launch_t(int L, void* const u[2], void* const v[2], int n, const Params& p, int64_t t,
                             unsigned* bar, int* err, uint64_t timeout_ns, cudaStream_t s)
{
    const int nxv = L / V;
    const long long rows_all = (long long)L * L;
    ResArgs<T, AR> a;
    a.u0 = (T*)u[0];
    a.v0 = (T*)v[0];
    a.u1 = (T*)u[1];
    a.v1 = (T*)v[1];
    a.L = L;
    // one CTA per SM, but at least 128 groups each (fewer gain nothing)
    const int cap = (int)std::min<long long>(num_sms(), std::max<long long>(1, rows_all * nxv / 128));
    int grid, rows;
    if (V == 4 || (V == 2 && AR > 0)) {
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
        // (or the narrow loads of V < 4) bounds the step, and bricks leave SMs
        // idle (IEEE FP64 64^3 without noise: 12.2 us against 13.3 us)
        grid = (int)std::min<long long>(cap, rows_all);
        rows = (int)((rows_all + grid - 1) / grid);
        a.ny = a.nz = 0;
    }
    // 512 threads of up to 128 registers while the fields fit L2; beyond that,
    // and with narrow loads, latency wants the 1024 (FP32 160^3: 10.4 against
    // 11.4 us; 192^3: 25.0 against 19.8 us; 101^3: 8.2 against 6.4 us)
    const bool wide = V < GsVec<T>::N || 4 * (long long)sizeof(T) * L * rows_all > kResL2Fit;
    const int maxt = wide ? 1024 : 512;
    const int ng = nxv * rows, turns = (ng + maxt - 1) / maxt;
    const int threads = ((ng + turns - 1) / turns + 31) / 32 * 32;
    a.n = n;
    a.t = t;
    a.seed = p.seed;
    a.c = res_coef<T, AR>(p);
    a.io = p.io;
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
    cfg.numAttrs = n > 1 || (AR > 0 && !CONV && !(p.io & 1)) ? 1 : 0;
    void (*kern)(const ResArgs<T, AR>);
    if constexpr (CONV && !HELD) {
        kern = gs_resident_kernel<T, V, NOISE, HELD, AR, CONV, false, 512>;  // (one step of at most 80^3 cells)
    } else {
        kern = gs_resident_kernel<T, V, NOISE, HELD, AR, CONV, false, 1024>;
        if constexpr (V > 1) {
            if (!wide) kern = gs_resident_kernel<T, V, NOISE, HELD, AR, CONV, false, 512>;
        }
        if constexpr (V == GsVec<T>::N && (sizeof(T) == 4 || AR > 0)) {
            if (a.ny && n > 1 && shell_pays(AR, sizeof(T), L, HELD))
                kern = wide ? gs_resident_kernel<T, V, NOISE, HELD, AR, CONV, true, 1024>
                            : gs_resident_kernel<T, V, NOISE, HELD, AR, CONV, true, 512>;
        }
    }
    // (a graph's launch does not report a cooperative kernel that cannot be
    // resident, and never ends)
    if (cfg.numAttrs && captured_on_part(s)) return kResidentTooLarge;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, a);
    if (e == cudaErrorCooperativeLaunchTooLarge) {
        // (a context that may use part of the SMs only)
        cudaGetLastError();
        return kResidentTooLarge;
    }
    GS_CUDA_TRY(e);
    return GS_OK;
}

// Up to 256^3 this kernel is the faster one, or (IEEE FP64) as fast as the
// others; above, the fields leave L2 and the z-march kernel's fewer loads win
// (FP32 320^3: 92 against 86 us; 384^3: 245 against 143 us).  FP32 edges that
// are no multiple of 4 leave it earlier, for the whole-row kernel (even: 210^3
// 37.5 / 49.3 us, 222^3 53.0 / 49.9; odd: 201^3 42.1 / 41.2, 215^3 56.4 / 52.5).
// The other FP64 arithmetics unpack each value at every use here and once in
// the z-march kernel: equal at 160^3 (fixed point with a remainder 35.5 / 35.9
// us; 128^3 15.2 / 21.3; 192^3 58.9 / 51.0), and odd edges, which only the plain
// kernel takes besides, gain up to about 180 (101^3 10.5 / 15.3 us, 201^3 101 / 95).
// With the held outer layer these convert at every use: up to 80 (64^3 12.9 us
// against 19.0 with the best z-march tile, 96^3 33.8 / 27.2), odd edges up to
// 120 (101^3 24.5 us, plain kernel 33.2).
bool resident_supported(int dtype, int L, int arith, bool held)
{
    if (arith != GS_ARITH_IEEE && held) return L <= (L % 2 == 0 ? 80 : 120);
    if (arith != GS_ARITH_IEEE) return L <= (L % 2 == 0 ? 160 : 180);
    if (dtype == GS_F32 && L % 4 != 0) return L <= (L % 2 == 0 ? 218 : 202);
    return L <= 256;
}

// A launch holds every SM until it ends, and work on other streams waits: about
// 60 ms at most (5 ps per cell and step in FP32, 201^3; 42 in IEEE FP64 and up to
// 60 in the other arithmetics with the held layer, 72^3), and 4096 steps.
int resident_max_steps(int dtype, int L)
{
    const long long cell_steps = dtype == GS_F32 ? 10'000'000'000ll : 1'200'000'000ll;
    return (int)std::min<long long>(4096, std::max<long long>(2, cell_steps / ((long long)L * L * L)));
}

// Calls that the kernel takes.  Periodic FP64 fields in another arithmetic than
// IEEE are packed in place, which a call of two or more steps may do (its second
// step overwrites the input anyway).  A call of one step leaves its input as it
// is, for a replay of a captured call or a program that compares the two states.
// Even edges convert at the loads, up to 80 as with the held layer; above, and
// with odd edges, the z-march or the plain kernel takes the call.  us in fixed
// point with a remainder, this rule (packing in place): 32^3 6.7 (7.2), 33^3 5.3
// (8.3), 64^3 15.4 (10.8), 96^3 25.0 (19.0), 128^3 46.5 (32.7), 160^3 76 (61).
bool resident_takes(int L, int arith, bool held, int64_t n)
{
    return arith == GS_ARITH_IEEE || held || n != 1 || (L % 2 == 0 && L <= 80);
}

int launch_resident(int dtype, int L, void* const u[2], void* const v[2], int n, const Params& p, bool held, int64_t t,
                    unsigned* bar, int* err, uint64_t timeout_ns, cudaStream_t s)
{
    const bool noise = p.noise != 0.0;
#define GS_RES(T, V, AR)                                                                                               \
    return noise ? (held ? resident_launch_t<T, V, true, true, AR>(L, u, v, n, p, t, bar, err, timeout_ns, s)          \
                         : resident_launch_t<T, V, true, false, AR>(L, u, v, n, p, t, bar, err, timeout_ns, s))        \
                 : (held ? resident_launch_t<T, V, false, true, AR>(L, u, v, n, p, t, bar, err, timeout_ns, s)         \
                         : resident_launch_t<T, V, false, false, AR>(L, u, v, n, p, t, bar, err, timeout_ns, s))
    if (dtype == GS_F32) {
        if (L % 4 == 0) GS_RES(float, 4, 0);
        if (L % 2 == 0) GS_RES(float, 2, 0);
        GS_RES(float, 1, 0);
    }
    const bool conv = n == 1 && !held && !(p.io & 3) && L % 2 == 0;
#define GS_RES_AR(AR)                                                                                                  \
    if (p.arith == AR) {                                                                                               \
        if (conv && noise)                                                                                             \
            return resident_launch_t<double, 2, true, false, AR, true>(L, u, v, n, p, t, bar, err, timeout_ns, s);     \
        if (conv)                                                                                                      \
            return resident_launch_t<double, 2, false, false, AR, true>(L, u, v, n, p, t, bar, err, timeout_ns, s);    \
        if (L % 2 == 0) GS_RES(double, 2, AR);                                                                         \
        GS_RES(double, 1, AR);                                                                                         \
    }
    GS_RES_AR(GS_ARITH_DS)
    GS_RES_AR(GS_ARITH_FX)
    GS_RES_AR(GS_ARITH_FXF)
    if (L % 2 == 0) GS_RES(double, 2, 0);
    GS_RES(double, 1, 0);
#undef GS_RES
#undef GS_RES_AR
}

}  // namespace gs

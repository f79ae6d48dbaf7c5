// Device side of the kernels that keep small grids in L2 and run many steps
// per launch (single grid: gs_resident.cu, batch: gs_batch.cu).
#pragma once

#include <type_traits>

#include "gs_common.cuh"
#include "gs_ds.cuh"
#include "gs_fx.cuh"
#include "gs_fxf.cuh"

// V cells: one 16-byte vector, or fewer for edges L that are no multiple of it
// (FP32 pairs for even L, single cells for odd L)
template <typename T, int V>
GS_D void res_load(const T* p, T* r)
{
    if constexpr (V == 1) {
        r[0] = *p;
    } else if constexpr (V < GsVec<T>::N) {
        const float2 t = *reinterpret_cast<const float2*>(p);
        r[0] = t.x;
        r[1] = t.y;
    } else {
        gs_unpack<T>(*reinterpret_cast<const typename GsVec<T>::type*>(p), r);
    }
}

template <typename T, int V>
GS_D void res_store(T* p, const T* r)
{
    if constexpr (V == 1) *p = r[0];
    else if constexpr (V < GsVec<T>::N) *reinterpret_cast<float2*>(p) = make_float2(r[0], r[1]);
    else *reinterpret_cast<typename GsVec<T>::type*>(p) = gs_pack<T>(r);
}

// A run of rows of one grid (x fastest, then y, then z): from row (ys, zs) on,
// nrow rows, each plane contributing its rows ylo..yhi-1 (a brick; 0..L-1 for
// a run in memory order).
struct ResRows {
    int L, ylo, yhi, ys, zs, nrow;
};

// This thread's first group of V cells of a run and the step to its next one
// (tid, tid + blockDim.x, ... of the groups in order) as (x, y, z) increments.
template <int V>
struct ResWalk {
    int xv0, y0, z0, dxv, dy, dz;
    GS_D ResWalk(const ResRows& r, int tid)
    {
        const int nxv = r.L / V, nr = r.yhi - r.ylo;
        const int r0 = tid / nxv, dr = blockDim.x / nxv, q0 = r.ys - r.ylo + r0;
        xv0 = tid - r0 * nxv;
        dxv = blockDim.x - dr * nxv;
        dz = dr / nr;
        dy = dr - dz * nr;
        z0 = r.zs + q0 / nr;
        y0 = r.ylo + q0 - q0 / nr * nr;
    }
};

// Coefficients of arithmetic AR (0: IEEE, 1: double-single, 2: fixed point, 3:
// fixed point with a float remainder).
template <typename T, int AR>
using ResCoef = std::conditional_t<AR == 0, GsCoef<T>,
                                   std::conditional_t<AR == 1, GsCoefDS, std::conditional_t<AR == 2, GsCoefFX, GsCoefFXF2>>>;

// V cells from FP64 to AR's packed values; false: a value out of its range
template <int V, int AR>
GS_D bool res_pack(double* x)
{
    bool ok = true;
#pragma unroll
    for (int e = 0; e < V; ++e) {
        bool o = false;
        if constexpr (AR == 1) x[e] = ds_pack(ds_from_double(x[e]));
        if constexpr (AR == 2) x[e] = fx_pack(fx_from_double(x[e], o));
        if constexpr (AR == 3) x[e] = fxf_pack(fxf_from_double(x[e], o));
        ok &= !o;
    }
    return ok;
}

template <int V, int AR>
GS_D void res_unpack(double* x)
{
#pragma unroll
    for (int e = 0; e < V; ++e) {
        if constexpr (AR == 1) x[e] = ds_to_double(ds_unpack(x[e]));
        if constexpr (AR == 2) x[e] = fx_to_double(fx_unpack(x[e]));
        if constexpr (AR == 3) x[e] = fxf_to_double(fxf_unpack(x[e]));
    }
}

// One cell whose inputs are AR's packed values (the group functions' arithmetic).
template <bool NOISE, int AR>
GS_D void res_cell(const ResCoef<double, AR>& c, int32_t rn, double cu, double cv, double xlu, double xru, double ymu,
                   double ypu, double pu, double nu, double xlv, double xrv, double ymv, double ypv, double pv, double nv,
                   double& ou, double& ov, uint32_t& rng)
{
    if constexpr (AR == 1) {
        GsDS a, b;
        const GsDS su = ds_nsum(ds_unpack(xlu), ds_unpack(xru), ds_unpack(ymu), ds_unpack(ypu), ds_unpack(pu), ds_unpack(nu));
        const GsDS sv = ds_nsum(ds_unpack(xlv), ds_unpack(xrv), ds_unpack(ymv), ds_unpack(ypv), ds_unpack(pv), ds_unpack(nv));
        gs_update_ds<NOISE>(c, ds_unpack(cu), ds_unpack(cv), su, sv, (float)rn, a, b);
        ou = ds_pack(a);
        ov = ds_pack(b);
    } else if constexpr (AR == 2) {
        const long long su = fx_unpack(xlu) + fx_unpack(xru) + fx_unpack(ymu) + fx_unpack(ypu) + fx_unpack(pu) + fx_unpack(nu);
        const long long sv = fx_unpack(xlv) + fx_unpack(xrv) + fx_unpack(ymv) + fx_unpack(ypv) + fx_unpack(pv) + fx_unpack(nv);
        long long a, b;
        gs_update_fx<NOISE>(c, fx_unpack(cu), fx_unpack(cv), su, sv, rn, a, b);
        ou = fx_pack(a);
        ov = fx_pack(b);
    } else {
        GsFxf a, b;
        int32_t SU, SV;
        float SLU, SLV;
        fxf_nsum(fxf_unpack(xlu), fxf_unpack(xru), fxf_unpack(ymu), fxf_unpack(ypu), fxf_unpack(pu), fxf_unpack(nu), SU, SLU);
        fxf_nsum(fxf_unpack(xlv), fxf_unpack(xrv), fxf_unpack(ymv), fxf_unpack(ypv), fxf_unpack(pv), fxf_unpack(nv), SV, SLV);
        gs_update_fxf<NOISE>(c, fxf_unpack(cu), fxf_unpack(cv), SU, SLU, SV, SLV, rn, a, b, rng);
        ou = fxf_pack(a);
        ov = fxf_pack(b);
    }
}

// One step of the V cells at (x, y, z).  u, v, un, vn without __restrict__: other
// CTAs write in one step what this one reads in the next.  AR > 0 (FP64): the
// inputs are packed values, the outputs too unless `unpack`; with CONV both are
// FP64 values and every load is converted (HELD, whose outer layer has to keep
// its values to the bit, and a call of one step, which leaves its input as it
// is).  Returns the range word of AR = 3 (fxf_range_bad; all ones: an input out
// of range).
template <typename T, int V, bool NOISE, bool HELD, int AR, bool CONV>
GS_D uint32_t res_group(int L, int x, int y, int z, const T* u, const T* v, T* un, T* vn, const ResCoef<T, AR>& c,
                        GsKeys k, uint32_t kk2, bool unpack)
{
    uint32_t rng = 0;
    const int LL = L * L, row = (z * L + y) * L, i = row + x;  // 32 bits: L <= 256
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
    T xlu = u[ixl], xru = u[ixr], xlv = v[ixl], xrv = v[ixr];
    [[maybe_unused]] T fu[V], fv[V];  // the FP64 values behind cu, cv
    if constexpr (CONV) {
#pragma unroll
        for (int e = 0; e < V; ++e) {
            fu[e] = cu[e];
            fv[e] = cv[e];
        }
        bool ok = true;
        for (T* q : {cu, cv, pu, pv, nu, nv, ymu, ypu, ymv, ypv}) ok &= res_pack<V, AR>(q);
        for (T* q : {&xlu, &xru, &xlv, &xrv}) ok &= res_pack<1, AR>(q);
        if (!ok) rng = ~0u;
    }
    if constexpr (AR > 0) {
        if constexpr (V == 1) {
            res_cell<NOISE, AR>(c, NOISE ? gs_noise_num((uint32_t)i, k) : 0, cu[0], cv[0], xlu, xru, ymu[0], ypu[0],
                                pu[0], nu[0], xlv, xrv, ymv[0], ypv[0], pv[0], nv[0], ou[0], ov[0], rng);
        } else {
            const uint32_t pre = NOISE ? gs_group_pre((uint32_t)i, k) : 0u;
            if constexpr (AR == 1)
                gs_update_group_ds<NOISE, GsFromPacked, true>(c, pre, kk2, cu, cv, pu, pv, nu, nv, ymu, ypu, ymv, ypv,
                                                              xlu, xru, xlv, xrv, ou, ov);
            else if constexpr (AR == 2)
                gs_update_group_fx<NOISE, true>(c, pre, kk2, cu, cv, pu, pv, nu, nv, ymu, ypu, ymv, ypv, xlu, xru, xlv,
                                                xrv, ou, ov);
            else
                gs_update_group_fxf<NOISE, true, 0>(c, pre, kk2, cu, cv, pu, pv, nu, nv, ymu, ypu, ymv, ypv, xlu, xru,
                                                    xlv, xrv, ou, ov, rng);
        }
        if (CONV || unpack) {
            res_unpack<V, AR>(ou);
            res_unpack<V, AR>(ov);
        }
        if constexpr (HELD) {
#pragma unroll
            for (int e = 0; e < V; ++e) {
                cu[e] = fu[e];
                cv[e] = fv[e];
            }
        }
    } else if constexpr (V < GsVec<T>::N) {
        const uint32_t pre = NOISE ? gs_group_pre((uint32_t)i, k) : 0u;
#pragma unroll
        for (int e = 0; e < V; ++e) {
            const T su = gs_nsum(e > 0 ? cu[0] : xlu, e + 1 < V ? cu[V - 1] : xru, ymu[e], ypu[e], pu[e], nu[e]);
            const T sv = gs_nsum(e > 0 ? cv[0] : xlv, e + 1 < V ? cv[V - 1] : xrv, ymv[e], ypv[e], pv[e], nv[e]);
            gs_update<T, NOISE>(c, cu[e], cv[e], su, sv, NOISE ? gs_num_as<T>(gs_group_num(pre, (uint32_t)e, kk2)) : (T)0,
                                ou[e], ov[e]);
        }
    } else {
        const uint32_t pre = NOISE ? gs_group_pre((uint32_t)i, k) : 0u;
        gs_update_group<T, NOISE>(c, pre, kk2, cu, cv, pu, pv, nu, nv, ymu, ypu, ymv, ypv, xlu, xru, xlv, xrv,
                                  ou, ov);
    }
    if constexpr (HELD) {
        // the outer layer keeps its values
        if (y == 0 || y == L - 1 || z == 0 || z == L - 1) {
#pragma unroll
            for (int e = 0; e < V; ++e) {
                ou[e] = cu[e];
                ov[e] = cv[e];
            }
        }
        if (x == 0) {
            ou[0] = cu[0];
            ov[0] = cv[0];
        }
        if (x + V == L) {
            ou[V - 1] = cu[V - 1];
            ov[V - 1] = cv[V - 1];
        }
    }
    res_store<T, V>(un + i, ou);
    res_store<T, V>(vn + i, ov);
    return rng;
}

// One step of all cells of a run.
template <typename T, int V, bool NOISE, bool HELD, int AR = 0, bool CONV = false>
GS_D uint32_t res_rows(const ResRows& r, const ResWalk<V>& w, const T* u, const T* v, T* un, T* vn,
                       const ResCoef<T, AR>& c, GsKeys k, int tid, bool unpack = false)
{
    uint32_t rng = 0;
    const int L = r.L, nxv = L / V, nr = r.yhi - r.ylo, ng = r.nrow * nxv;
    const uint32_t kk2 = gs_kk2(k);
    int xv = w.xv0, y = w.y0, z = w.z0;
    for (int g = tid; g < ng; g += blockDim.x) {
        rng |= res_group<T, V, NOISE, HELD, AR, CONV>(L, xv * V, y, z, u, v, un, vn, c, k, kk2, unpack);
        xv += w.dxv;
        y += w.dy;
        z += w.dz;
        if (xv >= nxv) { xv -= nxv; ++y; }
        if (y >= r.yhi) { y -= nr; ++z; }
    }
    return rng;
}

// The cells of a run from FP64 to AR's packed values in place; false: some
// value out of its range.
template <int V, int AR>
GS_D bool res_pack_rows(const ResRows& r, const ResWalk<V>& w, double* u, double* v, int tid)
{
    const int L = r.L, nxv = L / V, nr = r.yhi - r.ylo, ng = r.nrow * nxv;
    int xv = w.xv0, y = w.y0, z = w.z0;
    bool ok = true;
    for (int g = tid; g < ng; g += blockDim.x) {
        const int i = (z * L + y) * L + xv * V;
        double a[V], b[V];
        res_load<double, V>(u + i, a);
        res_load<double, V>(v + i, b);
        ok &= res_pack<V, AR>(a);
        ok &= res_pack<V, AR>(b);
        res_store<double, V>(u + i, a);
        res_store<double, V>(v + i, b);
        xv += w.dxv;
        y += w.dy;
        z += w.dz;
        if (xv >= nxv) { xv -= nxv; ++y; }
        if (y >= r.yhi) { y -= nr; ++z; }
    }
    return ok;
}

// A brick's rows with its shell (what other CTAs read) first: rows 0 .. nb - 1
// of h x d, then the rows whose neighbours all belong to this CTA.  The walk
// stops between the two, so that a CTA can announce its shell and go on.
struct ResShell {
    int L, ylo, zs, h, d, nb;
    uint32_t inv;  // ceil(2^32 / (h - 2)): exact division of row numbers by umulhi
};

GS_D ResShell res_shell(const ResRows& r)
{
    const int h = r.yhi - r.ylo, d = r.nrow / h;
    const int inner = h > 2 && d > 2 ? (h - 2) * (d - 2) : 0;
    return ResShell{r.L, r.ylo, r.zs, h, d, r.nrow - inner, 0xffffffffu / (uint32_t)max(1, h - 2) + 1u};
}

// row number -> (y, z)
GS_D void res_shell_row(const ResShell& q, int r, int& y, int& z)
{
    if (r >= q.nb) {
        const int n = r - q.nb;
        // (h = 3: inv = 2^32 does not fit)
        const int k = q.h == 3 ? n : (int)__umulhi((uint32_t)n, q.inv);
        y = q.ylo + 1 + n - k * (q.h - 2);
        z = q.zs + 1 + k;
    } else if (r < q.h || q.d == 1) {
        y = q.ylo + r;
        z = q.zs;
    } else if (r < 2 * q.h) {
        y = q.ylo + r - q.h;
        z = q.zs + q.d - 1;
    } else {
        // the planes between: their first and last row (h = 1: the one row)
        const int m = r - 2 * q.h, two = q.h > 1 ? 1 : 0;
        z = q.zs + 1 + (m >> two);
        y = q.ylo + ((m & two) ? q.h - 1 : 0);
    }
}

// One step of the walk's groups (g: the next row and group of the row) up to row re.
template <typename T, int V, bool NOISE, bool HELD, int AR, bool CONV>
GS_D uint32_t res_shell_rows(const ResShell& q, int2& g, int re, const T* u, const T* v, T* un, T* vn,
                             const ResCoef<T, AR>& c, GsKeys k, bool unpack)
{
    uint32_t rng = 0;
    const int nxv = q.L / V, dr = blockDim.x / nxv, dxv = blockDim.x - dr * nxv;
    const uint32_t kk2 = gs_kk2(k);
    while (g.x < re) {
        int y, z;
        res_shell_row(q, g.x, y, z);
        rng |= res_group<T, V, NOISE, HELD, AR, CONV>(q.L, g.y * V, y, z, u, v, un, vn, c, k, kk2, unpack);
        g.x += dr;
        g.y += dxv;
        if (g.y >= nxv) { g.y -= nxv; ++g.x; }
    }
    return rng;
}

// Bounded grid barrier of co-resident CTAs in two halves, all threads.
//
// res_grid_arrive: the CTA's stores so far are ordered before its arrival (the
// block barrier makes them thread 0's predecessors); only warp 0 waits for the
// others, they go on with work that no other CTA sees before the next arrival.
GS_D void res_grid_arrive(unsigned* bar)
{
    __syncwarp();
    if (threadIdx.x < 32) {
        asm volatile("barrier.cta.sync 1, %0;" ::"r"(blockDim.x) : "memory");
        if (threadIdx.x == 0) gs_red_add_release_gpu(bar, 1u);
        __syncwarp();
    } else {
        asm volatile("barrier.cta.arrive 1, %0;" ::"r"(blockDim.x) : "memory");
    }
}

// res_grid_wait: every other CTA's arrival before thread 0's acquire, and that
// (and this CTA's own work) before the CTA's next loads.  `target` = arrivals
// after which it opens.  True: timed out.
GS_D bool res_grid_wait(unsigned* bar, unsigned target, int* err, uint64_t timeout_ns)
{
    int bad = 0;
    if (threadIdx.x == 0) {
        // the counter and the target wrap modulo 2^32; their difference is exact
        if ((int)(gs_ld_acquire_gpu(bar) - target) < 0) {
            const uint64_t t0 = gs_globaltimer();
            while ((int)(gs_ld_acquire_gpu(bar) - target) < 0)
                if (gs_globaltimer() - t0 > timeout_ns) {
                    gs_report(err, GS_DERR_TIMEOUT);
                    bad = 1;
                    break;
                }
        }
    }
    return __syncthreads_or(bad) != 0;
}

GS_D bool res_grid_sync(unsigned* bar, unsigned target, int* err, uint64_t timeout_ns)
{
    __syncthreads();
    if (threadIdx.x == 0) gs_red_add_release_gpu(bar, 1u);
    return res_grid_wait(bar, target, err, timeout_ns);
}

// Device side of the kernels that keep small grids in L2 and run many steps
// per launch (single grid: gs_resident.cu, batch: gs_batch.cu).
#pragma once

#include "gs_common.cuh"

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

// One step of the cells of a run.  u, v, un, vn without __restrict__: other
// CTAs write in one step what this one reads in the next.
template <typename T, int V, bool NOISE, bool HELD>
GS_D void res_rows(const ResRows& r, const ResWalk<V>& w, const T* u, const T* v, T* un, T* vn, const GsCoef<T>& c,
                   GsKeys k, int tid)
{
    const int L = r.L, nxv = L / V, LL = L * L, nr = r.yhi - r.ylo, ng = r.nrow * nxv;
    const uint32_t kk2 = gs_kk2(k);
    int xv = w.xv0, y = w.y0, z = w.z0;
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
            gs_update<T, NOISE>(c, cu[0], cv[0], su, sv, NOISE ? (T)gs_noise_num((uint32_t)i, k) : (T)0, ou[0],
                                ov[0]);
        } else {
            const uint32_t pre = NOISE ? gs_group_pre((uint32_t)i, k) : 0u;
            gs_update_group<T, NOISE>(c, pre, kk2, cu, cv, pu, pv, nu, nv, ymu, ypu, ymv, ypv, xlu, xru, xlv, xrv,
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
        xv += w.dxv;
        y += w.dy;
        z += w.dz;
        if (xv >= nxv) { xv -= nxv; ++y; }
        if (y >= r.yhi) { y -= nr; ++z; }
    }
}

// Bounded grid barrier of co-resident CTAs, all threads: the CTA's stores are
// ordered before its arrival (bar.sync makes them thread 0's predecessors),
// every other CTA's before thread 0's acquire, and that before this CTA's
// next loads.  `target` = arrivals after which it opens.  True: timed out.
GS_D bool res_grid_sync(unsigned* bar, unsigned target, int* err, uint64_t timeout_ns)
{
    __syncthreads();
    int bad = 0;
    if (threadIdx.x == 0) {
        gs_red_add_release_gpu(bar, 1u);
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

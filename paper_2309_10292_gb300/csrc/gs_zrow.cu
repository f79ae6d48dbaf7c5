// FP32 step of a grid whose edge is no multiple of 4 cells.
//
// Its rows start at every alignment, so neither a tensor map (16-byte strides)
// nor 16-byte loads fit, and one thread per cell with scalar loads and 64-bit
// index arithmetic runs at 131 GCUPS (250^3).  gs_zrow_kernel is the z-march
// scheme on tiles of whole rows: the rows of a tile are one contiguous run of
// memory, and so is each halo row, so a producer warp stages a plane with three
// 1D bulk copies per field from the 16-byte boundary at or below its start; the
// consumers add the remainder (0-3 cells, another one every plane when the edge
// is odd) when they index shared memory.  The x wrap is an index wrap in the
// row.  A thread owns two rows of two cells: two single columns half a row
// apart when the edge is odd (any alignment, no bank conflicts), a pair when it
// is even (every row start is 8-byte aligned).
//
// Bound by instruction issue (ncu: 79 thread instructions per cell and 77 % of
// issue slots at 414^3, 103 and 68 % at 251^3, DRAM traffic 0.98 of 16 bytes a
// cell).  us per step with noise, plain kernel -> this one: 222^3 84 -> 50, 250^3
// 118 -> 59, 251^3 119 -> 68, 414^3 518 -> 199 (357 GCUPS), 501^3 914 -> 458, 777^3
// 3393 -> 1660, 1302^3 18000 -> 6680.  With four single cells per thread a block
// apart (y neighbours from shared memory too) 250^3 took 64, 414^3 231 us.
#include <algorithm>
#include <type_traits>

#include "gs_common.cuh"
#include "gs_internal.h"

namespace gs {

struct ZRowArgs {
    const float* in[2];  // u, v
    float* out[2];
    int L, ty, tz;
    int nty, ntiles;     // tiles per plane, tiles (y fastest, then z-chunk)
    int stages, cons;    // ring depth, consumer threads
    int main_elems, row_elems;  // floats of a stage's main block and of one halo row block, per field
    GsCoef<float> c;
    GsKeys keys;
    int* err;
    uint64_t timeout_ns;
    unsigned* tickets;   // [next unit, CTAs done], zeroed between launches
};

// 1D bulk copy global -> shared (both addresses and the size multiples of 16
// bytes), completion signalled on `bar`
GS_D void gs_bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     gs_smem_addr(dst)),
                 "l"(src), "r"(bytes), "r"(gs_smem_addr(bar))
                 : "memory");
}

// Next unit of work: the tiles in order, the last G / 2 (G = CTAs) cut along z
// into four pieces; odd chunks and pieces march down (nz < 0).  False: none left.
GS_D bool zrow_unit(const ZRowArgs& a, int& y0, int& z0, int& nz)
{
    const int m = min(a.ntiles, (int)gridDim.x / 2), whole = a.ntiles - m;
    for (;;) {
        const int u = (int)atomicAdd(&a.tickets[0], 1u);
        if (u >= whole + 4 * m) return false;
        const int tile = u < whole ? u : whole + (u - whole) / 4;
        const int part = u < whole ? 0 : (u - whole) % 4, parts = u < whole ? 1 : 4;
        const int zi = tile / a.nty, zb = zi * a.tz, n = min(a.tz, a.L - zb);
        const int lo = n * part / parts, hi = n * (part + 1) / parts;
        if (hi <= lo) continue;
        y0 = (tile - zi * a.nty) * a.ty;
        z0 = zb + lo;
        nz = ((zi + part) & 1) ? lo - hi : hi - lo;
        return true;
    }
}

template <int V, bool NOISE, bool HELD>
__global__ void __maxnreg__(72) gs_zrow_kernel(const ZRowArgs a)
{
    extern __shared__ __align__(128) float zrow_smem[];
    __shared__ __align__(8) uint64_t bars[16];
    __shared__ volatile int abort_flag;
    // (y0, z0, +-nz) of the units the producer hands on, nz == 0 after the
    // last; a slot is reused four units (at least 12 planes, the ring holds
    // 6) later
    __shared__ int4 s_unit[4];

    const int S = a.stages, L = a.L, tid = threadIdx.x, lane = tid & 31;
    const long long LL = (long long)L * L;
    uint64_t* full = bars;
    uint64_t* empty = bars + S;
    const int field_elems = a.main_elems + 2 * a.row_elems;
    const int stage_elems = 2 * field_elems;

    if (tid == 0) {
        for (int s = 0; s < S; ++s) {
            gs_mbar_init(&full[s], 1);
            gs_mbar_init(&empty[s], a.cons / 32);
        }
        abort_flag = 0;
        gs_fence_mbar_init();
    }
    __syncthreads();

    if (tid >= a.cons) {
        // ------------------------------ producer warp ------------------------------
        if (tid != a.cons) return;
        uint32_t pph = 0;
        int ps = 0, kd = 0;
        bool wrapped = false, ok = true;
        const long long total = LL * L;
        auto next_stage = [&]() {
            if (++ps == S) { ps = 0; pph ^= 1u; wrapped = true; }
        };
        auto stage_free = [&]() {
            if (wrapped && !gs_mbar_wait(&empty[ps], pph ^ 1u, a.timeout_ns)) {
                gs_report(a.err, GS_DERR_TIMEOUT);
                abort_flag = 1;
            }
            return abort_flag == 0;
        };
        int y0, z0, nzs;
        while (ok) {
            const bool more = zrow_unit(a, y0, z0, nzs);
            if (!(ok = stage_free())) break;
            if (!more) {
                s_unit[kd & 3] = make_int4(0, 0, 0, 0);
                gs_mbar_arrive(&full[ps]);  // no copy: the phase completes here
                next_stage();
                break;
            }
            s_unit[kd & 3] = make_int4(y0, z0, nzs, 0);
            ++kd;
            const bool down = nzs < 0;
            const int nz = down ? -nzs : nzs, nvy = min(a.ty, L - y0);
            // the three runs of rows: tile, row above, row below
            const int yr[3] = {y0, y0 == 0 ? L - 1 : y0 - 1, y0 + nvy == L ? 0 : y0 + nvy};
            int zp = down ? (z0 + nz) % L : (z0 - 1 + L) % L;
            for (int j = 0; j < nz + 2 && ok; ++j) {
                if (j > 0 && !(ok = stage_free())) break;
                float* b = zrow_smem + (size_t)ps * stage_elems;
                long long start[3];
                int cnt[3];
                uint32_t bytes = 0;
#pragma unroll
                for (int m = 0; m < 3; ++m) {
                    const long long e0 = zp * LL + (long long)yr[m] * L, e1 = e0 + (long long)(m == 0 ? nvy : 1) * L;
                    start[m] = e0 & ~3ll;
                    // whole 16-byte units, but never past the end of the field:
                    // its last 1-3 cells go by plain stores
                    const long long end = min((e1 + 3) & ~3ll, total & ~3ll);
                    cnt[m] = (int)(end - start[m]);
                    bytes += 8u * (uint32_t)cnt[m];
                    for (long long i = end; i < e1; ++i)
                        for (int f = 0; f < 2; ++f)
                            b[f * field_elems + (m == 0 ? 0 : a.main_elems + (m - 1) * a.row_elems) + (i - start[m])] =
                                a.in[f][i];
                    // (before the copy engine's next fill of the block)
                    if (end < e1) gs_fence_proxy_async();
                }
                gs_mbar_arrive_expect_tx(&full[ps], bytes);
                for (int f = 0; f < 2; ++f)
#pragma unroll
                    for (int m = 0; m < 3; ++m)
                        gs_bulk_load(b + f * field_elems + (m == 0 ? 0 : a.main_elems + (m - 1) * a.row_elems),
                                     a.in[f] + start[m], 4u * (uint32_t)cnt[m], &full[ps]);
                next_stage();
                if (down)
                    zp = zp == 0 ? L - 1 : zp - 1;
                else
                    zp = zp + 1 == L ? 0 : zp + 1;
            }
        }
        // the last CTA to finish zeroes the counter for the next launch
        // (before the wait below, which would put this at the launch's end)
        __threadfence();
        if (atomicAdd(&a.tickets[1], 1u) == gridDim.x - 1) {
            a.tickets[0] = 0;
            a.tickets[1] = 0;
        }
        // let every copy this thread issued land before the CTA can exit: the
        // consumers may have given up on one, before or after its last issue
        // (fixed 2 s budget: copies in flight always complete).  seq: planes issued,
        // modulo two rounds; counted along, it cost 1.5 % (414^3 202.5 -> 199 us)
        const uint32_t seq = (uint32_t)((wrapped ? (pph ? 1 : 2) : 0) * S + ps);
        for (uint32_t q = (seq > (uint32_t)S ? seq - S : 0); q < seq; ++q)
            gs_mbar_wait(&full[q % S], (q / S) & 1, 2000000000ull);
        return;
    }

    // ------------------------------- consumer warps --------------------------------
    // this thread's cells: rows r0, r0 + 1 of the tile, KX groups of V cells
    // from x[] on (their y neighbours within the pair of rows are registers)
    constexpr int KX = 2 / V, KY = 2;
    const uint32_t kk2 = gs_kk2(a.keys);
    const int H = (L + 1) / 2;
    const int pr = tid / H, col = tid - pr * H;
    const int r0 = pr * KY < a.ty ? pr * KY : 0;
    int x[KX], oxl[KX], oxr[KX];
    bool actx[KX];
#pragma unroll
    for (int i = 0; i < KX; ++i) {
        x[i] = V * col + i * H;
        actx[i] = pr * KY < a.ty && x[i] < L;
        if (x[i] >= L) x[i] = 0;
        oxl[i] = x[i] == 0 ? L - 1 : -1;
        oxr[i] = x[i] + V == L ? V - L : V;
    }
    int cs = 0, kd = 0;
    uint32_t cph = 0;
    auto advance = [&]() {
        if (++cs == S) { cs = 0; cph ^= 1u; }
    };
    auto release = [&](int s) {
        __syncwarp();
        if (lane == 0) gs_mbar_arrive(&empty[s]);
    };
    auto wait_full = [&]() -> bool {
        if (gs_mbar_wait(&full[cs], cph, a.timeout_ns)) return true;
        gs_report(a.err, GS_DERR_TIMEOUT);
        abort_flag = 1;
        return false;
    };
    auto ld = [](const float* p, float* r) {
        if constexpr (V == 2) {
            const float2 t = *reinterpret_cast<const float2*>(p);
            r[0] = t.x;
            r[1] = t.y;
        } else {
            r[0] = *p;
        }
    };

    // planes z-1, z, z+1 (in marching order) of this thread's groups, rotating by renaming
    float qu[3][KY][KX][V], qv[3][KY][KX][V];
    for (;;) {
        if (!wait_full()) return;
        const int4 un = s_unit[kd & 3];
        ++kd;
        if (un.z == 0) return;
        auto run = [&](auto down_tag) -> bool {
            constexpr bool DOWN = decltype(down_tag)::value;
            const int y0 = un.x, nz = DOWN ? -un.z : un.z, nvy = min(a.ty, L - y0);
            const int ytop = y0 == 0 ? L - 1 : y0 - 1, ybot = y0 + nvy == L ? 0 : y0 + nvy;
            const bool first = r0 == 0, last = r0 + KY >= nvy;
            const bool on0 = r0 < nvy, on1 = r0 + 1 < nvy;
            int zl = DOWN ? (un.y + nz) % L : (un.y - 1 + L) % L;  // plane to load next
            // remainder of a run's start, (z L^2 + y L) mod 4
            auto rem = [&](int z, int y) { return (z * (L & 3) * (L & 3) + y * (L & 3)) & 3; };
            auto load_centre = [&](float (&u)[KY][KX][V], float (&v)[KY][KX][V]) {
                const float* b = zrow_smem + cs * stage_elems + rem(zl, y0) + r0 * L;
#pragma unroll
                for (int j = 0; j < KY; ++j)
#pragma unroll
                    for (int i = 0; i < KX; ++i) {
                        ld(b + j * L + x[i], u[j][i]);
                        ld(b + field_elems + j * L + x[i], v[j][i]);
                    }
                zl = DOWN ? (zl == 0 ? L - 1 : zl - 1) : (zl + 1 == L ? 0 : zl + 1);
            };
            int sc = 0, zc = DOWN ? un.y + nz - 1 : un.y;
            long long g0 = zc * LL + (long long)(y0 + r0) * L;
            auto plane = [&](float (&pu)[KY][KX][V], float (&pv)[KY][KX][V], float (&cu)[KY][KX][V],
                             float (&cv)[KY][KX][V], float (&nu)[KY][KX][V], float (&nv)[KY][KX][V]) -> bool {
                if (!wait_full()) return false;
                load_centre(nu, nv);
                const float* b = zrow_smem + sc * stage_elems;
                const float* bm = b + rem(zc, y0) + r0 * L;
                const float* bt = first ? b + a.main_elems + rem(zc, ytop) : bm - L;
                const float* bbot = b + a.main_elems + a.row_elems + rem(zc, ybot);
                const float* bb = last ? bbot : bm + KY * L;
#pragma unroll
                for (int i = 0; i < KX; ++i) {
                    float ymu[V], ymv[V], ypu[V], ypv[V];
                    ld(bt + x[i], ymu);
                    ld(bt + field_elems + x[i], ymv);
                    ld(bb + x[i], ypu);
                    ld(bb + field_elems + x[i], ypv);
#pragma unroll
                    for (int j = 0; j < KY; ++j) {
                        const float* pm = bm + j * L + x[i];
                        const float xlu = pm[oxl[i]], xru = pm[oxr[i]];
                        const float xlv = pm[field_elems + oxl[i]], xrv = pm[field_elems + oxr[i]];
                        const long long g = g0 + j * L + x[i];
                        const uint32_t pre = NOISE ? gs_group_pre((uint32_t)g, a.keys) : 0u;
                        float ou[V], ov[V];
#pragma unroll
                        for (int e = 0; e < V; ++e) {
                            // z-1 and z+1: the plane before and after, marching up; the other way round, down
                            const float zmu = DOWN ? nu[j][i][e] : pu[j][i][e], zpu = DOWN ? pu[j][i][e] : nu[j][i][e];
                            const float zmv = DOWN ? nv[j][i][e] : pv[j][i][e], zpv = DOWN ? pv[j][i][e] : nv[j][i][e];
                            const float bu = j > 0 ? cu[0][i][e] : ymu[e], bv = j > 0 ? cv[0][i][e] : ymv[e];
                            // (an odd number of rows: the bottom run follows the pair's first row)
                            const float au = j + 1 < KY && (V == 2 || on1) ? cu[KY - 1][i][e] : ypu[e];
                            const float av = j + 1 < KY && (V == 2 || on1) ? cv[KY - 1][i][e] : ypv[e];
                            const float su = gs_nsum(e > 0 ? cu[j][i][0] : xlu, e + 1 < V ? cu[j][i][V - 1] : xru, bu, au, zmu, zpu);
                            const float sv = gs_nsum(e > 0 ? cv[j][i][0] : xlv, e + 1 < V ? cv[j][i][V - 1] : xrv, bv, av, zmv, zpv);
                            const float rn = NOISE ? (float)gs_group_num(pre, (uint32_t)e, kk2) : 0.f;
                            gs_update<float, NOISE>(a.c, cu[j][i][e], cv[j][i][e], su, sv, rn, ou[e], ov[e]);
                            if constexpr (HELD) {
                                const int y = y0 + r0 + j;
                                if (y == 0 || y == L - 1 || zc == 0 || zc == L - 1 || x[i] + e == 0 || x[i] + e == L - 1) {
                                    ou[e] = cu[j][i][e];
                                    ov[e] = cv[j][i][e];
                                }
                            }
                        }
                        if (actx[i] && (j == 0 ? on0 : on1)) {
                            if constexpr (V == 2) {
                                *reinterpret_cast<float2*>(a.out[0] + g) = make_float2(ou[0], ou[1]);
                                *reinterpret_cast<float2*>(a.out[1] + g) = make_float2(ov[0], ov[1]);
                            } else {
                                a.out[0][g] = ou[0];
                                a.out[1][g] = ov[0];
                            }
                        }
                    }
                }
                release(sc);
                sc = cs;
                advance();
                zc += DOWN ? -1 : 1;
                g0 += DOWN ? -LL : LL;
                return true;
            };

            // the plane before the first (waited for above), then the first
            load_centre(qu[0], qv[0]);
            release(cs);
            advance();
            if (!wait_full()) return false;
            load_centre(qu[1], qv[1]);
            sc = cs;
            advance();
            int zi = 0;
            for (; zi + 3 <= nz; zi += 3) {
                if (!plane(qu[0], qv[0], qu[1], qv[1], qu[2], qv[2])) return false;
                if (!plane(qu[1], qv[1], qu[2], qv[2], qu[0], qv[0])) return false;
                if (!plane(qu[2], qv[2], qu[0], qv[0], qu[1], qv[1])) return false;
            }
            if (zi < nz && !plane(qu[0], qv[0], qu[1], qv[1], qu[2], qv[2])) return false;
            if (zi + 1 < nz && !plane(qu[1], qv[1], qu[2], qv[2], qu[0], qv[0])) return false;
            release(sc);  // the plane after the last (only its centre was used)
            return abort_flag == 0;
        };
        if (!(un.z < 0 ? run(std::true_type{}) : run(std::false_type{}))) return;
    }
}

template <int V, bool NOISE, bool HELD>
static int zrow_launch_t(ZRowArgs& a, cudaStream_t s)
{
    auto kern = gs_zrow_kernel<V, NOISE, HELD>;
    const int threads = a.cons + 32;
    const size_t stage = sizeof(float) * 2 * (a.main_elems + 2 * a.row_elems);
    // as many CTAs per SM as the registers and a ring of at least 4 stages allow
    int ctas = 65536 / (threads * 72);
    while (ctas > 1 && 4 * stage * ctas > 220 * 1024) --ctas;
    a.stages = (int)std::min<size_t>(6, 220 * 1024 / ctas / stage);
    const size_t smem = stage * a.stages;
    GS_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int per_sm = 0;
    GS_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem));
    if (per_sm < 1) return fail(GS_EINVAL, "row tile of %d rows does not fit on an SM", a.ty);
    kern<<<std::min(a.ntiles, per_sm * num_sms()), threads, smem, s>>>(a);
    GS_CUDA_TRY(cudaGetLastError());
    return GS_OK;
}

bool zrow_supported(int dtype, int L) { return dtype == GS_F32 && L % 4 != 0 && L > 64; }

int launch_zrow(int L, const void* u, const void* v, void* un, void* vn, const Params& p, bool held, int64_t t,
                unsigned* tickets, int* err, uint64_t timeout_ns, cudaStream_t s)
{
    ZRowArgs a;
    a.in[0] = (const float*)u;
    a.in[1] = (const float*)v;
    a.out[0] = (float*)un;
    a.out[1] = (float*)vn;
    a.L = L;
    // pairs of rows; the halo rows are read again from L2.  Even edges: up to
    // 416 consumer threads, two CTAs per SM (250^3 60 us, with 528 70); odd ones,
    // bound by issue, up to 528 in one CTA and 24-plane chunks (251^3 68 us, with
    // 416 72, with 32 planes 74)
    const int H = (L + 1) / 2;
    a.ty = 2 * std::max(1, (L % 2 == 0 ? 416 : 528) / H);
    a.tz = L % 2 == 0 ? 32 : 24;
    a.nty = (L + a.ty - 1) / a.ty;
    a.ntiles = a.nty * ((L + a.tz - 1) / a.tz);
    a.cons = (H * (a.ty / 2) + 31) / 32 * 32;
    // a block holds its run and the rest of the 16-byte units at its ends
    a.main_elems = (a.ty * L + 8 + 31) / 32 * 32;
    a.row_elems = (L + 7 + 31) / 32 * 32;
    a.c = gs_make_coef<float>(p.Du, p.Dv, p.F, p.k, p.dt, p.noise);
    a.keys = gs_step_keys(p.seed, t);
    a.err = err;
    a.timeout_ns = timeout_ns;
    a.tickets = tickets;
    const bool noise = p.noise != 0.0;
#define GS_ZROW(V)                                                                                                  \
    return noise ? (held ? zrow_launch_t<V, true, true>(a, s) : zrow_launch_t<V, true, false>(a, s))                \
                 : (held ? zrow_launch_t<V, false, true>(a, s) : zrow_launch_t<V, false, false>(a, s))
    if (L % 2 == 0) GS_ZROW(2);
    GS_ZROW(1);
#undef GS_ZROW
}

}  // namespace gs

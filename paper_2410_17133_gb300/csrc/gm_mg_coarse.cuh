// The whole Chebyshev polynomial of the coarsest multigrid level in one launch.
//
// The coarsest grid (10 to 19 cells per direction) has a few thousand nodes and a
// polynomial of degree 24: as 47 launches of a K_b product or an update it took
// two thirds of the launches of a V-cycle, each one bound by its own latency
// (about 4 us in FP32 and 15 us in FP64 at 12^3..16^3, where the work is a few
// hundred nanoseconds of the chip).  Here one thread-block cluster runs all
// steps.  A CTA owns node rows in y (all x and z, so that the fault pairs spread
// over the CTAs and both lips of a pair are neighbours in one row), keeps their
// iterate in shared memory, reads the rows beside its own from its neighbours'
// shared memory, and meets the others once per step at the cluster barrier.
//
// What bounds it: latency, so the work of a row is cut into as many independent
// items as there are: elements of the two layers around the row (FP64: and
// output fields), then (node, component) twice.  FP32 multiplies in the parity
// basis like gm_bulk32.cuh; FP64 in wide fixed point like gm_bulkfx.cuh with the
// unit of the CTA's rows, and a step whose values that would not hold as exactly
// as FP64 (the same test, element by element) is done again in FP64 by that CTA.
// The march direction is y here: a mode's bit 1 (s & 2) separates a layer's lower
// and upper rows.
// Included by gm_mg.cu only.
#pragma once

#include <mutex>

#include <cooperative_groups.h>

#include "gm_bulkfx.cuh"

namespace {

template <typename T>
__host__ __device__ constexpr int mgc_threads() { return sizeof(T) == 8 ? 384 : 512; }
template <typename T>
__host__ __device__ constexpr int mgc_limbs() { return sizeof(T) == 8 ? 3 : 1; }

template <typename T, typename MT>
struct CoarseArgs {
    GridDesc g;
    const T* E;
    const uint8_t* mask;
    const T* b;
    T* x;                // result
    const MT* mi;
    PairPrec<T> pp;
    FaultK<T> fk;
    const double* coef;  // (c1, c2) per step
    int deg, rows;       // rows of a CTA at most
    unsigned m_rn, m_rowlen, m_nx, m_faces;   // ceil(2^32 / d): quotients by one multiplication
    const int* skip;
};

// x / d for x < 2^16, 2 <= d < 2^16 with m = ceil(2^32 / d): exact, since x (m d - 2^32) < 2^32
// (d = 1 would need 33 bits; every divisor is at least nx, so levels of one cell in x keep their launches)
__device__ inline int mgc_div(int x, unsigned m) { return (int)__umulhi((unsigned)x, m); }
inline unsigned mgc_magic(unsigned d) { return (unsigned)((0x100000000ull + d - 1) / d); }

// first node row of CTA r of n: the first CTAs take one row more, so that
// neighbouring rows are in neighbouring CTAs also where some have none
__host__ __device__ inline int mgc_row(const GridDesc& g, int r, int n)
{
    const int q = (g.ny + 1) / n, rem = (g.ny + 1) % n;
    return r * q + (r < rem ? r : rem);
}

// Shared memory of a CTA in bytes from the start: iterate (two buffers), right
// side, direction and residual of its rows, staged rows as words, what the layers around a row give
// it, modulus and mask of the staged part, nodal and pair inverses, tangents, and
// what each (node, component) item reads (the
// cluster barrier empties the L1 cache: what is read in every step would come
// from L2 each time).
struct MgcLayout {
    size_t x, b, d, r, st, out, E, mask, mi, item, P, D, total;
};
template <typename T, typename MT>
__host__ __device__ inline MgcLayout mgc_layout(const GridDesc& g, int rows)
{
    const size_t rn = (size_t)(g.nx + 1) * g.nplanes, faces = (size_t)g.nx * g.nz, NL = mgc_limbs<T>();
    MgcLayout L{};
    size_t at = 0;
    auto put = [&](size_t bytes) {
        const size_t p = at;
        at += (bytes + 15) & ~(size_t)15;
        return p;
    };
    L.x = put(2 * rows * 3 * rn * sizeof(T));
    L.b = put(rows * 3 * rn * sizeof(T));
    L.d = put(rows * 3 * rn * sizeof(T));
    L.r = put(rows * 3 * rn * sizeof(T));
    L.st = put((rows + 2) * 3 * NL * rn * 4);
    L.out = put(rows * 2 * 12 * NL * faces * 4);
    L.E = put((rows + 1) * faces * sizeof(T));
    L.mask = put((rows + 2) * rn);
    L.mi = put(rows * 6 * rn * sizeof(MT));
    L.item = put(rows * 3 * rn * sizeof(int2));
    if (g.kf >= 0) {
        L.P = put((size_t)rows * 36 * (g.nx + 1) * sizeof(T));
        L.D = put((size_t)rows * 6 * (g.nx + 1) * sizeof(T));
    }
    L.total = at;
    return L;
}

// Modes of the element whose lower row is `row` of the staged rows, first node nd.
template <typename W, int NL>
__device__ __forceinline__ void mgc_modes(const W* st, int row, int nd, int rn, int rowlen, W (&xv)[24][NL])
{
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int l = 0; l < NL; ++l) {
            W t[2][4];                                          // [ay][sx + 2 sz]
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const W* v = st + ((size_t)((row + s) * 3 + c) * NL + l) * rn + nd;
                const W a0 = v[0] + v[1], a1 = v[0] - v[1];
                const W b0 = v[rowlen] + v[rowlen + 1], b1 = v[rowlen] - v[rowlen + 1];
                t[s][0] = a0 + b0;
                t[s][1] = a1 + b1;
                t[s][2] = a0 - b0;
                t[s][3] = a1 - b1;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int s0 = (q & 1) | ((q & 2) << 1);        // mode (sx, 0, sz)
                xv[c * 8 + s0][l] = t[0][q] + t[1][q];
                xv[c * 8 + (s0 | 2)][l] = t[0][q] - t[1][q];
            }
        }
}

// What the element gives its upper (lay 0) or lower row in one field, corner by
// corner (ax + 2 az): mode(s, y) forms output mode s.
template <typename W, int NL, class Mode>
__device__ __forceinline__ void mgc_corners(W* w, int faces, int lay, Mode mode)
{
    W o[4][NL];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        W lo[NL] = {}, hi[NL];
        const int s0 = (q & 1) | ((q & 2) << 1);
        if (s0 != 0) mode(s0, lo);                              // the constant mode carries no force
        mode(s0 | 2, hi);
#pragma unroll
        for (int l = 0; l < NL; ++l) o[q][l] = lay == 0 ? lo[l] - hi[l] : lo[l] + hi[l];
    }
#pragma unroll
    for (int l = 0; l < NL; ++l) {
        const W p0 = o[0][l] + o[1][l], p1 = o[0][l] - o[1][l];
        const W q0 = o[2][l] + o[3][l], q1 = o[2][l] - o[3][l];
        w[(size_t)l * faces] = p0 + q0;
        w[(size_t)(NL + l) * faces] = p1 + q1;
        w[(size_t)(2 * NL + l) * faces] = p0 - q0;
        w[(size_t)(3 * NL + l) * faces] = p1 - q1;
    }
}

// The layers' results of a step in FP64, from staged doubles: as the fixed-point
// items, for the steps whose values those would not hold (see below).
template <int CLS>
__device__ __noinline__ void mgc_layers_f64(const RefOps<double>& R, const GridDesc& g, int j0, int own, unsigned m_faces,
                                            unsigned m_nx, const double* st, const double* sE, double* out)
{
    constexpr ParPat PP = gm_make_parpat(CLS);
    const int rowlen = g.nx + 1, rn = rowlen * g.nplanes, faces = g.nx * g.nz;
    for (int it = threadIdx.x; it < own * 6 * faces; it += blockDim.x) {
        const int blk = mgc_div(it, m_faces), f = it - blk * faces, rl = blk / 3, cc = blk - rl * 3;
        const int row = rl >> 1, lay = rl & 1, j = j0 + row;
        double* w = out + (size_t)(rl * 3 + cc) * 4 * faces + f;
        if (lay == 0 ? j == 0 : j == g.ny) {
            for (int q = 0; q < 4; ++q) w[(size_t)q * faces] = 0.0;
            continue;
        }
        const int ek = mgc_div(f, m_nx), fi = f - ek * g.nx;
        double xv[24][1];
        mgc_modes<double, 1>(st, row + lay, fi + rowlen * (ek + (g.kf >= 0 && ek >= g.kf ? 1 : 0)), rn, rowlen, xv);
        const double Ee = sE[(size_t)(row + lay) * faces + f];
        auto field = [&](auto c_) {
            constexpr int c = decltype(c_)::value;
            mgc_corners<double, 1>(w, faces, lay, [&](int s, double (&y)[1]) {
                double t = 0.0;
#pragma unroll
                for (int i = 0; i < 24; ++i)
                    if (PP.k[c * 8 + s][i] >= 0 && (i & 7) != 0) t = fma(R.K[PP.k[c * 8 + s][i]], xv[i][0], t);
                y[0] = Ee * t;
            });
        };
        if (cc == 0) field(std::integral_constant<int, 0>{});
        if (cc == 1) field(std::integral_constant<int, 1>{});
        if (cc == 2) field(std::integral_constant<int, 2>{});
    }
}

template <typename T, typename MT, int CLS>
__global__ void __launch_bounds__(mgc_threads<T>(), 1)
mg_coarse_kernel(int chained, const __grid_constant__ CoarseArgs<T, MT> a, const __grid_constant__ RefOps<float> R,
                 const __grid_constant__ RefFx F, const __grid_constant__ RefOps<double> R64)
{
    gm_chain(chained);
    constexpr bool FX = sizeof(T) == 8;
    constexpr int NL = mgc_limbs<T>(), NT = mgc_threads<T>();
    using W = typename std::conditional<FX, int, float>::type;      // word of a staged value
    constexpr ParPat PP = gm_make_parpat(CLS);
    if (a.skip && *a.skip) return;                                  // the same for every CTA
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), ncta = (int)cl.num_blocks();

    extern __shared__ __align__(16) unsigned char mgc_raw[];
    __shared__ int s_top[NT / 32], s_least[NT / 32];
    const GridDesc& g = a.g;
    const MgcLayout L = mgc_layout<T, MT>(g, a.rows);
    const int rowlen = g.nx + 1, rn = rowlen * g.nplanes, faces = g.nx * g.nz;
    const long long N = g.N;
    const int tid = threadIdx.x;
    T* sx = reinterpret_cast<T*>(mgc_raw + L.x);                    // [buffer][row][field][node]
    T* sb = reinterpret_cast<T*>(mgc_raw + L.b);                    // [row][field][node]
    T* sd = reinterpret_cast<T*>(mgc_raw + L.d);                    // [row][field][node]
    T* sr = reinterpret_cast<T*>(mgc_raw + L.r);                    // [row][field][node]
    MT* smi = reinterpret_cast<MT*>(mgc_raw + L.mi);                // [row][entry][node]
    int2* sit = reinterpret_cast<int2*>(mgc_raw + L.item);          // first word of its layers' results; flags
    T* sP = reinterpret_cast<T*>(mgc_raw + L.P);                    // [row][entry][pair of the row]
    T* sD = reinterpret_cast<T*>(mgc_raw + L.D);                    // [row][entry][pair of the row]
    W* st = reinterpret_cast<W*>(mgc_raw + L.st);                   // [staged row][field][limb][node]
    W* out = reinterpret_cast<W*>(mgc_raw + L.out);                 // [row][layer][field][corner][limb][face]
    T* sE = reinterpret_cast<T*>(mgc_raw + L.E);                    // [layer][face]
    uint8_t* sm = mgc_raw + L.mask;                                 // [staged row][node]
    const int j0 = mgc_row(g, rank, ncta), j1 = mgc_row(g, rank + 1, ncta), own = j1 - j0;
    const size_t buf = (size_t)a.rows * 3 * rn;

    // node i + rowlen kk of row j
    auto node = [&](int n, int j) -> long long {
        const int kk = mgc_div(n, a.m_rowlen);
        return (n - kk * rowlen) + (long long)rowlen * (j + (long long)(g.ny + 1) * kk);
    };
    if (own > 0) {
        for (int q = tid; q < (own + 2) * rn; q += NT) {
            const int sr_ = mgc_div(q, a.m_rn), n = q - sr_ * rn, j = j0 - 1 + sr_;
            sm[q] = j >= 0 && j <= g.ny ? a.mask[node(n, j)] : (uint8_t)7;
        }
        for (int q = tid; q < (own + 1) * faces; q += NT) {
            const int l = mgc_div(q, a.m_faces), f = q - l * faces, j = j0 - 1 + l;
            const int ek = mgc_div(f, a.m_nx);
            sE[q] = j >= 0 && j < g.ny ? a.E[(f - ek * g.nx) + (long long)g.nx * (j + (long long)g.ny * ek)] : T(0);
        }
    }
    if (g.kf >= 0)
        for (int q = tid; q < own * 42 * rowlen; q += NT) {
            const int row = q / (42 * rowlen), e = (q - row * 42 * rowlen) / rowlen, i = q % rowlen;
            const long long pair = i + (long long)rowlen * (j0 + row);
            if (e < 36) sP[(size_t)(row * 36 + e) * rowlen + i] = a.pp.inv[e * a.pp.nb + pair];
            else sD[(size_t)(row * 6 + e - 36) * rowlen + i] = a.fk.D[(e - 36) * g.nb + pair];
        }
    // the (node, component) items
    constexpr int FIXED = 16, LIP = 32, UPPER = 64;
    for (int it = tid; it < own * 3 * rn; it += NT) {
        const int blk = mgc_div(it, a.m_rn), n = it - blk * rn, row = blk / 3, c = blk - row * 3;
        const int kk = mgc_div(n, a.m_rowlen), i = n - kk * rowlen;
        const long long gn = node(n, j0 + row);
        const bool above = kk + 1 < g.nplanes && kk != g.kf, below = kk > 0 && kk - 1 != g.kf;
        // bit dx + 2 dz: the element to the left (dx) and below in z (dz) of the node exists
        int fl = 0;
        if (above && i < g.nx) fl |= 1;
        if (above && i > 0) fl |= 2;
        if (below && i < g.nx) fl |= 4;
        if (below && i > 0) fl |= 8;
        if ((sm[(size_t)(row + 1) * rn + n] >> c) & 1u) fl |= FIXED;
        if (g.kf >= 0 && (kk == g.kf || kk == g.kf + 1)) fl |= LIP | (kk > g.kf ? UPPER : 0);
        sit[it] = make_int2((row * 6 + c) * 4 * NL * faces + i + g.nx * (kk - (g.kf >= 0 && kk > g.kf ? 1 : 0)), fl);
        sb[it] = a.b[c * N + gn];
        for (int k = c; k < 6; k += 3) smi[(size_t)(row * 6 + k) * rn + n] = a.mi[k * N + gn];
    }
    __syncthreads();

    for (int step = 0; step < a.deg; ++step) {
        const T c1 = (T)a.coef[2 * step], c2 = (T)a.coef[2 * step + 1];
        const T* xi = sx + (step & 1 ? 0 : buf);                    // written by the step before
        T* xo = sx + (step & 1 ? buf : 0);
        double scale = 0.0;
        bool inexact = false, cut = false, f64 = false;             // FP64: see gm_fx_exact
        const T* from[2] = {xi, xi};
        // field f of staged node q: rows j0 - 1 .. j1, own rows and the neighbours' nearest ones
        auto value = [&](int q, int f) -> T {
            const int r = mgc_div(q, a.m_rn), n = q - r * rn, j = j0 - 1 + r;
            if (j < 0 || j > g.ny || ((sm[q] >> f) & 1u)) return T(0);
            const T* p = r == 0 ? from[0] : r == own + 1 ? from[1] : xi + (size_t)(r - 1) * 3 * rn;
            return p[(size_t)f * rn + n];
        };
        if (step > 0 && own > 0) {
            int top = 0, least = 0x7ff;
            if (rank > 0 && j0 > 0) from[0] = cl.map_shared_rank(const_cast<T*>(xi), rank - 1) +
                                              (size_t)(j0 - 1 - mgc_row(g, rank - 1, ncta)) * 3 * rn;
            if (rank + 1 < ncta && j1 <= g.ny) from[1] = cl.map_shared_rank(const_cast<T*>(xi), rank + 1);
            const int count = (own + 2) * rn;
            if constexpr (FX) {
                constexpr int MAXQ = 8;                             // values kept between the two passes
                auto extent = [&](T v) {
                    const int e = (__double2hiint(v) & 0x7fffffff) >> 20;
                    top = max(top, e);
                    if (v != T(0)) least = min(least, e);
                };
                T keep[MAXQ];
#pragma unroll
                for (int u = 0; u < MAXQ; ++u) {
                    const int i = tid + u * NT;
                    keep[u] = T(0);
                    if (i < 3 * count) {
                        const int f = (i >= count) + (i >= 2 * count);
                        keep[u] = value(i - f * count, f);
                        extent(keep[u]);
                    }
                }
                for (int i = tid + MAXQ * NT; i < 3 * count; i += NT) {
                    const int f = (i >= count) + (i >= 2 * count);
                    extent(value(i - f * count, f));
                }
                top = __reduce_max_sync(0xffffffffu, top);
                least = __reduce_min_sync(0xffffffffu, least);
                if ((tid & 31) == 0) { s_top[tid >> 5] = top; s_least[tid >> 5] = least; }
                __syncthreads();
#pragma unroll
                for (int w = 0; w < NT / 32; ++w) { top = max(top, s_top[w]); least = min(least, s_least[w]); }
                // values at the ends of the exponent range, or not finite: FP64
                const int qe = (top - 1022 - GM_FX_IN) + F.eK + F.topE - 1022;
                const bool ends = least != 0x7ff && (top == 0x7ff || top < 100 || qe > 900 || qe < -1000);
                cut = top - least > 22;
                inexact = ends;
                scale = ends || least == 0x7ff ? 0.0 : gm_fx_real((int64_t)(qe + 1023) << 52);
                auto limbs = [&](int i, T v) {
                    const int f = (i >= count) + (i >= 2 * count), q = i - f * count, r = mgc_div(q, a.m_rn), n = q - r * rn;
                    int l[3];
                    gm_fx_from_double(v, top, l);
#pragma unroll
                    for (int k = 0; k < 3; ++k) st[((size_t)(r * 3 + f) * 3 + k) * rn + n] = l[k];
                };
#pragma unroll
                for (int u = 0; u < MAXQ; ++u)
                    if (tid + u * NT < 3 * count) limbs(tid + u * NT, keep[u]);
                for (int i = tid + MAXQ * NT; i < 3 * count; i += NT) {
                    const int f = (i >= count) + (i >= 2 * count);
                    limbs(i, value(i - f * count, f));
                }
            } else {
                for (int q = tid; q < count; q += NT) {
                    const int r = mgc_div(q, a.m_rn), n = q - r * rn;
#pragma unroll
                    for (int f = 0; f < 3; ++f) st[(size_t)(r * 3 + f) * rn + n] = value(q, f);
                }
            }
        }
        __syncthreads();
        if (step > 0) {
            // layer 0: elements below the row (their upper part), layer 1: above it (lower part)
            constexpr int NC = FX ? 3 : 1;                      // FP64: one output field per item
            for (int it = tid; it < own * 2 * NC * faces; it += NT) {
                const int blk = mgc_div(it, a.m_faces), f = it - blk * faces;   // (row, layer, field)
                const int rl = NC == 1 ? blk : blk / NC, cc = blk - rl * NC;
                const int row = rl >> 1, lay = rl & 1, j = j0 + row;
                if (lay == 0 ? j == 0 : j == g.ny) {
#pragma unroll
                    for (int c = 0; c < 3; ++c)
                        if (NC == 1 || c == cc)
#pragma unroll
                            for (int q = 0; q < 4 * NL; ++q) out[(size_t)((rl * 3 + c) * 4 * NL + q) * faces + f] = W(0);
                    continue;
                }
                const int ek = mgc_div(f, a.m_nx), fi = f - ek * g.nx;
                const int nd = fi + rowlen * (ek + (g.kf >= 0 && ek >= g.kf ? 1 : 0));
                W xv[24][NL];
                mgc_modes<W, NL>(st, row + lay, nd, rn, rowlen, xv);
                const T Ee = sE[(size_t)(row + lay) * faces + f];
                int El[3] = {0, 0, 0};
                if constexpr (FX) gm_fx_coef22(Ee, F.topE, El);
                auto field = [&](auto c_) {
                    constexpr int c = decltype(c_)::value;
                    if constexpr (FX) inexact |= !gm_fx_exact<CLS, GM_M_K, c, 1>(F, xv, cut);
                    mgc_corners<W, NL>(out + (size_t)(rl * 3 + c) * 4 * NL * faces + f, faces, lay, [&](int s, W (&y)[NL]) {
                        if constexpr (FX) {
                            gm_fx_k_mode<CLS>(F, xv, c, s, El, y);
                        } else {
                            float t = 0.f;
#pragma unroll
                            for (int i = 0; i < 24; ++i)
                                if (PP.k[c * 8 + s][i] >= 0 && (i & 7) != 0) t = fmaf(R.K[PP.k[c * 8 + s][i]], xv[i][0], t);
                            y[0] = Ee * t;
                        }
                    });
                };
                if (NC == 1 || cc == 0) field(std::integral_constant<int, 0>{});
                if (NC == 1 || cc == 1) field(std::integral_constant<int, 1>{});
                if (NC == 1 || cc == 2) field(std::integral_constant<int, 2>{});
            }
            if constexpr (FX) {
                f64 = __syncthreads_or(inexact);
                if (f64) {
                    double* sv = reinterpret_cast<double*>(st);
                    for (int i = tid; i < 3 * (own + 2) * rn; i += NT) {
                        const int q = mgc_div(i, a.m_rn), n = i - q * rn, r = q / 3, f = q - 3 * r;
                        sv[i] = value(r * rn + n, f);
                    }
                    __syncthreads();
                    mgc_layers_f64<CLS>(R64, g, j0, own, a.m_faces, a.m_nx, sv, reinterpret_cast<const double*>(sE),
                                        reinterpret_cast<double*>(out));
                    __syncthreads();
                }
            } else {
                __syncthreads();
            }
        }
        // residual r = b - K_T x
        for (int it = tid; it < own * 3 * rn; it += NT) {
            const int2 item = sit[it];
            const int fl = item.y;
            T r = sb[it];
            if (step > 0 && !(fl & FIXED)) {
                if (FX && f64) {
                    // the item's first result, counted in values instead of limbs
                    const int blk = mgc_div(it, a.m_rn), rc = (blk / 3) * 6 + blk % 3;
                    const T* w0 = reinterpret_cast<const T*>(out) + item.x - (size_t)rc * 4 * (NL - 1) * faces;
                    T s = T(0);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const T* w = w0 + q * faces - (q & 1) - (q >> 1) * g.nx;
                        if (fl & (1 << q)) s += w[0] + w[(size_t)12 * faces];
                    }
                    r -= s;
                } else {
                    W s[NL];
#pragma unroll
                    for (int l = 0; l < NL; ++l) s[l] = W(0);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int dx = q & 1, dz = q >> 1;
                        const W* w = out + item.x + q * NL * faces - dx - dz * g.nx;
                        if (fl & (1 << q))
#pragma unroll
                            for (int l = 0; l < NL; ++l) s[l] += w[l * faces] + w[(12 * NL + l) * faces];
                    }
                    if constexpr (FX) r -= scale * gm_fx_to_double(s[0], s[1], s[2]);
                    else r -= s[0];
                }
                if (fl & LIP) {
                    // cohesive force +-A_i D [[x]]
                    const int blk = mgc_div(it, a.m_rn), row = blk / 3, c = blk - row * 3, j = j0 + row;
                    const int i = mgc_div(it - blk * rn, a.m_rowlen), p = it - blk * rn - i * rowlen;
                    const int nl = p + rowlen * g.kf, nu = nl + rowlen;
                    const int nqi = (p > 0) + (p < g.nx), nqj = (j > 0) + (j < g.ny);
                    const T Ai = a.fk.Aq * T(0.25) * T(nqi * nqj);
                    const uint8_t* mk = sm + (size_t)(row + 1) * rn;
                    T f = T(0);
#pragma unroll
                    for (int e = 0; e < 3; ++e) {
                        const T up = ((mk[nu] >> e) & 1u) ? T(0) : xi[(size_t)(row * 3 + e) * rn + nu];
                        const T um = ((mk[nl] >> e) & 1u) ? T(0) : xi[(size_t)(row * 3 + e) * rn + nl];
                        const int lo = c < e ? c : e, hi = c < e ? e : c;
                        f = fma(sD[(size_t)(row * 6 + (lo == 0 ? hi : lo + hi + 1)) * rowlen + p], up - um, f);
                    }
                    r = (fl & UPPER) ? fma(-Ai, f, r) : fma(Ai, f, r);
                }
            }
            sr[it] = r;
        }
        __syncthreads();
        // z = M^-1 r, d = c1 d + c2 z, x = x + d
        for (int it = tid; it < own * 3 * rn; it += NT) {
            const int fl = sit[it].y;
            const int blk = mgc_div(it, a.m_rn), n = it - blk * rn, row = blk / 3, c = blk - row * 3;
            const T* rr = sr + (size_t)row * 3 * rn;
            T z = T(0);
            if (fl & LIP) {
                const int p = n - mgc_div(n, a.m_rowlen) * rowlen, nl = p + rowlen * g.kf;
                const T* P = sP + (size_t)(row * 36 + ((fl & UPPER ? 3 : 0) + c) * 6) * rowlen + p;
#pragma unroll
                for (int e = 0; e < 6; ++e) z = fma(P[(size_t)e * rowlen], rr[(size_t)(e % 3) * rn + nl + (e < 3 ? 0 : rowlen)], z);
            } else {
#pragma unroll
                for (int e = 0; e < 3; ++e) {
                    const int lo = c < e ? c : e, hi = c < e ? e : c;
                    z = fma(mg_ld<T>(smi + (size_t)(row * 6 + (lo == 0 ? hi : lo + hi + 1)) * rn + n), rr[(size_t)e * rn + n], z);
                }
            }
            const T dn = step > 0 ? fma(c1, sd[it], c2 * z) : c2 * z;
            const T xn = step > 0 ? xi[it] + dn : dn;
            sd[it] = dn;
            if (step + 1 < a.deg) xo[it] = xn;
            else a.x[c * N + node(n, j0 + row)] = xn;
        }
        // the step's rows are complete; in the last step: nobody reads this CTA's rows any more
        cl.sync();
    }
}

// Cluster size the kernel runs with on this device (0: not available).  Solvers of
// several threads may ask at the same time: the second waits for the first's answer.
constexpr int MGC_SMEM = 226 * 1024;
template <typename T, typename MT, int CLS>
int mgc_setup(int dev)
{
    static std::mutex lock;
    static int size[64] = {};
    const std::lock_guard<std::mutex> held(lock);
    int& r = size[dev & 63];
    if (r != 0) return r < 0 ? 0 : r;
    const void* k = (const void*)mg_coarse_kernel<T, MT, CLS>;
    r = -1;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, MGC_SMEM) != cudaSuccess ||
        cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
        (void)cudaGetLastError();
        return 0;
    }
    for (int n : {16, 8}) {
        cudaLaunchConfig_t cfg{};
        cudaLaunchAttribute at{};
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = n;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        cfg.gridDim = dim3(n);
        cfg.blockDim = dim3(mgc_threads<T>());
        cfg.dynamicSmemBytes = MGC_SMEM;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        int active = 0;
        if (cudaOccupancyMaxActiveClusters(&active, k, &cfg) == cudaSuccess && active > 0) {
            r = n;
            break;
        }
        (void)cudaGetLastError();
    }
    return r < 0 ? 0 : r;
}

}  // namespace

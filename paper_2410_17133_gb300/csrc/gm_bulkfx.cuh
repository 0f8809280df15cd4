// FP64 bulk products in wide fixed point (gm_fixed.cuh): K_b (u -> u), A_pu
// (p -> u), A_up (u -> p) and S + dt C (p -> p) of gm_bulk.cuh, same operator, tiling and march.
//
// Why: the FP64 kernel is bound by the FP64 pipe (2 lanes per clock and SM).
// In the parity basis a K_b element takes about 210 FP64 instructions, 64
// issue slots each; the same element takes about 2350 integer instructions here
// (560 of them IMAD.WIDE, 2 slots each).  Measured against the FP64 kernel, us
// per product: K_T on 128^3 dipping cells 1256 -> 413; K_T + A_pu + A_up + A22 on
// 61x127x46 cells sheared both ways 806 -> 287 (A22 121 -> 48); J on 8^3 cells
// 90 -> 46.
//
// Each CTA first looks over its inputs: the largest exponent sets the tile's
// unit, and the smallest of the elements' largest exponents says how far the
// field is graded inside the tile.  A tile that is graded by more than 16 bits
// (less the contrast of the moduli), not finite, subnormal, or near the ends of the
// exponent range takes the FP64 tile of gm_bulk.cuh.
//
// The values alone do not say how exact FP64 would be: a field that is constant
// over an element exerts no force however large it is, and the small ones beside
// it (another component, a small strain on a large translation) keep all their
// bits in FP64.  What counts is each element's modes, and they are at hand in
// registers: FP64 rounds a term K_ij x_j by 2^-54 of itself, fixed point loses
// about one unit, so an element is exact enough if, for every field of its
// output, some mode that reaches the field's rows is above the limit from
// which that rounding is the larger (RefFx.limK, limU; FlowFx.lim), or if all of
// them are zero and none of the tile's inputs lost bits.  If an element is not,
// the CTA starts over in FP64, so every element is at least as exact as in
// FP64.  The look costs one comparison per mode and field (K_T on 128^3: 403 -> 410 us).
//
// A thread owns one face, 16 x 16 faces per CTA.  The limbs of the element's
// modes take 63 registers and those of the carried tuples 36: kept in registers
// (232 a thread, 8 warps per SM) the kernel waited for the latency of its own
// multiply-add chains (issue slots 33 % used); with the carry in shared memory
// and both planes of a layer transformed from the ring of staged planes it
// runs 16 warps per SM.  Chunks of planes are as long as fill whole waves (the
// halo layer of a chunk costs as much as an owned one).  The two node rows of
// a face column meet by a shuffle in x and one shared word per limb in y.
#pragma once

#include "gm_bulk.cuh"
#include "gm_fixed.cuh"

constexpr int GM_FX_FLOW = GM_M_S | GM_M_C;
template <int MODE>
struct FxSmem {
    static constexpr int NI = MODE == GM_M_APU || MODE == GM_FX_FLOW ? 1 : 3;
    static constexpr int NO = MODE == GM_M_AUP || MODE == GM_FX_FLOW ? 1 : 3;
    static constexpr int NL = MODE == GM_FX_FLOW ? 4 : 3;   // limbs of a result
    static constexpr bool CARRY = MODE == GM_M_K;      // K_b: the carried tuples live here, not in registers
    int plane[3][NI][3][17 * 17];                      // ring of node planes, limb by limb
    int face[2][NO][NL][256];                          // upper node row of the faces, by plane parity
    int carry[CARRY ? NO * 4 * NL : 1][CARRY ? 256 : 1];
};
template <int MODE>
constexpr size_t gm_fx_smem()
{
    constexpr size_t tile = sizeof(BulkTileSmem<double, MODE == GM_M_AUP ? GM_M_AUP | GM_FX_FLOW : MODE>);
    return sizeof(FxSmem<MODE>) > tile ? sizeof(FxSmem<MODE>) : tile;
}

// Output mode s of displacement field c of one element with modulus limbs E:
// K_b row times the element's input modes, times E (limbs of gm_fx_coef22).
template <int CLS>
__device__ __forceinline__ void gm_fx_k_mode(const RefFx& F, const int (&xv)[24][3], int c, int s, const int (&E)[3],
                                             int (&y)[3])
{
    constexpr ParPat PP = gm_make_parpat(CLS);
    FxAcc acc{0, 0, 0};
#pragma unroll
    for (int j = 0; j < 24; ++j)
        if (PP.k[c * 8 + s][j] >= 0 && (j & 7) != 0) {
            const int* k = F.k[PP.k[c * 8 + s][j]];
            gm_fx_mac3(acc, xv[j], k[2], k[1], k[0]);
        }
    int r[3];
    gm_fx_carry(acc, r);
    FxAcc ae{0, 0, 0};
    gm_fx_mac(ae, r, E[2], E[1], E[0]);
    gm_fx_carry(ae, y);
}

// The FP64 tile as a function of its own: it needs twice the registers, and
// inlined its spills would reach into the fixed-point part.  A_up that adds to the
// flow block's result runs both blocks: its own planes may be written already.
template <int CLS, int MODE>
__device__ __noinline__ void gm_fx_fp64_tile(const BulkArgs<double>& a, const RefOps<double>& R, void* sm)
{
    if constexpr (MODE == GM_M_AUP) {
        constexpr int BOTH = GM_M_AUP | GM_FX_FLOW;
        if (a.accumulate) {
            BulkArgs<double> b = a;
            b.accumulate = 0;
            gm_bulk_tile<double, CLS, BOTH, false>(b, R, *static_cast<BulkTileSmem<double, BOTH>*>(sm));
            return;
        }
    }
    gm_bulk_tile<double, CLS, MODE, false>(a, R, *static_cast<BulkTileSmem<double, MODE>*>(sm));
}

// Input mode j reaches the rows of displacement field c.
template <int CLS>
__host__ __device__ constexpr bool gm_fx_reaches(const ParPat& PP, int c, int j)
{
    for (int s = 1; s < 8; ++s)
        if (PP.k[c * 8 + s][j] >= 0) return true;
    return false;
}
template <int CLS>
__host__ __device__ constexpr bool gm_fx_drains(const ParPat& PP, int j)
{
    for (int s = 0; s < 8; ++s)
        if (PP.a[j][s] >= 0) return true;
    return false;
}

// Whether the element's modes hold its part of K_b x (fields C0 to C0 + NC - 1; or of
// A_up x) as exactly as FP64 would; cut: some input of the tile lost bits below the unit.
template <int CLS, int MODE, int C0 = 0, int NC = MODE == GM_M_K ? 3 : 1>
__device__ __forceinline__ bool gm_fx_exact(const RefFx& F, const int (&xv)[24][3], bool cut)
{
    constexpr ParPat PP = gm_make_parpat(CLS);
    bool ok[NC] = {};
#pragma unroll
    for (int j = 0; j < 24; ++j) {
        if ((j & 7) == 0) continue;
        const int m = abs(xv[j][2]);
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            if constexpr (MODE == GM_M_K) {
                if (gm_fx_reaches<CLS>(PP, C0 + c, j)) ok[c] |= m > F.limK[C0 + c][j];
            } else {
                if (gm_fx_drains<CLS>(PP, j)) ok[c] |= m > F.limU[j];
            }
        }
    }
    bool all = true;
#pragma unroll
    for (int c = 0; c < NC; ++c) all &= ok[c];
    if (all) return true;
    if (cut) return false;
    int any = 0;
#pragma unroll
    for (int c = 0; c < NC; ++c)
        if (!ok[c])
#pragma unroll
            for (int j = 0; j < 24; ++j)
                if ((j & 7) != 0 && (MODE == GM_M_K ? gm_fx_reaches<CLS>(PP, C0 + c, j) : gm_fx_drains<CLS>(PP, j)))
                    any |= xv[j][0] | xv[j][1] | xv[j][2];
    return any == 0;
}
// The same for the flow block: a Darcy mode, or the storage of the mean pressure.
__device__ __forceinline__ bool gm_fx_exact_flow(const FlowFx& Q, const int (&xv)[8][3], bool cut)
{
    bool ok = false;
#pragma unroll
    for (int s = 0; s < 8; ++s) ok |= abs(xv[s][2]) > Q.lim[s];
    if (ok) return true;
    int any = cut;
#pragma unroll
    for (int s = 1; s < 8; ++s) any |= xv[s][0] | xv[s][1] | xv[s][2];
    return any == 0;
}

template <int CLS, int MODE, bool DOT>
__global__ void __launch_bounds__(256, 2)
gm_bulk_fx_kernel(int chained, const __grid_constant__ BulkArgs<double> a, const __grid_constant__ RefFx F,
                  const __grid_constant__ RefOps<double> R, const __grid_constant__ FlowFx Q)
{
    gm_chain(chained);
    constexpr bool DO_K = MODE == GM_M_K;
    constexpr bool DO_APU = MODE == GM_M_APU;
    constexpr bool DO_AUP = MODE == GM_M_AUP;
    constexpr bool DO_Q = MODE == GM_FX_FLOW;
    static_assert(DO_K || DO_APU || DO_AUP || DO_Q, "one block at a time");
    static_assert(!DOT || DO_K || DO_Q, "the dot product belongs to K_b and S + dt C");
    constexpr bool IN_P = DO_APU || DO_Q, OUT_P = DO_AUP || DO_Q;
    constexpr int NI = IN_P ? 1 : 3;
    constexpr int NO = OUT_P ? 1 : 3;
    constexpr int NL = FxSmem<MODE>::NL;
    constexpr int TN = 17, PL = TN * TN;
    constexpr ParPat PP = gm_make_parpat(CLS);
    extern __shared__ __align__(16) unsigned char raw[];
    __shared__ int s_mx[8], s_mn[8], s_lo[8];
    __shared__ double s_dot[8];

    if (a.skip != nullptr && *a.skip != 0) return;

    const GridDesc& g = a.g;
    const int tid = threadIdx.x;
    const int tx = tid & 15, ty = tid >> 4;
    const int x0 = blockIdx.x * 15, y0 = blockIdx.y * 15;
    const int fi = x0 - 1 + tx, fj = y0 - 1 + ty;
    const bool fval = fi >= 0 && fi < g.nx && fj >= 0 && fj < g.ny;
    const int z0 = blockIdx.z * a.zchunk;
    const int z1 = min(z0 + a.zchunk, g.nplanes);
    const int N = (int)g.N, nb = (int)g.nb, rowlen = g.nx + 1;
    const double* xin = IN_P ? a.xp : a.xu;
    auto layer_exists = [&](int kb) -> bool { return kb >= 0 && kb + 1 < g.nplanes && kb != g.kf; };
    auto layer_index = [&](int kb) -> int { return (g.kf >= 0 && kb > g.kf) ? kb - 1 : kb; };
    // node whose value plane kk's node takes: a tied upper lip reads the pressure of the lower lip
    auto src_plane = [&](int kk) -> int { return (IN_P && g.tied && kk == g.kf + 1) ? kk - 1 : kk; };

    // ---- the tile's unit and grading -------------------------------------
    const int kbeg = layer_exists(z0 - 1) ? z0 - 1 : z0;
    const int kend = layer_exists(z1 - 1) ? z1 : z1 - 1;      // last plane read
    int mx = 0, mn = 0x7fffffff, least = 0x7fffffff;    // least: the smallest input that is not zero
    {
        int below = 0;
        for (int kk = kbeg; kk <= kend; ++kk) {
            int m4 = 0;
            if (fval) {
                const int node0 = src_plane(kk) * nb + fj * rowlen + fi;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int node = node0 + (q & 1) + (q >> 1) * rowlen;
                    const unsigned m = a.mask[node];
#pragma unroll
                    for (int f = 0; f < NI; ++f) {
                        // exponent and upper bits; 1 for a value below 2^-1042, which is not zero either
                        const double v = xin[(long long)f * N + node];
                        const int h = __double2hiint(v) & 0x7fffffff, hi = h | (int)(__double2loint(v) != 0);
                        if (!((m >> (IN_P ? 3 : f)) & 1u)) {
                            m4 = max(m4, hi);
                            if (hi != 0) least = min(least, hi);
                        }
                    }
                }
                if (layer_exists(kk - 1) && kk > kbeg) {
                    const int e = max(below, m4);
                    mx = max(mx, e);
                    if (e != 0) mn = min(mn, e);
                }
            }
            below = m4;
        }
        mx = __reduce_max_sync(0xffffffffu, mx);
        mn = __reduce_min_sync(0xffffffffu, mn);
        least = __reduce_min_sync(0xffffffffu, least);
        if ((tid & 31) == 0) { s_mx[tid >> 5] = mx; s_mn[tid >> 5] = mn; s_lo[tid >> 5] = least; }
        __syncthreads();
#pragma unroll
        for (int w = 0; w < 8; ++w) { mx = max(mx, s_mx[w]); mn = min(mn, s_mn[w]); least = min(least, s_lo[w]); }
    }
    const bool zero = mx == 0;
    mx >>= 20;
    mn = min(mn >> 20, mx);
    // a double keeps its 53 bits above the unit, 75 bits below 2^(mx - 1022), within 2^22 of the largest
    const bool cut = mx - min(least >> 20, mx) > 22;
    const int top = zero ? 1023 : mx;
    const int qe = (top - 1022 - GM_FX_IN) + (DO_K ? F.eK + F.topE - 1022 : DO_Q ? Q.eU : F.eA);
    const bool fixed_ok = top < 0x7ff && top >= 100 && qe >= -1000 && qe <= 900 &&
                          (zero || mx - mn <= (DO_K ? F.gradeK : DO_Q ? Q.grade : DO_AUP ? GM_FX_GRADE : F.gradeA));
    auto fp64_tile = [&]() {
        gm_fx_fp64_tile<CLS, MODE>(a, R, raw);
        if constexpr (DOT) {
            // the thread's own outputs times its inputs, off the lips
            double dot = 0.0;
            const int gi = x0 - 1 + tx, gj = y0 - 1 + ty;
            if (tx >= 1 && ty >= 1 && gi <= g.nx && gj <= g.ny)
                for (int kk = z0; kk < z1; ++kk) {
                    if (g.kf >= 0 && (kk == g.kf || kk == g.kf + 1)) continue;
                    const int node = kk * nb + gj * rowlen + gi;
                    if constexpr (DO_Q) dot = fma(a.xp[node], a.yp[node], dot);
                    else
#pragma unroll
                        for (int f = 0; f < 3; ++f)
                            dot = fma(a.xu[(long long)f * N + node], a.yu[(long long)f * N + node], dot);
                }
            gm_cta_dot(dot, s_dot, a.part);
        }
    };
    if (!fixed_ok) {                   // uniform over the CTA
        fp64_tile();
        return;
    }
    FxSmem<MODE>& S = *reinterpret_cast<FxSmem<MODE>*>(raw);
    const double scale = gm_fx_real((int64_t)(qe + 1023) << 52) * a.cfx;

    // ---- staging: tile nodes tid and tid + 256 ------------------------------
    int sl_off[2];
    bool sl_in[2];
#pragma unroll
    for (int sl = 0; sl < 2; ++sl) {
        const int idx = tid + sl * 256;
        const int ni = idx % TN, nj = idx / TN;
        const int gi = x0 - 1 + ni, gj = y0 - 1 + nj;
        sl_in[sl] = idx < PL && gi >= 0 && gi <= g.nx && gj >= 0 && gj <= g.ny;
        sl_off[sl] = gi + rowlen * gj;
    }
    double pf[2][NI];
    auto fetch = [&](int kk) {
#pragma unroll
        for (int sl = 0; sl < 2; ++sl) {
#pragma unroll
            for (int f = 0; f < NI; ++f) pf[sl][f] = 0.0;
            if (!sl_in[sl]) continue;
            const int node = src_plane(kk) * nb + sl_off[sl];
            const unsigned m = a.mask[node];
#pragma unroll
            for (int f = 0; f < NI; ++f)
                if (!((m >> (IN_P ? 3 : f)) & 1u)) pf[sl][f] = xin[(long long)f * N + node];
        }
    };
    auto store = [&](int buf) {
#pragma unroll
        for (int sl = 0; sl < 2; ++sl) {
            if (tid + sl * 256 >= PL) continue;
#pragma unroll
            for (int f = 0; f < NI; ++f) {
                int l[3];
                gm_fx_from_double(pf[sl][f], top, l);
#pragma unroll
                for (int i = 0; i < 3; ++i) S.plane[buf][f][i][tid + sl * 256] = l[i];
            }
        }
    };
    // xy part of the forward transform of the face, limb by limb
    auto fwd_xy = [&](int buf, int f, int (&t)[4][3]) {
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const int* s = &S.plane[buf][f][i][ty * TN + tx];
            const int v00 = s[0], v10 = s[1], v01 = s[TN], v11 = s[TN + 1];
            const int a0 = v00 + v10, a1 = v00 - v10, b0 = v01 + v11, b1 = v01 - v11;
            t[0][i] = a0 + b0;
            t[1][i] = a1 + b1;
            t[2][i] = a0 - b0;
            t[3][i] = a1 - b1;
        }
    };

    // top contributions of the layer below, per output field and tuple
    constexpr bool SC = FxSmem<MODE>::CARRY;
    int rcarry[SC ? 1 : NO][4][NL];
#pragma unroll
    for (int f = 0; f < NO; ++f)
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int i = 0; i < NL; ++i) {
                if constexpr (SC) S.carry[(f * 4 + q) * NL + i][tid] = 0;
                else rcarry[f][q][i] = 0;
            }

    // Output mode `s` of field c from the element's input modes xv.
    auto out_mode = [&](const int (&xv)[NI * 8][3], int c, int s, const int (&E)[3], int (&y)[NL]) {
        FxAcc acc{0, 0, 0};
        if constexpr (DO_K) {
            gm_fx_k_mode<CLS>(F, xv, c, s, E, y);
        } else if constexpr (DO_APU) {
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (PP.a[c * 8 + s][j] >= 0) {
                    const int* k = F.a[PP.a[c * 8 + s][j]];
                    gm_fx_mac(acc, xv[j], k[2], k[1], k[0]);
                }
            gm_fx_carry(acc, y);
        } else if constexpr (DO_Q) {
            // E holds the limbs of the element's dt k/mu; mode 0 has no flow.  The
            // results keep a fourth limb: elements of low permeability lie far
            // below the unit that the most permeable one sets
            FxAcc4 sum{0, 0, 0, 0};
            if (s != 0 && a.cC != 0.0) {
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (PP.l[s][j] >= 0) {
                        const int* k = Q.l[PP.l[s][j]];
                        gm_fx_mac(acc, xv[j], k[2], k[1], k[0]);
                    }
                int r[3];
                gm_fx_carry(acc, r);
                gm_fx_mac4(sum, r, E[2], E[1], E[0]);
            }
            const int* m = Q.m[s];
            gm_fx_mac4(sum, xv[s], m[3], m[2], m[1]);
            sum.am += (int64_t)xv[s][2] * m[0];
            gm_fx_carry4_signed(sum, y);
        } else {
#pragma unroll
            for (int j = 0; j < 24; ++j)
                if (PP.a[j][s] >= 0 && (j & 7) != 0) {
                    const int* k = F.a[PP.a[j][s]];
                    gm_fx_mac(acc, xv[j], k[2], k[1], k[0]);
                }
            gm_fx_carry_signed(acc, y);
        }
    };

    // Layer kb between planes kb and kb + 1 of the ring.  With `plane`, field by
    // field: complete the face tuples of plane kb, transform them back and
    // exchange; in any case the layer's top contributions become the carry.
    int low[NO][NL];
    bool inexact = false;
    auto layer = [&](int kb, bool exists, bool plane) {
        const bool work = exists && fval;
        int xv[NI * 8][3];
        int E[3] = {0, 0, 0};
        if (work) {
            double Ed = 0.0;
            if constexpr (DO_Q) Ed = a.cC * a.kap[fi + (long long)g.nx * (fj + (long long)g.ny * layer_index(kb))];
            if constexpr (DO_K) Ed = a.E[fi + (long long)g.nx * (fj + (long long)g.ny * layer_index(kb))];
            const int sb = (kb - kbeg) % 3, st = (kb + 1 - kbeg) % 3;
#pragma unroll
            for (int f = 0; f < NI; ++f) {
                int b[4][3], t[4][3];
                fwd_xy(sb, f, b);
                fwd_xy(st, f, t);
#pragma unroll
                for (int q = 0; q < 4; ++q)
#pragma unroll
                    for (int i = 0; i < 3; ++i) {
                        xv[f * 8 + q][i] = b[q][i] + t[q][i];
                        xv[f * 8 + q + 4][i] = b[q][i] - t[q][i];
                    }
            }
            if constexpr (DO_K) gm_fx_coef22(Ed, F.topE, E);
            if constexpr (DO_Q) gm_fx_coef(Ed, Q.topW, E);
            if constexpr (DO_K || DO_AUP) inexact |= !gm_fx_exact<CLS, MODE>(F, xv, cut);
            if constexpr (DO_Q)
                if (a.cC != 0.0) inexact |= !gm_fx_exact_flow(Q, xv, cut);
        }
#pragma unroll
        for (int c = 0; c < NO; ++c) {
            int o[4][NL];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                int lo[NL] = {}, hi[NL] = {};
                if (work) {
                    if (OUT_P || q != 0) out_mode(xv, c, q, E, lo);   // mode 0 of u carries no force
                    out_mode(xv, c, q + 4, E, hi);
                }
#pragma unroll
                for (int i = 0; i < NL; ++i) {
                    if constexpr (SC) {
                        int& cy = S.carry[(c * 4 + q) * NL + i][tid];
                        o[q][i] = cy + lo[i] + hi[i];
                        cy = lo[i] - hi[i];
                    } else {
                        o[q][i] = rcarry[c][q][i] + lo[i] + hi[i];
                        rcarry[c][q][i] = lo[i] - hi[i];
                    }
                }
            }
            if (plane) {
#pragma unroll
                for (int i = 0; i < NL; ++i) {
                    const int c0 = o[0][i] + o[1][i], c1 = o[0][i] - o[1][i];
                    const int d0 = o[2][i] + o[3][i], d1 = o[2][i] - o[3][i];
                    const int p10 = __shfl_up_sync(0xffffffffu, c1 + d1, 1, 16);
                    const int p11 = __shfl_up_sync(0xffffffffu, c1 - d1, 1, 16);
                    low[c][i] = c0 + d0 + p10;
                    S.face[kb & 1][c][i][tid] = c0 - d0 + p11;
                }
            }
        }
    };

    double dot = 0.0;
    const int gi = x0 - 1 + tx, gj = y0 - 1 + ty;
    const bool owner = tx >= 1 && ty >= 1 && gi <= g.nx && gj <= g.ny;
    auto node_stage = [&](int kk) {
        if (!owner) return;
        const int node = kk * nb + gj * rowlen + gi;
        const unsigned m = a.mask[node];
        const bool lip = g.kf >= 0 && (kk == g.kf || kk == g.kf + 1);
        // raw value on a tied slave lip: the fault kernel folds it
        const bool slave = OUT_P && g.tied && kk == g.kf + 1;
#pragma unroll
        for (int f = 0; f < NO; ++f) {
            const int(&up)[NL][256] = S.face[kk & 1][f];
            int l[NL];
#pragma unroll
            for (int i = 0; i < NL; ++i) l[i] = low[f][i] + up[i][tid - 16];
            double v;
            if constexpr (DO_Q) v = scale * gm_fx_to_double4(l[0], l[1], l[2], l[3]);
            else v = scale * gm_fx_to_double(l[0], l[1], l[2]);
            double* y = OUT_P ? a.yp + node : a.yu + (long long)f * N + node;
            const bool fixed = !slave && ((m >> (OUT_P ? 3 : f)) & 1u);
            if (a.accumulate) {
                if (!fixed) *y += v;
            } else {
                *y = fixed ? 0.0 : v;
            }
            if constexpr (DOT)
                if (!lip && !fixed) dot = fma(DO_Q ? a.xp[node] : a.xu[(long long)f * N + node], v, dot);
        }
    };

    // Plane k sits in ring slot (k - kbeg) % 3.  While layer kk is computed,
    // plane kk + 2 is on its way into registers; it is stored over plane kk - 1,
    // which nobody reads after this iteration's barrier.  The nodes of plane
    // kk - 1 are written after that barrier too, so a layer needs one barrier.
    fetch(kbeg);
    store(0);
    if (kbeg + 1 <= kend) {
        fetch(kbeg + 1);
        store(1);
    }
    for (int kk = kbeg; kk < z1; ++kk) {
        const bool next = kk + 2 <= kend;
        if (next) fetch(kk + 2);
        if (__syncthreads_or(inexact)) {
            fp64_tile();
            return;
        }
        if (kk > z0) node_stage(kk - 1);
        layer(kk, layer_exists(kk), kk >= z0);
        if (next) store((kk + 2 - kbeg) % 3);
    }
    if (__syncthreads_or(inexact)) {
        fp64_tile();
        return;
    }
    node_stage(z1 - 1);
    if constexpr (DOT) gm_cta_dot(dot, s_dot, a.part);
}

// The whole PCG solve of K in one launch, one CTA per SM, for meshes whose rows
// fit the SMs' shared memory (about 20 k nodes).
//
// On these meshes an iteration is bound by latency: as two launches (product
// with direction and alpha, then the vector step) it took 18.8 us on 4.9 k nodes,
// of which the FP64 pipes worked about 4; this way it takes 13 (a time step of
// 30 such solves: 98 -> 68 ms), more than half of it in the two sums.  Here a CTA
// owns a range of nodes for the whole solve.  Its rows of K, the direction at each of its entries (so p is
// never exchanged), its preconditioner blocks and vectors stay in shared memory
// and registers; only z travels, once per iteration.  The two sums of an
// iteration double as the grid's barriers: each CTA sends its partials to every
// other CTA's box and reads its own, so a store and a load through L2 replace a
// ticket, a last block and a launch, and each word has one reader (with one
// table that all CTAs polled, an iteration took 16 us).
//
// An unwritten word of a box holds the bit pattern GRID_EMPTY (a NaN that no sum
// is stored as); three sets of words take turns.  Waits are bounded: a CTA that
// gives up marks the solve and returns, and so do the others.  The launch is
// cooperative, so all CTAs are resident.  Where the launch is refused or a wait
// runs out, the caller solves with two launches per iteration instead.
// Included by gm_tet.cu only.
#pragma once

#include <type_traits>

namespace {

constexpr int TGRID_NT = 512;
constexpr int TGRID_VW = 10;                          // nodes per warp in the vector part: a lane per component
constexpr int TGRID_ROWS = TGRID_VW * (TGRID_NT / 32);
constexpr int TGRID_MIN_ROWS = 16;                    // fewer do not fill the four schedulers
constexpr int TGRID_CTAS = 256;
constexpr size_t TGRID_SMEM = 208 * 1024;              // beside 12 KB of row vectors
constexpr unsigned long long GRID_EMPTY = ~0ull;
constexpr int TGRID_POLLS = 1 << 23;                  // polls of an L2 word before a wait runs out: some seconds
constexpr int TGRID_LOST = -1;
inline size_t tgrid_box_bytes(int grid) { return (size_t)grid * 3 * TGRID_CTAS * sizeof(ulonglong2); }

struct TetGridArgs {
    int N, rows, maxit;
    double tol2;
    const int* row;
    const int* col;
    const double* K;                     // 9 per entry, as TetCsr
    const double* Kinv;                  // (3 i + j) N + n
    const uint8_t* mask;
    const double* b;
    double* x;
    double* z;                           // 3N: (z0, z1) of each node, then all z2
    ulonglong2* box;                     // per CTA 3 sets of TGRID_CTAS partials; empty at the start
    TetPcgState* st;
    int polls;
};

// entries of a CTA: 9 of K, 3 of the direction, the column
inline size_t tgrid_smem(long long entries) { return (size_t)entries * (9 * 8 + 3 * 8 + 4); }

__device__ inline unsigned long long tgrid_word(double v)
{
    const unsigned long long bits = (unsigned long long)__double_as_longlong(v);
    return bits == GRID_EMPTY ? 0x7ff8000000000000ull : bits;
}
__device__ inline void tgrid_store(ulonglong2* p, ulonglong2 v)
{
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(v.x), "l"(v.y) : "memory");
}
__device__ inline ulonglong2 tgrid_load(const ulonglong2* p)
{
    ulonglong2 v;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(p) : "memory");
    return v;
}

__global__ void __launch_bounds__(TGRID_NT, 1) tet_pcg_grid(const TetGridArgs a)
{
    constexpr int NW = TGRID_NT / 32;
    extern __shared__ double s_dyn[];
    __shared__ double s_q[3][TGRID_ROWS], s_p[3][TGRID_ROWS], s_z[3][TGRID_ROWS];
    __shared__ double s_w[2][NW], s_ab;
    __shared__ int s_row[TGRID_ROWS + 1], s_stop;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, N = a.N;
    const int n0 = blockIdx.x * a.rows, R = min(a.rows, N - n0), G = gridDim.x;
    const int e0 = a.row[n0];
    for (int i = tid; i <= R; i += TGRID_NT) s_row[i] = a.row[n0 + i] - e0;
    if (tid < 2 * NW) s_w[tid / NW][tid % NW] = 0.0;      // warps without nodes add nothing
    __syncthreads();
    const int E = s_row[R];
    double* const s_K = s_dyn;
    double* const s_pe = s_dyn + 9 * (size_t)E;
    int* const s_col = reinterpret_cast<int*>(s_pe + 3 * (size_t)E);
    for (int i = tid; i < 9 * E; i += TGRID_NT) s_K[i] = a.K[9LL * e0 + i];
    for (int i = tid; i < 3 * E; i += TGRID_NT) s_pe[i] = 0.0;
    for (int i = tid; i < E; i += TGRID_NT) s_col[i] = a.col[e0 + i];
    for (int i = tid; i < 3 * TGRID_ROWS; i += TGRID_NT) s_p[i / TGRID_ROWS][i % TGRID_ROWS] = 0.0;

    // vector part: node vr, component vc of this thread
    const int vr = warp * TGRID_VW + lane / 3, vc = lane % 3;
    const bool vec = lane < 3 * TGRID_VW && vr < R;
    const int vwarps = (R + TGRID_VW - 1) / TGRID_VW, vn = n0 + vr;
    double r = 0.0, x = 0.0, ki[3] = {0.0, 0.0, 0.0};
    bool fixed = false;
    if (vec) {
        r = a.b[(long long)vc * N + vn];
        fixed = (a.mask[vn] >> vc) & 1u;
#pragma unroll
        for (int j = 0; j < 3; ++j) ki[j] = a.Kinv[(long long)(3 * vc + j) * N + vn];
    }

    // Sums of va (TWO: and vb) over the vector warps' threads of all CTAs, in ga
    // (gb) of warp 0; one warp polls, so the words see one reader per CTA
    int set = 0;
    double ga = 0.0, gb = 0.0;
    bool lost = false;                   // a wait ran out
    auto grid_sum = [&](double va, double vb, auto two) {
        constexpr bool TWO = decltype(two)::value;
        constexpr int PER = TGRID_CTAS / 32;
        if (warp < vwarps) {
            if constexpr (TWO) {
                // lower half of the warp sums a, the upper half b
                const bool upper = lane >= 16;
                const double give = upper ? va : vb;
                double v = (upper ? vb : va) + __shfl_xor_sync(0xffffffffu, give, 16);
#pragma unroll
                for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                if ((lane & 15) == 0) s_w[upper][warp] = v;
            } else {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) va += __shfl_xor_sync(0xffffffffu, va, o);
                if (lane == 0) s_w[0][warp] = va;
            }
        }
        __syncthreads();
        if (warp == 0) {
            double v = TWO || lane < 16 ? s_w[lane >> 4][lane & 15] : 0.0;
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            ulonglong2 mine;
            mine.x = tgrid_word(__shfl_sync(0xffffffffu, v, 0));
            mine.y = tgrid_word(__shfl_sync(0xffffffffu, v, 16));
            ulonglong2* const here = a.box + (size_t)set * TGRID_CTAS;
            asm volatile("fence.acq_rel.gpu;" ::: "memory");     // releases z of the CTA too
#pragma unroll
            for (int j = 0; j < PER; ++j)
                if (32 * j + lane < G) tgrid_store(here + (size_t)(32 * j + lane) * 3 * TGRID_CTAS + blockIdx.x, mine);
            ulonglong2* from = here + (size_t)blockIdx.x * 3 * TGRID_CTAS + lane;
            ulonglong2 got[PER];
#pragma unroll
            for (int j = 0; j < PER; ++j) {
                got[j].x = got[j].y = 32 * j + lane < G ? GRID_EMPTY : 0ull;
            }
            bool wait = true;
            for (int spin = 0; wait && spin < a.polls; ++spin) {
#pragma unroll
                for (int j = 0; j < PER; ++j)
                    if (got[j].x == GRID_EMPTY || got[j].y == GRID_EMPTY) got[j] = tgrid_load(from + 32 * j);
                wait = false;
#pragma unroll
                for (int j = 0; j < PER; ++j) wait = wait || got[j].x == GRID_EMPTY || got[j].y == GRID_EMPTY;
            }
            asm volatile("fence.acq_rel.gpu;" ::: "memory");
            lost = __any_sync(0xffffffffu, wait);
            double t = 0.0, u = 0.0;
#pragma unroll
            for (int j = 0; j < PER; ++j)
                if (32 * j < G) {
                    t += __longlong_as_double((long long)got[j].x);
                    if constexpr (TWO) u += __longlong_as_double((long long)got[j].y);
                }
            if constexpr (TWO) {
                const bool upper = lane >= 16;
                const double give = upper ? t : u;
                t = (upper ? u : t) + __shfl_xor_sync(0xffffffffu, give, 16);
            } else {
                t += __shfl_xor_sync(0xffffffffu, t, 16);
            }
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            ga = __shfl_sync(0xffffffffu, t, 0);
            gb = __shfl_sync(0xffffffffu, t, 16);
            // Every CTA has sent this sum, so all have read the one before: that set of
            // this CTA's box is emptied for the next but one, whose senders will have
            // acquired this CTA's next partial.
            const int old = set == 0 ? 2 : set - 1;
            from += (old - set) * TGRID_CTAS;
#pragma unroll
            for (int j = 0; j < PER; ++j)
                if (32 * j + lane < G) __stcg(from + 32 * j, make_ulonglong2(GRID_EMPTY, GRID_EMPTY));
            set = set == 2 ? 0 : set + 1;
        }
    };
    // z = M^-1 r of this thread's component, published; terms of r.z and r.r
    auto precondition = [&](double& rz, double& rr) {
        rz = rr = 0.0;
        if (warp < vwarps) {
            const int l0 = lane < 3 * TGRID_VW ? lane - vc : 0;
            const double r0 = __shfl_sync(0xffffffffu, r, l0), r1 = __shfl_sync(0xffffffffu, r, l0 + 1),
                         r2 = __shfl_sync(0xffffffffu, r, l0 + 2);
            if (vec) {
                const double zv = ki[0] * r0 + ki[1] * r1 + ki[2] * r2;
                s_z[vc][vr] = zv;
                __stcg(vc < 2 ? a.z + 2LL * vn + vc : a.z + 2LL * N + vn, zv);
                rz = r * zv;
                rr = r * r;
            }
        }
    };
    using One = std::integral_constant<bool, false>;
    using Two = std::integral_constant<bool, true>;

    double rz, rr, old_rz = 0.0, rr0 = 0.0, beta = 0.0;
    int its = 0, done = 0;
    precondition(rz, rr);
    grid_sum(rz, rr, Two{});
    if (warp == 0) {
        old_rz = ga;
        rr0 = gb;
        done = lost ? TGRID_LOST : gb > 0.0 ? (isfinite(gb) ? 0 : 2) : 1;
        if (lane == 0) s_stop = done;
    }
    __syncthreads();
    done = s_stop;

    while (done == 0) {
        // q = K p by rows, p = z + beta p_old at each entry and at the row's own
        // node; 8 lanes per row
        for (int base = warp * 4; base < R; base += NW * 4) {
            const int lr = base + (lane >> 3), l8 = lane & 7;
            const bool valid = lr < R;
            double q0 = 0.0, q1 = 0.0, q2 = 0.0, u0 = 0.0, u1 = 0.0, u2 = 0.0;
            if (valid) {
                const int rs = s_row[lr], len = s_row[lr + 1] - rs;
                u0 = fma(beta, s_p[0][lr], s_z[0][lr]);
                u1 = fma(beta, s_p[1][lr], s_z[1][lr]);
                u2 = fma(beta, s_p[2][lr], s_z[2][lr]);
                for (int e = l8; e < len; e += 16) {
                    // two entries at a time, so that their loads of z overlap
                    const bool more = e + 8 < len;
                    const int m = s_col[rs + e], m2 = s_col[rs + (more ? e + 8 : e)];
                    const double2 za = __ldcg(reinterpret_cast<const double2*>(a.z) + m);
                    const double zc = __ldcg(a.z + 2LL * N + m);
                    const double2 zb = __ldcg(reinterpret_cast<const double2*>(a.z) + m2);
                    const double zd = __ldcg(a.z + 2LL * N + m2);
                    auto entry = [&](int at, double2 zv, double zw) {
                        double* const pe = s_pe + rs + at;
                        const double p0 = fma(beta, pe[0], zv.x), p1 = fma(beta, pe[E], zv.y),
                                     p2 = fma(beta, pe[2 * E], zw);
                        pe[0] = p0;
                        pe[E] = p1;
                        pe[2 * E] = p2;
                        const double d0 = p0 - u0, d1 = p1 - u1, d2 = p2 - u2;
                        const double* const k = s_K + 9 * rs + at;
                        q0 = fma(k[0], d0, q0);
                        q0 = fma(k[len], d1, q0);
                        q0 = fma(k[2 * len], d2, q0);
                        q1 = fma(k[3 * len], d0, q1);
                        q1 = fma(k[4 * len], d1, q1);
                        q1 = fma(k[5 * len], d2, q1);
                        q2 = fma(k[6 * len], d0, q2);
                        q2 = fma(k[7 * len], d1, q2);
                        q2 = fma(k[8 * len], d2, q2);
                    };
                    entry(e, za, zc);
                    if (more) entry(e + 8, zb, zd);
                }
            }
            // the 8 lanes' sums in four adds: lanes 0-3 keep components 0 and 1,
            // lanes 4-7 component 2, then one component per lane pair
            const bool hi = (lane & 4) != 0, md = (lane & 2) != 0;
            double k0 = (hi ? q2 : q0) + __shfl_xor_sync(0xffffffffu, hi ? q0 : q2, 4);
            double k1 = (hi ? 0.0 : q1) + __shfl_xor_sync(0xffffffffu, hi ? q1 : 0.0, 4);
            double v = (md ? k1 : k0) + __shfl_xor_sync(0xffffffffu, md ? k0 : k1, 2);
            v += __shfl_xor_sync(0xffffffffu, v, 1);
            __syncwarp();                        // the rows' s_p have been read
            if (valid && (lane & 1) == 0 && l8 < 6) {
                const int c = l8 >> 1;
                s_q[c][lr] = v;
                s_p[c][lr] = c == 0 ? u0 : c == 1 ? u1 : u2;
            }
        }
        __syncthreads();
        double pv = 0.0, qv = 0.0;
        if (vec) {
            pv = s_p[vc][vr];
            qv = fixed ? 0.0 : s_q[vc][vr];
        }
        grid_sum(pv * qv, 0.0, One{});
        if (warp == 0) {
            if (lost) done = TGRID_LOST;
            else if (!(ga > 0.0) || !isfinite(ga)) done = 2;
            const double alpha = old_rz / ga;
            if (lane == 0) {
                s_ab = alpha;
                s_stop = done;
            }
        }
        __syncthreads();
        done = s_stop;
        if (done) break;
        const double alpha = s_ab;
        if (vec) {
            r -= alpha * qv;
            x += alpha * pv;
        }
        precondition(rz, rr);
        grid_sum(rz, rr, Two{});
        its += 1;
        if (warp == 0) {
            const double bt = ga / old_rz;
            old_rz = ga;
            if (lost) done = TGRID_LOST;
            else if (!isfinite(gb) || !isfinite(ga)) done = 2;
            else if (gb <= a.tol2 * rr0) done = 1;
            else if (its >= a.maxit) done = 3;
            if (lane == 0) {
                s_ab = bt;
                s_stop = done;
            }
        }
        __syncthreads();
        done = s_stop;
        beta = s_ab;
    }
    if (done == TGRID_LOST) {
        if (tid == 0) a.st->ticket = 1u;
        return;
    }
    if (done == 1 && vec) a.x[(long long)vc * N + vn] = x;
    if (blockIdx.x == 0 && tid == 0) {
        a.st->its = its;
        a.st->done = done;
    }
}

// Node rows per CTA for the mesh, 0 where the solve keeps its two launches per
// iteration: rows that do not fit (more FP64 work than latency by then), or a
// device without cooperative launches, or GM_TET_GRID=0.  crow: N + 1 row starts.
inline int tgrid_plan(int device, int N, const std::vector<int>& crow, size_t& smem, int& grid)
{
    const char* wanted = std::getenv("GM_TET_GRID");
    if (wanted && std::atoi(wanted) == 0) return 0;
    int sms = 0, coop = 0, occ = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess ||
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, device) != cudaSuccess || !coop) {
        (void)cudaGetLastError();
        return 0;
    }
    const int ctas = std::min(sms, TGRID_CTAS);
    const int rows = std::max(TGRID_MIN_ROWS, (N + ctas - 1) / ctas);
    if (rows > TGRID_ROWS) return 0;
    long long most = 0;
    for (int n = 0; n < N; n += rows) most = std::max<long long>(most, crow[std::min(N, n + rows)] - crow[n]);
    smem = tgrid_smem(most);
    grid = (N + rows - 1) / rows;
    if (smem > TGRID_SMEM) return 0;
    if (cudaFuncSetAttribute(tet_pcg_grid, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TGRID_SMEM) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, tet_pcg_grid, TGRID_NT, smem) != cudaSuccess || occ < 1) {
        (void)cudaGetLastError();
        return 0;
    }
    return rows;
}

// polls of a wait: GM_TET_GRID_POLLS for the tests of what follows when one runs out
inline int tgrid_polls()
{
    const char* v = std::getenv("GM_TET_GRID_POLLS");
    const int n = v ? std::atoi(v) : TGRID_POLLS;
    return n < 0 ? 0 : n < TGRID_POLLS ? n : TGRID_POLLS;
}

// x = K^-1 b on the stream; 0, 2 / 3 (breakdown / iteration limit), 5 (not solved: the
// launch was refused or a wait between the CTAs ran out) or -1 (CUDA error); *its += iterations
inline int tgrid_solve(const TetGridArgs& a, int grid, size_t smem, cudaStream_t s, long long* its)
{
    if (cudaMemsetAsync(a.box, 0xff, tgrid_box_bytes(grid), s) != cudaSuccess ||
        cudaMemsetAsync(a.st, 0, sizeof(TetPcgState), s) != cudaSuccess)
        return -1;
    TetGridArgs copy = a;
    void* args[] = {&copy};
    if (cudaLaunchCooperativeKernel((const void*)tet_pcg_grid, dim3(grid), dim3(TGRID_NT), args, smem, s) != cudaSuccess) {
        (void)cudaGetLastError();
        return 5;
    }
    TetPcgState h;
    if (cudaMemcpyAsync(&h, a.st, sizeof(h), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return -1;
    if (h.ticket != 0u) return 5;
    *its += h.its;
    return h.done == 1 ? 0 : h.done;
}

}  // namespace

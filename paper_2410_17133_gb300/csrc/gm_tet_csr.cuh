// Assembled operators of the tetrahedral path: one block row per node.
//
// The mesh and the uniform materials stay fixed over many products, and GB300
// issues FP64 at 2 lanes per clock and SM.  Walking a node's ~24 incident
// elements recomputes each element's strain at each of its four nodes, about
// 60 FP64 instructions per visit, 1,440 per node and K product; the assembled
// row has ~15 entries of 9 products.  Per entry (node n, vertex m of one of its
// elements): K (9), A_pu and A_up (3 + 3, alpha in them), S and C (1 + 1); the
// rows of an entry kind are stored component by component inside the node's
// row, so 8 lanes of a row read neighbouring words.  8 lanes per row: with 32
// half of them idle on 15 entries and the FP64 adds of the shuffle tree cost
// as much as the products, with 1 the small meshes leave most SMs without work.
// Measured (36 k nodes, 197 k tetrahedra, FP64; K, A_pu, A_up, A22 and J in
// turn): 652 us walking the elements, 94 us by rows.  What bounds it: the FP64
// pipe (K: 12 instructions per entry and 9 for the lanes' sums), then the rows'
// 140 B per entry from L2.
//
// Sums run in a fixed order (the node's elements as stored, then lanes), so
// results repeat bit by bit.  Included by gm_tet.cu only.
#pragma once

namespace {

constexpr int TCSR_CAND = 256;       // candidate vertices of a node kept in shared memory (per warp)

// Distinct vertices of the elements around each node, in order of first
// appearance: their number (cols null) or the list itself, with each entry's
// row.  One warp per node.
__global__ void __launch_bounds__(128) tcsr_neighbours(int N, const int* rowptr, const int* adj, const int* tets,
                                                       int* count, const int* crow, int* cols, int* rows)
{
    __shared__ int s_v[4][TCSR_CAND];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long wid = (long long)blockIdx.x * 4 + w;
    if (wid >= N) return;
    const int n = (int)wid;
    const int r0 = rowptr[n];
    const long long C = 4LL * (rowptr[n + 1] - r0);
    auto vertex = [&](long long c) -> int { return tets[4 * (adj[r0 + (c >> 2)] >> 2) + (int)(c & 3)]; };
    for (long long c = lane; c < C && c < TCSR_CAND; c += 32) s_v[w][c] = vertex(c);
    __syncwarp();
    int found = 0;
    for (long long c0 = 0; c0 < C; c0 += 32) {
        const long long c = c0 + lane;
        bool first = c < C;
        const int v = first ? (c < TCSR_CAND ? s_v[w][c] : vertex(c)) : -1;
        for (long long d = 0; first && d < c; ++d)
            if ((d < TCSR_CAND ? s_v[w][d] : vertex(d)) == v) first = false;
        const unsigned b = __ballot_sync(0xffffffffu, first);
        if (cols != nullptr && first) {
            const long long at = crow[n] + found + __popc(b & ((1u << lane) - 1u));
            cols[at] = v;
            rows[at] = n;
        }
        found += __popc(b);
    }
    if (cols == nullptr && lane == 0) count[n] = found;
}

// Entry values from the elements that hold both its nodes (one thread per entry):
//   K = sum V (lambda g_n g_m^T + mu g_m g_n^T + mu (g_n.g_m) I),  A_pu = alpha sum (V/4) g_n,
//   A_up = alpha sum (V/4) g_m,  S = sum (V/20 M)(1 + delta_nm),  C = (k/mu_f) sum V g_n.g_m
__global__ void __launch_bounds__(128) tcsr_values(long long nnz, const int* rowptr, const int* adj, const int* tets,
                                                   const double* G, const double* V, const int* crow, const int* cols,
                                                   const int* rows, double lam, double mu, double alpha, double invM,
                                                   double cond, double* K, double* A, double* SC)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nnz) return;
    const int n = rows[i], m = cols[i];
    double M[3][3] = {}, a[3] = {}, b[3] = {}, vol = 0.0;
    for (int q = rowptr[n]; q < rowptr[n + 1]; ++q) {
        const int e = adj[q] >> 2, la = adj[q] & 3;
        int lb = -1;
#pragma unroll
        for (int v = 0; v < 4; ++v)
            if (tets[4 * e + v] == m) lb = v;
        if (lb < 0) continue;
        const double* ga = G + 12LL * e + 3 * la;
        const double* gb = G + 12LL * e + 3 * lb;
        const double ve = V[e];
#pragma unroll
        for (int x = 0; x < 3; ++x) {
            const double vg = ve * ga[x];
            a[x] += vg;
            b[x] = fma(ve, gb[x], b[x]);
#pragma unroll
            for (int y = 0; y < 3; ++y) M[x][y] = fma(vg, gb[y], M[x][y]);
        }
        vol += ve;
    }
    const long long base = crow[n];
    const int len = crow[n + 1] - crow[n], at = (int)(i - base);
    const double tr = M[0][0] + M[1][1] + M[2][2];
#pragma unroll
    for (int x = 0; x < 3; ++x) {
#pragma unroll
        for (int y = 0; y < 3; ++y) {
            double k = fma(lam, M[x][y], mu * M[y][x]);
            if (x == y) k = fma(mu, tr, k);
            K[9 * base + (long long)(3 * x + y) * len + at] = k;
        }
        A[6 * base + (long long)x * len + at] = 0.25 * alpha * a[x];
        A[6 * base + (long long)(3 + x) * len + at] = 0.25 * alpha * b[x];
    }
    SC[2 * base + at] = 0.05 * invM * vol * (n == m ? 2.0 : 1.0);
    SC[2 * base + len + at] = cond * tr;
}

__global__ void __launch_bounds__(256) tcsr_cast(long long n, const double* x, float* y)
{
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        y[i] = (float)x[i];
}

template <typename T>
struct TetCsr {
    const int* row;      // N + 1
    const int* col;
    const T* K;          // 9 per entry
    const T* A;          // 6 per entry
    const T* SC;         // 2 per entry
};

// y = A x by rows, 8 lanes each.  Rows of K, A_up and C sum to zero (the
// gradients of an element do), so these act on the differences x_m - x_n: the
// result keeps the accuracy of strains formed from differences, also where x
// is nearly constant.  PCG (K only): x is the new direction z + beta p_old,
// formed where it is gathered and written to p_new by its own row; constrained
// entries of y are set to 0, p.q is summed over the grid and the last block
// forms alpha.
template <typename T, int MODE, bool PCG>
__global__ void __launch_bounds__(TPCG_NT) tcsr_apply(int chained, int N, const TetCsr<T> A, T cApu, T cC, const T* xu, const T* xp,
                                                      T* yu, T* yp, const int* skip, const TetDir<T> dir)
{
    gm_chain(chained);
    if (skip != nullptr && *skip != 0) return;
    constexpr bool IN_U = (MODE & (TM_K | TM_AUP)) != 0;
    constexpr bool IN_P = (MODE & (TM_APU | TM_S | TM_C)) != 0;
    constexpr bool OUT_U = (MODE & (TM_K | TM_APU)) != 0;
    constexpr bool OUT_P = (MODE & (TM_AUP | TM_S | TM_C)) != 0;
    const long long id = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int n = (int)(id >> 3), lane = threadIdx.x & 7;
    const bool valid = (id >> 3) < N;
    T au[3] = {T(0), T(0), T(0)}, ap = T(0);
    T un[3] = {T(0), T(0), T(0)}, pn = T(0);
    const T beta = PCG ? (T)dir.st->beta : T(0);
    auto in_u = [&](int m, T (&u)[3]) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const long long k = (long long)c * N + m;
            if constexpr (PCG) u[c] = fma(beta, dir.p_old[k], dir.z[k]);
            else u[c] = xu[k];
        }
    };
    if (valid) {
        if constexpr (IN_U) in_u(n, un);
        if constexpr (IN_P) pn = xp[n];
        const long long base = A.row[n];
        const int len = A.row[n + 1] - A.row[n];
        for (int e = lane; e < len; e += 8) {
            const int m = A.col[base + e];
            T u[3] = {T(0), T(0), T(0)}, p = T(0);
            if constexpr (IN_U) {
                in_u(m, u);
#pragma unroll
                for (int c = 0; c < 3; ++c) u[c] -= un[c];
            }
            if constexpr (IN_P) p = xp[m];
            if constexpr ((MODE & TM_K) != 0) {
                const T* k = A.K + 9 * base + e;
#pragma unroll
                for (int x = 0; x < 3; ++x)
#pragma unroll
                    for (int y = 0; y < 3; ++y) au[x] = fma(k[(long long)(3 * x + y) * len], u[y], au[x]);
            }
            if constexpr ((MODE & TM_APU) != 0) {
                const T* k = A.A + 6 * base + e;
                const T pc = cApu * p;
#pragma unroll
                for (int x = 0; x < 3; ++x) au[x] = fma(k[(long long)x * len], pc, au[x]);
            }
            if constexpr ((MODE & TM_AUP) != 0) {
                const T* k = A.A + 6 * base + 3LL * len + e;
#pragma unroll
                for (int x = 0; x < 3; ++x) ap = fma(k[(long long)x * len], u[x], ap);
            }
            if constexpr ((MODE & (TM_S | TM_C)) != 0) {
                const T* k = A.SC + 2 * base + e;
                ap = fma(k[0], p, ap);
                ap = fma(cC * k[len], p - pn, ap);
            }
        }
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
        if constexpr (OUT_U) {
#pragma unroll
            for (int c = 0; c < 3; ++c) au[c] += __shfl_xor_sync(0xffffffffu, au[c], o);
        }
        if constexpr (OUT_P) ap += __shfl_xor_sync(0xffffffffu, ap, o);
    }
    double pq = 0.0;
    if constexpr (OUT_U) {
        // lanes 0-2 of the row write one component each
        if (valid && lane < 3) {
            T v = lane == 0 ? au[0] : lane == 1 ? au[1] : au[2];
            if constexpr (PCG) {
                const T pl = lane == 0 ? un[0] : lane == 1 ? un[1] : un[2];
                dir.p_new[(long long)lane * N + n] = pl;
                if ((dir.mask[n] >> lane) & 1u) v = T(0);
                pq = (double)pl * (double)v;
            }
            yu[(long long)lane * N + n] = v;
        }
    }
    if constexpr (OUT_P) {
        if (valid && lane == 3) yp[n] = ap;
    }
    if constexpr (PCG) {
        double PQ, unused;
        if (tpcg_reduce2(pq, 0.0, dir.part, &dir.st->ticket, PQ, unused)) {
            if (!(PQ > 0.0) || !isfinite(PQ)) dir.st->done = 2;
            else dir.st->alpha = dir.st->rz / PQ;
        }
    }
}

}  // namespace

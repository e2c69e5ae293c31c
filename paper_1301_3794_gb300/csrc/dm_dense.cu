// Dense kernels of the coarsest multigrid level: blocked Gauss-Jordan inversion
// with partial pivoting, the dense product of the coarsest solve,
// and connected components of the active coarsest cells (the scalar Laplacian
// D A D^T has one constant null vector per component; the lowest-index cell of
// each component is pinned to zero).
#include <cooperative_groups.h>

#include "dm_common.cuh"

namespace dm {

namespace {

// ---- in-place inverse by blocked Gauss-Jordan elimination ---------------------
// The steps of a panel of NB columns act on the rest of the matrix as one
// update: with E the product of the panel's elimination steps and J its rows,
// E v = (v with its J entries zeroed) + M v_J, and the in-place panel holds M.
// So a cluster of blocks eliminates within the panel (its rows in registers), the
// row swaps are carried to the other columns, and one rank-NB update over the whole
// chip follows.  The panels bound it, 5 to 6 us a column in two cluster barriers, the
// pivot search and a divide (89 us a panel against 20 an update on the smoke test's
// 400 columns, 5.3 ms against 1.3 in all on the 16^3 sphere, 16.7 against 13.3 on the 96^3
// ellipsoid); the n^3 FP64 FMAs of the updates (two per clock and SM) come next.  A
// step per column instead, as an n x 2n elimination of [A | I], did twice those FMAs
// and two launches for each of the n columns, every launch waiting on one block's
// pivot search.
// Measured (CUDA events), both coarsest inverses of an operator: 96^3 ellipsoid (2,600
// columns in all) 80 -> 31.5 ms, 16^3 sphere (920 columns) 20 -> 7.1 ms.

// The panel goes to a cluster of eight blocks, an eighth of the rows each: its
// own n NB^2 FMAs on one SM's FP64 pipe took 180-290 us, more than the update.
constexpr int kPanelBlocks = 8, kPanelThreads = 256, kPanel = 16;

// Eliminate the panel of columns k0 .. k0 + nb - 1 (nb <= kPanel) of the n x n
// row-major W in place, with partial pivoting over the rows k0 + p and below;
// RPT rows per thread.  piv[k0 + p]: the row swapped with k0 + p.
// Mt[p n + r]: the panel after it; swaps[0 .. 2 nb): destination rows of the
// swaps, swaps[2 kPanel .. 2 kPanel + 2 nb): the rows their contents come from.
template <int RPT>
__global__ void __cluster_dims__(kPanelBlocks, 1, 1) __launch_bounds__(kPanelThreads)
    k_gj_panel(double* __restrict__ W, int n, int k0, int nb, int* __restrict__ piv, double* __restrict__ Mt,
               int* __restrict__ swaps, int* __restrict__ flag) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    constexpr int NB = kPanel, NW = kPanelThreads / 32, NC = kPanelBlocks * NW;   // NC candidates per column
    // by column parity: a block may write the next column's entries while another still reads this one's
    __shared__ double s_best[2][NC];
    __shared__ int s_idx[2][NC];
    __shared__ double s_prow[2][NB], s_krow[2][NB];   // the scaled pivot row, and row k0 + p
    __shared__ int s_piv[NB];
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5, rank = (int)cluster.block_rank();
    const int per = (n + kPanelBlocks - 1) / kPanelBlocks;
    const int rend = min(n, (rank + 1) * per);
    const int r0 = rank * per + t;   // this thread's rows: r0 + i kPanelThreads, below rend
    double a[RPT][NB];
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
        const int r = r0 + i * kPanelThreads;
#pragma unroll
        for (int q = 0; q < NB; ++q) a[i][q] = (r < rend && q < nb) ? W[(size_t)r * n + k0 + q] : 0.0;
    }
    cluster.sync();   // every block runs before another writes to its shared memory
#pragma unroll
    for (int p = 0; p < NB; ++p) {
        if (p < nb) {
            const int buf = p & 1;
            double bv = -1.0;
            int bi = k0 + p;
#pragma unroll
            for (int i = 0; i < RPT; ++i) {
                const int r = r0 + i * kPanelThreads;
                const double v = fabs(a[i][p]);
                if (r >= k0 + p && r < rend && v > bv) {
                    bv = v;
                    bi = r;
                }
            }
            auto best = [&](int o) {
                const double ov = __shfl_xor_sync(0xffffffffu, bv, o);
                const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
                if (ov > bv || (ov == bv && oi < bi)) {
                    bv = ov;
                    bi = oi;
                }
            };
            for (int o = 16; o > 0; o >>= 1) best(o);
            if (lane < kPanelBlocks) {
                *cluster.map_shared_rank(&s_best[buf][rank * NW + wid], lane) = bv;
                *cluster.map_shared_rank(&s_idx[buf][rank * NW + wid], lane) = bi;
            }
            cluster.sync();
            bv = s_best[buf][lane];
            bi = s_idx[buf][lane];
#pragma unroll
            for (int e = 32; e < NC; e += 32) {
                const double ov = s_best[buf][e + lane];
                const int oi = s_idx[buf][e + lane];
                if (ov > bv || (ov == bv && oi < bi)) {
                    bv = ov;
                    bi = oi;
                }
            }
            for (int o = 16; o > 0; o >>= 1) best(o);
            const int pr = bi;   // the same in every thread of the cluster
            const bool found = bv > 1e-300;
            if (!found) {   // every thread alike: no block is left waiting
                if (rank == 0 && t == 0) *flag = 1;
                return;
            }
            if (t == 0) s_piv[p] = pr;
            // the warps that hold the pivot row and row k0 + p send them to every block
#pragma unroll
            for (int i = 0; i < RPT; ++i) {
                const int w0 = rank * per + i * kPanelThreads + 32 * wid;   // this warp's rows: w0 .. w0 + 31, below rend
                const int wend = min(rend, w0 + 32);
                if (pr >= w0 && pr < wend) {
                    const double inv = 1.0 / __shfl_sync(0xffffffffu, a[i][p], pr - w0);
#pragma unroll
                    for (int q = 0; q < NB; ++q) {
                        const double v = __shfl_sync(0xffffffffu, a[i][q], pr - w0);
                        if (lane < kPanelBlocks) *cluster.map_shared_rank(&s_prow[buf][q], lane) = q == p ? inv : v * inv;
                    }
                }
                if (k0 + p >= w0 && k0 + p < wend) {
#pragma unroll
                    for (int q = 0; q < NB; ++q) {
                        const double v = __shfl_sync(0xffffffffu, a[i][q], k0 + p - w0);
                        if (lane < kPanelBlocks) *cluster.map_shared_rank(&s_krow[buf][q], lane) = v;
                    }
                }
            }
            cluster.sync();
#pragma unroll
            for (int i = 0; i < RPT; ++i) {
                const int r = r0 + i * kPanelThreads;
                if (r == k0 + p && r < rend) {
#pragma unroll
                    for (int q = 0; q < NB; ++q) a[i][q] = s_prow[buf][q];
                } else if (r < rend) {
                    if (r == pr) {
#pragma unroll
                        for (int q = 0; q < NB; ++q) a[i][q] = s_krow[buf][q];
                    }
                    const double f = -a[i][p];
                    a[i][p] = 0.0;
#pragma unroll
                    for (int q = 0; q < NB; ++q) a[i][q] = fma(f, s_prow[buf][q], a[i][q]);
                }
            }
        }
    }
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
        const int r = r0 + i * kPanelThreads;
        if (r < rend) {
#pragma unroll
            for (int q = 0; q < NB; ++q)
                if (q < nb) {
                    W[(size_t)r * n + k0 + q] = a[i][q];
                    Mt[(size_t)q * n + r] = a[i][q];
                }
        }
    }
    __syncthreads();
    if (rank == 0 && t < nb) piv[k0 + t] = s_piv[t];
    if (rank == 0 && t < 2 * nb) {
        // the row a destination's content comes from: follow the swaps backwards
        const int d = t < nb ? k0 + t : s_piv[t - nb];
        int from = d;
        for (int p = nb - 1; p >= 0; --p) {
            if (from == k0 + p) from = s_piv[p];
            else if (from == s_piv[p]) from = k0 + p;
        }
        swaps[t] = d;
        swaps[2 * NB + t] = from;
    }
}

// Carry the panel's row swaps to the other columns (one thread each) and copy
// their rows k0 .. k0 + nb - 1 to B[p n + j].
__global__ void k_gj_swap(double* __restrict__ W, int n, int k0, int nb, const int* __restrict__ swaps,
                          double* __restrict__ B, const int* __restrict__ flag) {
    constexpr int NB = kPanel;
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (*flag || j >= n || (j >= k0 && j < k0 + nb)) return;
    double v[2 * NB];
#pragma unroll
    for (int e = 0; e < 2 * NB; ++e)
        if (e < 2 * nb) v[e] = W[(size_t)swaps[2 * NB + e] * n + j];
#pragma unroll
    for (int e = 0; e < 2 * NB; ++e)
        if (e < 2 * nb) W[(size_t)swaps[e] * n + j] = v[e];
#pragma unroll
    for (int e = 0; e < NB; ++e)
        if (e < nb) B[(size_t)e * n + j] = v[e];
}

// W(i, j) <- (0 in the panel's rows, else W(i, j)) + sum_p M(i, p) B(p, j) off
// the panel's columns; 64 x 64 tiles, 4 x 4 per thread
__global__ void __launch_bounds__(256) k_gj_update(double* __restrict__ W, int n, int k0, int nb,
                                                   const double* __restrict__ Mt, const double* __restrict__ B,
                                                   const int* __restrict__ flag) {
    constexpr int NB = kPanel;
    if (*flag) return;
    __shared__ double sm[NB][64], sb[NB][64];
    const int i0 = blockIdx.y * 64, j0 = blockIdx.x * 64;
    const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
    for (int e = t; e < NB * 64; e += 256) {
        const int p = e >> 6, c = e & 63;
        sm[p][c] = (p < nb && i0 + c < n) ? Mt[(size_t)p * n + i0 + c] : 0.0;
        sb[p][c] = (p < nb && j0 + c < n) ? B[(size_t)p * n + j0 + c] : 0.0;
    }
    double acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int i = i0 + ty + 16 * a, j = j0 + tx + 16 * b;
            acc[a][b] = (i < n && j < n && !(i >= k0 && i < k0 + nb)) ? W[(size_t)i * n + j] : 0.0;
        }
    __syncthreads();
#pragma unroll
    for (int p = 0; p < NB; ++p) {
        double m[4], v[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            m[a] = sm[p][ty + 16 * a];
            v[a] = sb[p][tx + 16 * a];
        }
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) acc[a][b] = fma(m[a], v[b], acc[a][b]);
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int i = i0 + ty + 16 * a, j = j0 + tx + 16 * b;
            if (i < n && j < n && !(j >= k0 && j < k0 + nb)) W[(size_t)i * n + j] = acc[a][b];
        }
}

// The row swaps of the elimination are column swaps of the inverse, in reverse
// order: src[d] = the column of W that belongs in column d.
__global__ void k_gj_columns(int n, const int* __restrict__ piv, int* __restrict__ src) {
    __shared__ int sp[1024];
    const int d = blockIdx.x * blockDim.x + threadIdx.x;
    int from = d;
    for (int k0 = 0; k0 < n; k0 += 1024) {
        __syncthreads();
        for (int e = threadIdx.x; e < 1024; e += blockDim.x) sp[e] = k0 + e < n ? piv[k0 + e] : k0 + e;
        __syncthreads();
        const int m = min(1024, n - k0);
        for (int e = 0; e < m; ++e) {
            const int k = k0 + e, q = sp[e];
            from = from == k ? q : (from == q ? k : from);
        }
    }
    if (d < n) src[d] = from;
}
__global__ void k_gj_gather(const double* __restrict__ W, double* __restrict__ M, int n, const int* __restrict__ src) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < n) M[(size_t)blockIdx.y * n + j] = W[(size_t)blockIdx.y * n + src[j]];
}

template <int RPT>
void gj_eliminate(double* W, int n, int* piv, double* Mt, double* B, int* swaps, int* d_flag, cudaStream_t s) {
    const int nt = (n + 63) / 64;
    for (int k0 = 0; k0 < n; k0 += kPanel) {
        const int nb = std::min(kPanel, n - k0);
        launch("k_gj_panel", k_gj_panel<RPT>, kPanelBlocks, kPanelThreads, 0, s, W, n, k0, nb, piv, Mt, swaps, d_flag);
        launch("k_gj_swap", k_gj_swap, (n + 63) / 64, 64, 0, s, W, n, k0, nb, (const int*)swaps, B, (const int*)d_flag);
        launch("k_gj_update", k_gj_update, dim3(nt, nt), 256, 0, s, W, n, k0, nb, (const double*)Mt, (const double*)B,
               (const int*)d_flag);
    }
}

// x[list[r]] = sum_c M(r, c) f[list[c]]: the coarsest solve in one launch (a
// gather, a product and a scatter before, and a memset of x, whose other entries
// nothing writes).  Every block gathers f into shared memory; one warp per row,
// whose first loads are issued before the gather is waited for.
// FP32 inverse (storage types FP32 and BF16): the products of two FP32 numbers
// are summed in three FP32 numbers (error-free products and sums, only the third
// rounds: about 70 bits), because converting and adding in FP64 issues at two per
// clock and SM where this takes two dozen FP32 instructions at 128.  An FP64 sum
// keeps 53 bits; two FP32 numbers, about 48, leave 30 to 100 times its error where
// a sum cancels.  Where FP32's range could show (a product or sum past its end, or
// a result so small that its products' errors fall below it) the row is summed
// again in FP64.
// Measured (CUDA events, of which some 4 us a launch are the events): n = 1,990
// in FP32, 24.9 + 6.7 + 6.4 -> 14.9 us a solve with two FP32 numbers.  The third took 2 us
// more, which four gathers in flight at a time (one before) give back: n = 650 / 1,817 /
// 2,278 with two numbers 8.5 / 14.5 / 14.5 us, with three 10.2 / 16.5 / 16.5, and now 8.8 /
// 14.4 / 16.5; in FP64 10.6 / 19.0 / 18.8 -> 9.8 / 18.5 / 19.3.  (Eight in flight, 16 warps a
// block or packed pairs of FP32 numbers are no faster.)
constexpr int kSolveWarps = 8, kSolveGather = 4;
template <typename T>
__global__ void __launch_bounds__(32 * kSolveWarps) k_coarse_solve(int n, const double* __restrict__ M64,
                                                                   const float* __restrict__ M32,
                                                                   const int* __restrict__ list,
                                                                   const unsigned char* __restrict__ zero_rows,
                                                                   const T* f, T* __restrict__ x) {
    using C = typename Compute<T>::type;
    extern __shared__ __align__(16) unsigned char solve_smem[];
    C* const sf = reinterpret_cast<C*>(solve_smem);
    const int lane = threadIdx.x & 31;
    const int row = blockIdx.x * kSolveWarps + (threadIdx.x >> 5);
    const C* m;
    if constexpr (std::is_same<C, double>::value) m = M64;
    else m = M32;
    m += (size_t)min(row, n - 1) * n;
    constexpr int U = sizeof(C) == 8 ? 8 : 16;
    C v[U];
#pragma unroll
    for (int e = 0; e < U; ++e) v[e] = lane + 32 * e < n ? m[lane + 32 * e] : C(0);
    // f's places, kSolveGather at a time, so that their loads and f's are in flight together (the
    // places need nothing from the kernels before)
    constexpr int NT = 32 * kSolveWarps;
    int at[kSolveGather];
    auto places = [&](int c0) {
#pragma unroll
        for (int e = 0; e < kSolveGather; ++e) {
            const int c = c0 + NT * e;
            at[e] = c < n ? list[c] : -1;
            if (zero_rows && c < n && zero_rows[c]) at[e] = -1;
        }
    };
    places(threadIdx.x);
    chain_wait();
    for (int c0 = threadIdx.x; c0 < n; c0 += NT * kSolveGather) {
        C fv[kSolveGather];
#pragma unroll
        for (int e = 0; e < kSolveGather; ++e) fv[e] = at[e] >= 0 ? (C)to_c(f[at[e]]) : C(0);
        places(c0 + NT * kSolveGather);
#pragma unroll
        for (int e = 0; e < kSolveGather; ++e)
            if (c0 + NT * e < n) sf[c0 + NT * e] = fv[e];
    }
    __syncthreads();
    if (row >= n) return;
    C s = C(0), e1 = C(0), e2 = C(0);
    // a + b exactly as the rounded sum (into a) and its error
    [[maybe_unused]] auto two_sum = [](C& a, C b) {
        const C t = a + b, bp = t - a;
        const C err = (a - (t - bp)) + (b - bp);
        a = t;
        return err;
    };
    for (int c0 = lane; c0 < n; c0 += 32 * U) {
        C cur[U];
#pragma unroll
        for (int e = 0; e < U; ++e) cur[e] = v[e];
#pragma unroll
        for (int e = 0; e < U; ++e) {
            const int c = c0 + 32 * (U + e);
            v[e] = c < n ? m[c] : C(0);
        }
#pragma unroll
        for (int e = 0; e < U; ++e) {
            const int c = c0 + 32 * e;
            if (c < n) {
                if constexpr (std::is_same<C, double>::value) {
                    s = fma(cur[e], sf[c], s);
                } else {
                    const float pr = __fmul_rn(cur[e], sf[c]);
                    const float pe = fmaf(cur[e], sf[c], -pr);
                    const float err = two_sum(s, pr);
                    const float r1 = two_sum(e1, err), r2 = two_sum(e1, pe);
                    e2 += r1 + r2;
                }
            }
        }
    }
    double tot = (double)s + ((double)e1 + (double)e2);
    auto over_lanes = [&] {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) tot += __shfl_down_sync(0xffffffffu, tot, o);
    };
    over_lanes();
    if constexpr (!std::is_same<C, double>::value) {
        const double mag = fabs(__shfl_sync(0xffffffffu, tot, 0));
        if (!(mag >= 0x1p-60 && mag <= 0x1p126)) {
            tot = 0.0;
            for (int c = lane; c < n; c += 32) tot = fma((double)m[c], (double)sf[c], tot);
            over_lanes();
        }
    }
    if (lane == 0) x[list[row]] = to_store<T>(tot);
}

__device__ int find_in_list(const int* list, int n, int key) {
    int lo = 0, hi = n - 1;
    while (lo <= hi) {
        const int mid = (lo + hi) >> 1;
        const int v = list[mid];
        if (v == key) return mid;
        if (v < key) lo = mid + 1;
        else hi = mid - 1;
    }
    return -1;
}

// label propagation (single block); list sorted ascending (natural order)
__global__ void k_components(Grid3 g, const double* __restrict__ A, const int* __restrict__ list, int n,
                             int* __restrict__ label, unsigned char* __restrict__ pinned) {
    __shared__ int changed;
    for (int r = threadIdx.x; r < n; r += blockDim.x) label[r] = r;
    __syncthreads();
    const int X = 1, Y = g.sx, Z = g.sxy, N = g.np;
    for (int it = 0; it < n + 1; ++it) {
        if (threadIdx.x == 0) changed = 0;
        __syncthreads();
        for (int r = threadIdx.x; r < n; r += blockDim.x) {
            const int p = list[r];
            int best = label[r];
            // neighbours across open faces: (face index, neighbour cell)
            const int faces[6] = {p, p + X, N + p, N + p + Y, 2 * N + p, 2 * N + p + Z};
            const int nbr[6] = {p - X, p + X, p - Y, p + Y, p - Z, p + Z};
            for (int f = 0; f < 6; ++f) {
                if (A[faces[f]] > 0.0) {
                    const int pos = find_in_list(list, n, nbr[f]);
                    if (pos >= 0) best = min(best, label[pos]);
                }
            }
            if (best < label[r]) {
                label[r] = best;
                changed = 1;
            }
        }
        __syncthreads();
        if (!changed) break;
        __syncthreads();
    }
    // components with an open face on the outer wall (a magnetic symmetry
    // plane) are regular: the potential beyond the wall is zero.  pinned[]
    // first marks their roots, then takes the final flags.
    for (int r = threadIdx.x; r < n; r += blockDim.x) pinned[r] = 0;
    __syncthreads();
    for (int r = threadIdx.x; r < n; r += blockDim.x) {
        const int p = list[r];
        const int i = (p - g.off0) % g.sx, j = ((p - g.off0) / g.sx) % g.sy, k = (p - g.off0) / g.sxy;
        const bool wall = (i == 0 && A[p] > 0.0) || (i == g.nx - 1 && A[p + X] > 0.0) ||
                          (j == 0 && A[N + p] > 0.0) || (j == g.ny - 1 && A[N + p + Y] > 0.0) ||
                          (k == 0 && A[2 * N + p] > 0.0) || (k == g.nz - 1 && A[2 * N + p + Z] > 0.0);
        if (wall) pinned[label[r]] = 2;   // benign race: every writer stores the same value
    }
    __syncthreads();
    for (int r = threadIdx.x; r < n; r += blockDim.x) {
        const bool root = label[r] == r;
        pinned[r] = (root && pinned[r] != 2) ? 1 : 0;
    }
}

}  // namespace

size_t dense_inverse_work(int n) { return (size_t)n * n + (2 * kPanel + 1) * (size_t)n + 2 * kPanel; }

bool dense_inverse(double* M, int n, double* work, int* d_flag, cudaStream_t s) {
    double* W = work;
    double* Mt = W + (size_t)n * n;
    double* B = Mt + kPanel * (size_t)n;
    int* piv = reinterpret_cast<int*>(B + kPanel * (size_t)n);
    int* src = piv + n;
    int* swaps = src + n;   // 4 kPanel entries
    constexpr int rows = kPanelBlocks * kPanelThreads;   // of one row per thread
    // 6,000 faces at most on the coarsest vector level, and so 12,000 cells (an active
    // cell has an open face, a face two cells): up to six rows a thread
    DM_REQUIRE(n <= kDenseMax && kDenseMax <= 6 * rows, DM_ERR_INVALID_ARG, "dense inverse: more rows than a panel holds");
    DM_CUDA(cudaMemsetAsync(d_flag, 0, sizeof(int), s));
    DM_CUDA(cudaMemcpyAsync(W, M, sizeof(double) * (size_t)n * n, cudaMemcpyDeviceToDevice, s));
    if (n <= rows) gj_eliminate<1>(W, n, piv, Mt, B, swaps, d_flag, s);
    else if (n <= 2 * rows) gj_eliminate<2>(W, n, piv, Mt, B, swaps, d_flag, s);
    else if (n <= 3 * rows) gj_eliminate<3>(W, n, piv, Mt, B, swaps, d_flag, s);
    else gj_eliminate<6>(W, n, piv, Mt, B, swaps, d_flag, s);
    int h = 0;
    DM_CUDA(cudaMemcpyAsync(&h, d_flag, sizeof(int), cudaMemcpyDeviceToHost, s));
    DM_CUDA(cudaStreamSynchronize(s));
    if (h) return false;   // the pivots after the failing one were never written
    launch("k_gj_columns", k_gj_columns, (n + 127) / 128, 128, 0, s, n, (const int*)piv, src);
    launch("k_gj_gather", k_gj_gather, dim3((n + 127) / 128, n), 128, 0, s, (const double*)W, M, n, (const int*)src);
    return true;
}

template <typename T>
void dense_coarse_solve(const double* Minv64, const float* Minv32, int n, const int* list, const unsigned char* zero_rows,
                        const T* f, T* x, cudaStream_t s) {
    using C = typename Compute<T>::type;
    if (n <= 0) return;
    DM_REQUIRE(n <= kDenseMax, DM_ERR_INVALID_ARG, "coarsest solve: too many rows");
    const size_t smem = sizeof(C) * (size_t)n;
    // above the 48 KB a kernel may use unasked; the setting belongs to the current device
    if (smem > 48 * 1024)
        DM_CUDA(cudaFuncSetAttribute(k_coarse_solve<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    launch_chain("k_coarse_solve", (double)n * n * sizeof(C) + 2.0 * n * sizeof(T), k_coarse_solve<T>,
             (n + kSolveWarps - 1) / kSolveWarps, 32 * kSolveWarps, smem, s, n, Minv64, Minv32, list, zero_rows, f, x);
}

void cell_components_pin(const Grid3& g, const double* A, const int* list, int n, int* label, unsigned char* pinned,
                         cudaStream_t s) {
    if (n <= 0) return;
    launch("k_components", k_components, 1, 512, 0, s, g, A, list, n, label, pinned);
}

template void dense_coarse_solve<double>(const double*, const float*, int, const int*, const unsigned char*,
                                         const double*, double*, cudaStream_t);
template void dense_coarse_solve<float>(const double*, const float*, int, const int*, const unsigned char*,
                                        const float*, float*, cudaStream_t);
template void dense_coarse_solve<__nv_bfloat16>(const double*, const float*, int, const int*, const unsigned char*,
                                                const __nv_bfloat16*, __nv_bfloat16*, cudaStream_t);

}  // namespace dm

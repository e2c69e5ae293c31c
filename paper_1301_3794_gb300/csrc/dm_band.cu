// Cut-cell band smoother: a restricted additive Schwarz step on the band faces.
//
// The band holds the open faces next to a cell within one cell of a cut cell
// (0 < V < 1).  It is covered by bricks of b^3 nodes (a face belongs to the
// node at its lower corner).  The subdomain of a brick is every band face whose
// node lies within one node of the brick; the brick owns the faces whose node
// lies inside it.  From r0 = f - (K - sigma A) x, each subdomain runs `sweeps`
// damped Jacobi sweeps d <- d + omega D^-1 (r0 - K_SS d) from d = 0 on its own
// rows (couplings to faces outside the subdomain stay frozen), and x takes d
// on the owned faces.  With one brick covering the grid this is plain
// band-restricted Jacobi.
//
// Bricks of up to 8 nodes (the default is 8) take k_band_node or its FP64 form on
// clusters: one thread per node or row of the subdomain, boxes of a fixed layout.
// Larger and very small bricks (band_nodes_fit, band_nodes_best) take
// k_band_schwarz, one thread per few rows, boxes clipped to the subdomain, one block per
// subdomain.  In both the correction d lives in shared memory on the
// subdomain's local box of nodes (all three components, zero wherever the
// subdomain has no row), so a row's couplings are reached at fixed offsets: the
// 15 slots of band_slot.
#include <cooperative_groups.h>

#include <algorithm>
#include <vector>

#include "dm_common.cuh"

namespace dm {

namespace {

// Couplings of a row in the subdomain's local box: component c at local node
// n (index within one component's box), box strides st = {1, lx, lx ly}, l3
// nodes per component.  The 15 slots of band_slot, in order, are
//   same component:   n, n -/+ 1, n -/+ lx, n -/+ lx ly;
//   component c + k (k = 1, 2), its stride sk = st[(c + k) % 3]:
//     m, m + sk, m + sc, m + sc + sk  with m = n - sc (sc = st[c]) in that component.
struct RowAddr {
    int b0, b1, b2;   // n, and m in components c + 1 and c + 2 (offsets into the box)
    int sc, s1, s2;
};
__device__ __forceinline__ RowAddr row_addr(int p, int l3, int lx, int lxy) {
    RowAddr a;
    const int c = p / l3, n = p - c * l3;
    const int st[3] = {1, lx, lxy};
    const int c1 = c == 2 ? 0 : c + 1, c2 = c == 0 ? 2 : c - 1;
    a.sc = st[c];
    a.s1 = st[c1];
    a.s2 = st[c2];
    a.b0 = p;
    a.b1 = c1 * l3 + n - a.sc;
    a.b2 = c2 * l3 + n - a.sc;
    return a;
}
// `self` is the row's own entry d[a.b0] (kept in a register by the sweeps)
template <typename C>
__device__ __forceinline__ C row_dot(const C* v, C self, const C* d, const RowAddr& a, int lx, int lxy) {
    C acc = v[0] * self;
    acc += v[1] * d[a.b0 - 1] + v[2] * d[a.b0 + 1];
    acc += v[3] * d[a.b0 - lx] + v[4] * d[a.b0 + lx];
    acc += v[5] * d[a.b0 - lxy] + v[6] * d[a.b0 + lxy];
    acc += v[7] * d[a.b1] + v[8] * d[a.b1 + a.s1] + v[9] * d[a.b1 + a.sc] + v[10] * d[a.b1 + a.sc + a.s1];
    acc += v[11] * d[a.b2] + v[12] * d[a.b2 + a.s2] + v[13] * d[a.b2 + a.sc] + v[14] * d[a.b2 + a.sc + a.s2];
    return acc;
}

// R > 0: each thread owns up to R rows (row r = threadIdx.x + k blockDim.x) with
// their coefficients and addresses in registers.  R == 0: any row count; r0
// and omega/D in shared memory and the coefficients re-read on every sweep.
// Block b handles subdomain sub0 + b.
template <typename T, typename TC, int R, int NT>
__global__ void __launch_bounds__(NT)
    k_band_schwarz(int sub0, const int* __restrict__ off, const int* __restrict__ copy, const int* __restrict__ pos,
                   const int* __restrict__ dims, const int* __restrict__ org, const TC* __restrict__ vals, int ncopies,
                   const int* __restrict__ band, const TC* __restrict__ invD, const T* __restrict__ f,
                   const T* __restrict__ x, double* __restrict__ u, typename Compute<T>::type om, int sweeps, Grid3 g,
                   int maxbox, int maxrows) {
    using C = typename Compute<T>::type;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* const buf0 = reinterpret_cast<C*>(smem_raw);
    C* const buf1 = buf0 + maxbox;
    C* s_r0 = buf1 + maxbox;          // R == 0 only
    C* s_w = s_r0 + maxrows;
    const int sd = sub0 + blockIdx.x;
    const int b0 = off[sd];
    const int nr = off[sd + 1] - b0;
    const int dm = dims[sd];
    const int lx = dm & 1023, ly = (dm >> 10) & 1023, lz = dm >> 20;
    const int lxy = lx * ly, l3 = lxy * lz;
    // x over the local box (nodes org + local coordinates; outside the padded
    // grid's -1 .. n+1 it is zero), so that the start residuals read it from
    // shared memory at the rows' slot offsets: one coalesced pass over the box
    // instead of 15 scattered loads per row
    {
        const int ox = org[3 * sd], oy = org[3 * sd + 1], oz = org[3 * sd + 2];
        for (int k = threadIdx.x; k < 3 * l3; k += blockDim.x) {
            const int comp = k / l3, n = k - comp * l3;
            const int lk = n / lxy, rem = n - lk * lxy;
            const int lj = rem / lx, li = rem - lj * lx;
            const int i = ox + li, j = oy + lj, kk = oz + lk;
            const bool in = i >= -1 && j >= -1 && kk >= -1 && i <= g.nx + 1 && j <= g.ny + 1 && kk <= g.nz + 1;
            buf0[k] = C(0);
            buf1[k] = in ? (C)to_c(x[(size_t)comp * g.np + g.idx(i, j, kk)]) : C(0);
        }
    }
    __syncthreads();
    constexpr int RR = R > 0 ? R : 1;
    C v[RR][kBandSlots];
    C r0[RR], w[RR], dself[RR];   // dself: the row's current correction (R > 0)
    RowAddr ad[RR];
    bool cm[RR];
    // residual of the full row at the start values, and the first sweep from d = 0
    auto start_row = [&](int r, C* ve, C& rr, C& ww) {
        const int ct = copy[b0 + r];
        if (ct == kDummyCopy) {   // an empty lane of a warp group: no row, no loads
#pragma unroll
            for (int e = 0; e < kBandSlots; ++e) ve[e] = C(0);
            rr = C(0);
            ww = C(0);
            return;
        }
        const int t = ct >= 0 ? ct : -1 - ct;
        const int q = band[t];
        const int ps = pos[b0 + r];
#pragma unroll
        for (int e = 0; e < kBandSlots; ++e) ve[e] = (C)vals[(size_t)e * ncopies + b0 + r];
        const C acc = row_dot(ve, buf1[ps], buf1, row_addr(ps, l3, lx, lxy), lx, lxy);
        rr = (C)to_c(f[q]) - acc;
        ww = om * (C)invD[q];
        buf0[ps] = ww * rr;
    };
    if constexpr (R > 0) {
#pragma unroll
        for (int k = 0; k < R; ++k) {
            const int r = threadIdx.x + k * blockDim.x;
            cm[k] = false;
            if (r < nr) {
                start_row(r, v[k], r0[k], w[k]);
                dself[k] = w[k] * r0[k];
                const int ps = pos[b0 + r];
                if (ps >= 0) {
                    ad[k] = row_addr(ps, l3, lx, lxy);
                    cm[k] = true;
                }
            }
        }
    } else {
        for (int r = threadIdx.x; r < nr; r += blockDim.x) start_row(r, v[0], s_r0[r], s_w[r]);
    }
    __syncthreads();
    // buf1 becomes the second correction buffer: zero outside the rows
    for (int k = threadIdx.x; k < 3 * l3; k += blockDim.x) buf1[k] = C(0);
    __syncthreads();
    C* dc = buf0;
    C* dn = buf1;
    for (int s = 1; s < sweeps; ++s) {
        if constexpr (R > 0) {
#pragma unroll
            for (int k = 0; k < RR; ++k) {
                const int r = threadIdx.x + k * blockDim.x;
                if (r < nr && cm[k]) {
                    const C acc = row_dot(v[k], dself[k], dc, ad[k], lx, lxy);
                    dself[k] = dself[k] + w[k] * (r0[k] - acc);
                    dn[ad[k].b0] = dself[k];
                }
            }
        } else {
            for (int r = threadIdx.x; r < nr; r += blockDim.x) {
                const int ps = pos[b0 + r];
                if (ps < 0) continue;
                const RowAddr a = row_addr(ps, l3, lx, lxy);
                C ve[kBandSlots];
#pragma unroll
                for (int e = 0; e < kBandSlots; ++e) ve[e] = (C)vals[(size_t)e * ncopies + b0 + r];
                const C self = dc[a.b0];
                dn[a.b0] = self + s_w[r] * (s_r0[r] - row_dot(ve, self, dc, a, lx, lxy));
            }
        }
        __syncthreads();
        C* const tmp = dc;
        dc = dn;
        dn = tmp;
    }
    for (int r = threadIdx.x; r < nr; r += blockDim.x) {
        const int ct = copy[b0 + r];
        if (ct >= 0) u[ct] = (double)dc[pos[b0 + r]];
    }
}

// ---- node kernel -------------------------------------------------------------
// Every thread owns one node: its three faces' rows share the couplings they
// read (24 distinct entries of d for 3 rows, where three separate rows read
// 42), because the shared-memory loads of the sweeps are what bounds the FP32
// kernel once a block fills its SM.  Rows are stored scaled by D^-1, so that a
// sweep is d <- c0 + (1 - omega) d - omega sum_e s_e d_e with the row's own
// slot equal to 1 and not stored: 42 coefficients and 3 constants per node in
// registers, which is what lets a full 10^3-node subdomain run as one block of
// 1024 threads with 64 registers each (no spills).  The x box and the couplings
// arrive in one batch of independent loads: with a plain staging loop (ten
// dependent round trips and 500 index instructions a thread) the FP32 pass took
// 170 us where it now takes 134.
// Measured (CUDA events, classes one after another; a kernel of one thread per
// row before): fine level of a 192^3 ellipsoid, FP32, 24 sweeps 241 -> 134 us a
// pass; its coarser levels 24.5 -> 18.5 us a launch; 128^3 sphere, BF16, fine
// 171 -> 83 us.  The shared-memory loads alone would take 43 us at 192^3; the
// rest is the start of each block and the last wave.
//
// Local layout: the up to 10^3 nodes of a subdomain at li + 11 lj + 121 lk in
// each component.  Column 10 of every row, row 10 of every plane and one plane
// before and after each component hold no node and stay zero, and serve as the
// zero neighbours of both of their sides.
constexpr int kNodeBrick = 8;                    // largest brick of the node kernels
constexpr int kNB = kNodeBrick + 2;              // nodes per axis of a subdomain
constexpr int kNX = kNB + 1, kNXY = kNX * kNX, kNC = kNXY * kNX;   // strides: row, plane, component
constexpr int kN0 = kNXY + kNX + 1;              // position of local node (0, 0, 0) of component 0
constexpr int kNBuf = ((kN0 + 3 * kNC + kNXY + kNX + 1) + 3) & ~3; // entries of one correction buffer
constexpr int kNodeVals = 45;                    // per node: 14 scaled couplings of each face's row, then 3 values of 1 / D
// the x box of the start residual: the subdomain's nodes and one ring
constexpr int kXX = kNB + 2, kXXY = kXX * kXX, kXC = kXXY * kXX;

// info word of a node copy: local position (12 bits), faces present (bits 12..14), owned (bit 15)
__host__ __device__ inline int node_info(int pos, int mask, bool owned) { return pos | (mask << 12) | (owned ? 1 << 15 : 0); }

// The 24 neighbours of a node's three faces at q (component blocks of C3
// entries, strides 1, Y, Z) against the 42 couplings v (14 per row, slots 1..14
// of band_slot): ax, ay, az += sum.
template <typename C, int Y, int Z, int C3, typename Ptr>
__device__ __forceinline__ void node_dot(const C* v, Ptr q, C xs, C ys, C zs, C& ax, C& ay, C& az) {
    constexpr int X = 1;
    C t;
    // x faces
    t = q[-X]; ax += v[0] * t;
    t = q[X]; ax += v[1] * t; ay += v[14 + 13] * t; az += v[28 + 9] * t;
    t = q[-Y]; ax += v[2] * t; ay += v[14 + 10] * t;
    t = q[Y]; ax += v[3] * t;
    t = q[-Z]; ax += v[4] * t; az += v[28 + 6] * t;
    t = q[Z]; ax += v[5] * t;
    t = q[X - Y]; ay += v[14 + 11] * t;
    t = q[X - Z]; az += v[28 + 7] * t;
    ay += v[14 + 12] * xs; az += v[28 + 8] * xs;
    // y faces
    t = q[C3 - X]; ay += v[14 + 0] * t; ax += v[6] * t;
    t = q[C3 + X]; ay += v[14 + 1] * t;
    t = q[C3 - Y]; ay += v[14 + 2] * t;
    t = q[C3 + Y]; ay += v[14 + 3] * t; ax += v[9] * t; az += v[28 + 13] * t;
    t = q[C3 - Z]; ay += v[14 + 4] * t; az += v[28 + 10] * t;
    t = q[C3 + Z]; ay += v[14 + 5] * t;
    t = q[C3 + Y - X]; ax += v[7] * t;
    t = q[C3 + Y - Z]; az += v[28 + 11] * t;
    ax += v[8] * ys; az += v[28 + 12] * ys;
    // z faces
    t = q[2 * C3 - X]; az += v[28 + 0] * t; ax += v[10] * t;
    t = q[2 * C3 + X]; az += v[28 + 1] * t;
    t = q[2 * C3 - Y]; az += v[28 + 2] * t; ay += v[14 + 6] * t;
    t = q[2 * C3 + Y]; az += v[28 + 3] * t;
    t = q[2 * C3 - Z]; az += v[28 + 4] * t;
    t = q[2 * C3 + Z]; az += v[28 + 5] * t; ax += v[13] * t; ay += v[14 + 9] * t;
    t = q[2 * C3 + Z - X]; ax += v[11] * t;
    t = q[2 * C3 + Z - Y]; ay += v[14 + 7] * t;
    ax += v[12] * zs; ay += v[14 + 8] * zs;
}

template <typename T, typename TC>
struct NodeArgs {
    const int* off;      // first copy of each subdomain
    const int* node;     // padded node of each copy (-1: empty lane)
    const int* info;
    const int* org;      // node coordinates of each subdomain's local node (0, 0, 0)
    const TC* vals;      // [kNodeVals][ncopies]
    int ncopies;
    const T* f;
    const T* x;
    typename Compute<T>::type* u;   // [3][ncopies], the owned nodes' corrections
    typename Compute<T>::type om;
    int sweeps;
    Grid3 g;
};

// 4-byte asynchronous copy into shared memory (zero when !in): no register
// holds the value, so a thread's twelve copies and its node's couplings are all
// in flight at once
__device__ __forceinline__ void copy4_async(void* dst, const void* src, bool in) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    const int n = in ? 4 : 0;
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void copy_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// One block per subdomain, one thread per node (FP32 arithmetic).
template <typename T, typename TC, int NT>
__global__ void __launch_bounds__(NT, 1024 / NT) k_band_node(int sub0, NodeArgs<T, TC> a) {
    using C = typename Compute<T>::type;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* const buf = reinterpret_cast<C*>(smem_raw);
    const int sd = sub0 + blockIdx.x;
    const int b0 = a.off[sd];
    const bool has = (int)threadIdx.x < a.off[sd + 1] - b0;
    const int ct = b0 + threadIdx.x;
    const int p = has ? a.node[ct] : -1;
    const int info = p >= 0 ? a.info[ct] : 0;
    const bool live = p >= 0;
    // the couplings and the zeroed buffers need nothing from the kernels before
    C v[42], cx = C(0), cy = C(0), cz = C(0), dx = C(0), dy = C(0), dz = C(0), fx = C(0), fy = C(0), fz = C(0);
#pragma unroll
    for (int e = 0; e < 42; ++e) v[e] = live ? (C)a.vals[(size_t)e * a.ncopies + ct] : C(0);
    if (live) {
        dx = (C)a.vals[(size_t)42 * a.ncopies + ct];   // 1 / D, 0 on faces without a row
        dy = (C)a.vals[(size_t)43 * a.ncopies + ct];
        dz = (C)a.vals[(size_t)44 * a.ncopies + ct];
    }
    for (int k = threadIdx.x; k < 2 * kNBuf / 4; k += NT) reinterpret_cast<float4*>(buf)[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    chain_wait();
    // x over the local box (zero outside the padded grid's -1 .. n+1): every
    // thread copies whole columns along z, twelve independent loads each
    {
        C* const xb = buf + 2 * kNBuf;
        const int ox = a.org[3 * sd] - 1, oy = a.org[3 * sd + 1] - 1, oz = a.org[3 * sd + 2] - 1;
        for (int col = threadIdx.x; col < 3 * kXXY; col += NT) {
            const int c = col / kXXY, r = col - c * kXXY, lj = r / kXX, li = r - lj * kXX;
            const int i = ox + li, j = oy + lj;
            const bool inxy = i >= -1 && j >= -1 && i <= a.g.nx + 1 && j <= a.g.ny + 1;
            const T* src = a.x + (inxy ? (size_t)c * a.g.np + a.g.idx(i, j, 0) : 0);
            C* dst = xb + c * kXC + r;
            if constexpr (std::is_same<T, float>::value) {
#pragma unroll
                for (int lk = 0; lk < kXX; ++lk) {
                    const bool in = inxy && oz + lk >= -1 && oz + lk <= a.g.nz + 1;
                    copy4_async(dst + lk * kXXY, in ? src + (oz + lk) * a.g.sxy : a.x, in);
                }
            } else {
                C tmp[kXX];
#pragma unroll
                for (int lk = 0; lk < kXX; ++lk) {
                    const bool in = inxy && oz + lk >= -1 && oz + lk <= a.g.nz + 1;
                    tmp[lk] = in ? (C)to_c(src[(oz + lk) * a.g.sxy]) : C(0);
                }
#pragma unroll
                for (int lk = 0; lk < kXX; ++lk) dst[lk * kXXY] = tmp[lk];
            }
        }
    }
    if (live) {
        fx = (C)to_c(a.f[p]);
        fy = (C)to_c(a.f[a.g.np + p]);
        fz = (C)to_c(a.f[2 * a.g.np + p]);
    }
    const int pos = info & 4095;   // li + 11 lj + 121 lk
    if constexpr (std::is_same<T, float>::value) copy_async_wait();
    __syncthreads();
    if (live) {
        const int lk = pos / kNXY, lj = (pos / kNX) % kNX, li = pos % kNX;
        const C* q = buf + 2 * kNBuf + (lk + 1) * kXXY + (lj + 1) * kXX + li + 1;
        const C xs = q[0], ys = q[kXC], zs = q[2 * kXC];
        cx = xs; cy = ys; cz = zs;
        node_dot<C, kXX, kXXY, kXC>(v, q, xs, ys, zs, cx, cy, cz);
        cx = dx != C(0) ? a.om * (dx * fx - cx) : C(0);
        cy = dy != C(0) ? a.om * (dy * fy - cy) : C(0);
        cz = dz != C(0) ? a.om * (dz * fz - cz) : C(0);
    }
#pragma unroll
    for (int e = 0; e < 42; ++e) v[e] *= -a.om;
    C* const mine = buf + kN0 + pos;
    const C keep = C(1) - a.om;
    C ex = cx, ey = cy, ez = cz;   // the node's correction
    if (live) {
        mine[0] = ex;
        mine[kNC] = ey;
        mine[2 * kNC] = ez;
    }
    __syncthreads();
    int cur = 0;
    for (int s = 1; s < a.sweeps; ++s) {
        if (live) {
            const C* q = mine + cur;
            C ax = fma(keep, ex, cx), ay = fma(keep, ey, cy), az = fma(keep, ez, cz);
            node_dot<C, kNX, kNXY, kNC>(v, q, ex, ey, ez, ax, ay, az);
            ex = ax; ey = ay; ez = az;
            C* w = mine + (kNBuf - cur);
            w[0] = ex;
            w[kNC] = ey;
            w[2 * kNC] = ez;
        }
        cur = kNBuf - cur;
        __syncthreads();
    }
    if ((info >> 15) & 1) {
        a.u[ct] = ex;
        a.u[(size_t)a.ncopies + ct] = ey;
        a.u[2 * (size_t)a.ncopies + ct] = ez;
    }
}

// One row (face component c) of node_dot: sum over the 14 couplings w of the row
// (component block strides as there)
template <typename C, int c, typename Ptr>
__device__ __forceinline__ C row_dot_at(const C* w, Ptr q, int Y, int Z, int C3, C acc) {
    constexpr int c1 = (c + 1) % 3, c2 = (c + 2) % 3;
    const int st[3] = {1, Y, Z};
    const int m1 = (c1 - c) * C3, m2 = (c2 - c) * C3, sc = st[c], s1 = st[c1], s2 = st[c2];
    const int o[14] = {-1, 1, -Y, Y, -Z, Z, m1 - sc, m1 - sc + s1, m1, m1 + s1, m2 - sc, m2 - sc + s2, m2, m2 + s2};
#pragma unroll
    for (int e = 0; e < 14; ++e) acc += w[e] * (C)to_c(q[o[e]]);
    return acc;
}

// FP64: a cluster of CS blocks per subdomain.  The FP64 pipe issues two FMAs
// per clock and SM, so a subdomain's 45 FMAs per node and sweep are what its
// time goes on; the cluster spreads them over CS SMs.  One thread per row, not
// per node: a warp's FMA occupies its scheduler's FP64 unit for 64 clocks, so on
// small grids, where an SM holds few nodes, the length of a thread's chain is the
// sweep's time (45 FMAs 1.5 us, 15 FMAs 0.5); the rows of one component share a
// warp, and the three warps of the same nodes sit on three schedulers.  Every
// block keeps the whole correction box; a row's new value goes to the blocks
// whose rows read it (positions within one plane, row and column) through
// distributed shared memory, and a cluster barrier closes each sweep.
// Measured, one pass (one block per subdomain before): 16^3 sphere (27
// subdomains) 190 -> 42 us (63 with one thread per node); 72 x 56 x 88 ellipsoid
// fine level 326 -> 277 us with the classes one after another.
constexpr int kClusterNodes = 128, kClusterThreads = 3 * kClusterNodes;
template <typename T, typename TC, int CS>
__global__ void __cluster_dims__(CS, 1, 1) __launch_bounds__(kClusterThreads) k_band_node_cluster(int sub0, NodeArgs<T, TC> a) {
    using C = typename Compute<T>::type;
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* const buf = reinterpret_cast<C*>(smem_raw);
    constexpr int NT = kClusterThreads;
    const int rank = (int)cluster.block_rank();
    const int sd = sub0 + blockIdx.x / CS;
    const int b0 = a.off[sd], n = a.off[sd + 1] - b0;
    const int per = (n + CS - 1) / CS;               // nodes of each block, in box order
    const int warp = threadIdx.x >> 5, comp = warp % 3;
    const int inblock = (warp / 3) * 32 + (threadIdx.x & 31), local = rank * per + inblock;
    const int ct = b0 + local;
    const bool node = inblock < per && local < n;
    const int info = node ? a.info[ct] : 0;
    const bool live = (info >> (12 + comp)) & 1;     // the node has this row
    const int p = live ? a.node[ct] + comp * a.g.np : 0;
    const int pos = info & 4095;
    // the blocks that hold a neighbour of this row
    int r0 = CS, r1 = -1;
    if (live) {
#pragma unroll
        for (int r = 0; r < CS; ++r) {
            const int lo = r * per, hi = min(n, lo + per) - 1;
            if (lo <= hi && (a.info[b0 + lo] & 4095) <= pos + kN0 && (a.info[b0 + hi] & 4095) >= pos - kN0) {
                r0 = min(r0, r);
                r1 = max(r1, r);
            }
        }
    }
    C w[14], rd = C(0);
#pragma unroll
    for (int e = 0; e < 14; ++e) w[e] = live ? (C)a.vals[(size_t)(14 * comp + e) * a.ncopies + ct] : C(0);
    if (live) rd = (C)a.vals[(size_t)(42 + comp) * a.ncopies + ct];
    for (int k = threadIdx.x; k < 2 * kNBuf; k += NT) buf[k] = C(0);
    chain_wait();
    C c0 = C(0);
    if (live) {
        // start residual from global memory: the neighbours' loads are independent of one another
        const T* q = a.x + p;
        const C xs = (C)to_c(q[0]);
        const int Y = a.g.sx, Z = a.g.sxy, N = a.g.np;
        const C kx = comp == 0 ? row_dot_at<C, 0>(w, q, Y, Z, N, xs)
                               : (comp == 1 ? row_dot_at<C, 1>(w, q, Y, Z, N, xs) : row_dot_at<C, 2>(w, q, Y, Z, N, xs));
        c0 = a.om * (rd * (C)to_c(a.f[p]) - kx);
    }
#pragma unroll
    for (int e = 0; e < 14; ++e) w[e] *= -a.om;
    cluster.sync();   // every block's buffers are zero
    const C keep = C(1) - a.om;
    const int at = kN0 + comp * kNC + pos;
    C d = c0;
    int cur = 0;      // offset of the buffer the sweep reads
    for (int r = r0; r <= r1; ++r) cluster.map_shared_rank(buf, r)[at] = d;
    for (int s = 1; s < a.sweeps; ++s) {
        cluster.sync();
        if (live) {
            const C* q = buf + at + cur;
            const C acc = fma(keep, d, c0);
            d = comp == 0 ? row_dot_at<C, 0>(w, q, kNX, kNXY, kNC, acc)
                          : (comp == 1 ? row_dot_at<C, 1>(w, q, kNX, kNXY, kNC, acc)
                                       : row_dot_at<C, 2>(w, q, kNX, kNXY, kNC, acc));
            if (s + 1 < a.sweeps)
                for (int r = r0; r <= r1; ++r) cluster.map_shared_rank(buf, r)[at + (kNBuf - cur)] = d;
        }
        cur = kNBuf - cur;
    }
    if (live && ((info >> 15) & 1)) a.u[(size_t)comp * a.ncopies + ct] = d;
    cluster.sync();   // no block leaves while another may still write to it
}

// x <- x + u on the band faces (uidx: where each face's owner put its correction)
template <typename T>
__global__ void k_band_add_node(const int* __restrict__ band, const int* __restrict__ uidx, int nband,
                                const typename Compute<T>::type* u, T* x) {
    using C = typename Compute<T>::type;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int q = t < nband ? band[t] : 0, at = t < nband ? uidx[t] : 0;
    chain_wait();
    if (t < nband) x[q] = to_store<T>((C)to_c(x[q]) + u[at]);
}

// Scaled couplings of every node copy from the band rows (15 slots, slot-major)
// and, for the owners, where each face's correction will be.  tmap: position of
// a face in the band list, -1 off the band.
template <typename TC>
__global__ void k_band_node_vals(int ncopies, const int* __restrict__ node, const int* __restrict__ info, int np,
                                 const int* __restrict__ tmap, const double* __restrict__ rows, int nband,
                                 const double* __restrict__ invD, TC* __restrict__ vals, int* __restrict__ uidx) {
    const int ct = blockIdx.x * blockDim.x + threadIdx.x;
    if (ct >= ncopies) return;
    const int p = node[ct];
    const int in = p >= 0 ? info[ct] : 0;
    for (int c = 0; c < 3; ++c) {
        const bool row = (in >> (12 + c)) & 1;
        const int t = row ? tmap[c * np + p] : 0;
        const double d = row ? invD[c * np + p] : 0.0;
        for (int e = 1; e < kBandSlots; ++e)
            vals[(size_t)(14 * c + e - 1) * ncopies + ct] = row ? (TC)(d * rows[(size_t)e * nband + t]) : TC(0);
        vals[(size_t)(42 + c) * ncopies + ct] = (TC)d;
        if (row && ((in >> 15) & 1)) uidx[t] = c * ncopies + ct;
    }
}

template <typename T>
__global__ void k_band_add(const int* __restrict__ band, int nband, const double* __restrict__ u,
                           T* __restrict__ x) {
    using C = typename Compute<T>::type;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nband) return;
    const int q = band[t];
    x[q] = to_store<T>((C)to_c(x[q]) + (C)u[t]);
}

__global__ void k_band_copy_vals(const int* __restrict__ copy, int ncopies, const double* __restrict__ band_vals,
                                 int nband, double* __restrict__ out) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= ncopies) return;
    const int ct = copy[c];
    if (ct == kDummyCopy) {
        for (int e = 0; e < kBandSlots; ++e) out[(size_t)e * ncopies + c] = 0.0;
        return;
    }
    const int t = ct >= 0 ? ct : -1 - ct;
    for (int e = 0; e < kBandSlots; ++e) out[(size_t)e * ncopies + c] = band_vals[(size_t)e * nband + t];
}

template <typename T>
size_t schwarz_smem(int maxbox, int maxrows, int R) {
    using C = typename Compute<T>::type;
    return sizeof(C) * (2 * (size_t)maxbox + (R == 0 ? 2 * (size_t)maxrows : 0));
}

}  // namespace

// k_band_schwarz: levels with at most this many subdomains are smoothed in a single launch
constexpr int kSingleLaunchSubdomains = 304;

// Size classes of its subdomains (rows): each class is launched with its own
// block size and rows per thread (class_shape), so that small subdomains are not held
// to the register and thread budget of the largest.
int schwarz_class(int rows) {
    return rows <= 256 ? 0 : (rows <= 512 ? 1 : (rows <= 1024 ? 2 : (rows <= 2048 ? 3 : 4)));
}

// (Counting sorts throughout: with comparison sorts of the copies an operator with bricks of
// 2 nodes on 128^3 took 157 ms to make, now 68; 51 with the node kernels' layout.)
void band_schwarz_setup(const Grid3& g, const int* band_dev, int nband, int brick, SchwarzLayout& out,
                        cudaStream_t s) {
    DM_REQUIRE(brick >= 1, DM_ERR_INVALID_ARG, "band brick must be >= 1 node");
    out = SchwarzLayout{};
    if (nband <= 0) return;
    std::vector<int> band(nband);
    DM_CUDA(cudaMemcpyAsync(band.data(), band_dev, sizeof(int) * nband, cudaMemcpyDeviceToHost, s));
    DM_CUDA(cudaStreamSynchronize(s));

    // node (i, j, k) and component of every band face: q = c np + off0 + i + sx (j + sy k)
    const int n[3] = {g.nx, g.ny, g.nz};
    const int nb[3] = {(g.nx + brick) / brick, (g.ny + brick) / brick, (g.nz + brick) / brick};
    const size_t nbk = (size_t)nb[0] * nb[1] * nb[2];
    struct Face {
        int node[3];
        int comp;
    };
    std::vector<Face> face(nband);
    std::vector<char> owner(nbk, 0);
    auto key = [&](int bx, int by, int bz) { return ((size_t)bz * nb[1] + by) * nb[0] + bx; };
    for (int t = 0; t < nband; ++t) {
        const int comp = band[t] / g.np, r = band[t] - comp * g.np - g.off0;
        const int k = r / g.sxy, rem = r - k * g.sxy;
        const int j = rem / g.sx, i = rem - j * g.sx;
        face[t] = Face{{i, j, k}, comp};
        owner[key(i / brick, j / brick, k / brick)] = 1;
    }
    // copies (brick, face), grouped by brick with a counting sort: brick B holds node P when
    // B b - 1 <= P <= B b + b on every axis, i.e. ceil(P / b) - 1 <= B <= floor((P + 1) / b);
    // t for the owner's copy, -1 - t for another's
    auto each_copy = [&](auto&& visit) {
        for (int t = 0; t < nband; ++t) {
            int lo[3], hi[3], own[3];
            for (int a = 0; a < 3; ++a) {
                const int P = face[t].node[a];
                own[a] = P / brick;
                lo[a] = std::max((P + brick - 1) / brick - 1, 0);
                hi[a] = std::min((P + 1) / brick, nb[a] - 1);
            }
            for (int bz = lo[2]; bz <= hi[2]; ++bz)
                for (int by = lo[1]; by <= hi[1]; ++by)
                    for (int bx = lo[0]; bx <= hi[0]; ++bx) {
                        const size_t kb = key(bx, by, bz);
                        if (owner[kb]) visit(kb, bx == own[0] && by == own[1] && bz == own[2] ? t : -1 - t);
                    }
        }
    };
    std::vector<int> start(nbk + 1, 0);
    each_copy([&](size_t kb, int) { ++start[kb + 1]; });
    for (size_t b = 0; b < nbk; ++b) start[b + 1] += start[b];
    const int nc = start[nbk];
    std::vector<int> cp(nc);
    {
        std::vector<int> fill(start.begin(), start.end() - 1);
        each_copy([&](size_t kb, int ct) { cp[fill[kb]++] = ct; });
    }
    // subdomains class by class; slots of one: its rows per component rounded up to whole warp groups
    struct Run {
        size_t brick;
        int rows[3], slots;
    };
    std::vector<Run> runs;
    for (size_t b = 0; b < nbk; ++b) {
        if (start[b + 1] == start[b]) continue;
        Run r{b, {0, 0, 0}, 0};
        for (int c = start[b]; c < start[b + 1]; ++c) ++r.rows[face[cp[c] >= 0 ? cp[c] : -1 - cp[c]].comp];
        for (int e : r.rows) r.slots += 32 * ((e + 31) / 32);
        runs.push_back(r);
    }
    std::stable_sort(runs.begin(), runs.end(),
                     [&](const Run& x, const Run& y) { return schwarz_class(x.slots) < schwarz_class(y.slots); });
    for (int k = 0; k < kSchwarzClasses; ++k) {
        out.cls_first[k] = out.cls_count[k] = 0;
        out.cls_copies[k] = out.cls_owned[k] = 0;
    }
    out.copy.reserve((size_t)nc + 96 * runs.size());
    out.pos.reserve((size_t)nc + 96 * runs.size());
    std::vector<int> at;   // box position of each copy of a run
    for (size_t rI = 0; rI < runs.size(); ++rI) {
        const size_t kb = runs[rI].brick;
        const int c0 = start[kb], c1 = start[kb + 1];
        const int cl = schwarz_class(runs[rI].slots);
        if (out.cls_count[cl] == 0) out.cls_first[cl] = (int)rI;
        ++out.cls_count[cl];
        const int B[3] = {(int)(kb % nb[0]), (int)((kb / nb[0]) % nb[1]), (int)(kb / ((size_t)nb[0] * nb[1]))};
        // local box: the subdomain's nodes and their neighbours (within the padded grid)
        int lo[3], l[3];
        for (int a = 0; a < 3; ++a) {
            lo[a] = std::max(B[a] * brick - 2, -1);
            const int hi = std::min(B[a] * brick + brick + 1, n[a] + 1);
            l[a] = hi - lo[a] + 1;
        }
        DM_REQUIRE(l[0] < 1024 && l[1] < 1024 && l[2] < 1024, DM_ERR_INVALID_ARG, "band brick too large");
        out.off.push_back((int)out.copy.size());
        out.dims.push_back(l[0] | (l[1] << 10) | (l[2] << 20));
        out.org.insert(out.org.end(), {lo[0], lo[1], lo[2]});
        out.maxbox = std::max(out.maxbox, 3 * l[0] * l[1] * l[2]);
        out.cls_copies[cl] += c1 - c0;
        // Rows are laid out in warp groups of 32 slots.  Per component, the rows
        // are sorted by their shared-memory bank (box position mod 32) and dealt
        // round-robin over the component's ceil(n / 32) groups, so the lanes of
        // a warp mostly sit in distinct banks; every slot offset is the same for
        // the rows of one component, so each of the 15 loads of a sweep is then
        // (nearly) free of bank conflicts.  Unfilled slots are empty lanes.
        at.resize(c1 - c0);
        int cnt[3][33] = {};
        for (int c = c0; c < c1; ++c) {
            const Face& f = face[cp[c] >= 0 ? cp[c] : -1 - cp[c]];
            if (cp[c] >= 0) ++out.cls_owned[cl];
            const int p = ((f.comp * l[2] + f.node[2] - lo[2]) * l[1] + f.node[1] - lo[1]) * l[0] + f.node[0] - lo[0];
            at[c - c0] = p;
            ++cnt[f.comp][(p & 31) + 1];
        }
        int ng[3];
        size_t base[3], end = out.copy.size();
        for (int comp = 0; comp < 3; ++comp) {
            for (int k = 0; k < 32; ++k) cnt[comp][k + 1] += cnt[comp][k];
            ng[comp] = (runs[rI].rows[comp] + 31) / 32;
            base[comp] = end;
            end += 32 * (size_t)ng[comp];
        }
        out.copy.resize(end, kDummyCopy);
        out.pos.resize(end, -1);
        for (int c = c0; c < c1; ++c) {
            const int comp = face[cp[c] >= 0 ? cp[c] : -1 - cp[c]].comp, p = at[c - c0];
            const int rk = cnt[comp][p & 31]++;
            const size_t slot = base[comp] + (size_t)(rk % ng[comp]) * 32 + rk / ng[comp];
            out.pos[slot] = p;
            out.copy[slot] = cp[c];
        }
        out.maxrows = std::max(out.maxrows, (int)out.copy.size() - out.off.back());
    }
    out.off.push_back((int)out.copy.size());
}

void band_copy_vals(const int* copy, int ncopies, const double* band_vals, int nband, double* out, cudaStream_t s) {
    if (ncopies <= 0) return;
    launch("k_band_copy_vals", k_band_copy_vals, (ncopies + 255) / 256, 256, 0, s, copy, ncopies, band_vals, nband,
           out);
}

// ---- node kernels: layout and launches ----------------------------------------

constexpr int kSMs = 152;

// Small bricks stay with k_band_schwarz: the node kernels' local layout and x box
// are those of 8-node bricks, whose clearing and copying outweighs the sweeps of a
// subdomain of a few nodes, and a warp of nodes is three warps of rows.
// Measured, a V-cycle by rows against one by nodes (96^3 / 128^3 ellipsoid, 48 x 48 x 576
// nine-cell cavity): FP32 bricks of 2 nodes 1.11 / 1.68 / 2.20 ms against 1.20 / 1.89 / 2.40,
// of 3 nodes 0.94 / 1.38 / 1.64 against 0.95 / 1.35 / 1.56; BF16 of 3 nodes 0.94 / 1.38 / 1.65
// against 0.99 / 1.50 / 1.79, of 4 nodes 0.93 / 1.36 / 1.52 against 0.89 / 1.28 / 1.41; FP64 of
// 3 nodes 3.7 / 6.0 / 8.8 against 4.5 / 7.5 / 11.4, of 6 nodes 2.8 / 4.6 / 5.8 against 2.6 / 4.2 / 5.4.
bool band_nodes_fit(int brick, int prec) { return brick > (prec == DM_PREC_F32 ? 2 : 3) && brick <= kNodeBrick; }

void band_nodes_setup(const Grid3& g, const int* band_dev, int nband, int brick, bool by_bank, NodeLayout& out,
                      cudaStream_t s) {
    out = NodeLayout{};
    if (nband <= 0) return;
    std::vector<int> band(nband);
    DM_CUDA(cudaMemcpyAsync(band.data(), band_dev, sizeof(int) * nband, cudaMemcpyDeviceToHost, s));
    DM_CUDA(cudaStreamSynchronize(s));
    // the band's nodes in ascending order, with the faces each carries
    std::vector<unsigned char> mask(g.np, 0);
    for (int q : band) mask[q % g.np] |= (unsigned char)(1 << (q / g.np));
    std::vector<int> nodes;
    nodes.reserve(nband / 2 + 1);
    for (int p = 0; p < g.np; ++p)
        if (mask[p]) nodes.push_back(p);
    const int nb[3] = {(g.nx + brick) / brick, (g.ny + brick) / brick, (g.nz + brick) / brick};
    const size_t nbk = (size_t)nb[0] * nb[1] * nb[2];
    auto coords = [&](int p, int c[3]) {
        const int r = p - g.off0;
        c[2] = r / g.sxy;
        const int rem = r - c[2] * g.sxy;
        c[1] = rem / g.sx;
        c[0] = rem - c[1] * g.sx;
    };
    std::vector<unsigned char> owner(nbk, 0);
    auto key = [&](int bx, int by, int bz) { return ((size_t)bz * nb[1] + by) * nb[0] + bx; };
    for (int p : nodes) {
        int c[3];
        coords(p, c);
        owner[key(c[0] / brick, c[1] / brick, c[2] / brick)] = 1;
    }
    // brick B holds node P when B b - 1 <= P <= B b + b on every axis
    auto each = [&](auto&& visit) {
        for (int p : nodes) {
            int c[3], lo[3], hi[3];
            coords(p, c);
            for (int ax = 0; ax < 3; ++ax) {
                lo[ax] = std::max((c[ax] + brick - 1) / brick - 1, 0);
                hi[ax] = std::min((c[ax] + 1) / brick, nb[ax] - 1);
            }
            for (int bz = lo[2]; bz <= hi[2]; ++bz)
                for (int by = lo[1]; by <= hi[1]; ++by)
                    for (int bx = lo[0]; bx <= hi[0]; ++bx) {
                        const size_t kb = key(bx, by, bz);
                        if (owner[kb]) visit(kb, p, c, bx, by, bz);
                    }
        }
    };
    std::vector<int> start(nbk + 1, 0);
    each([&](size_t kb, int, const int*, int, int, int) { ++start[kb + 1]; });
    for (size_t b = 0; b < nbk; ++b) start[b + 1] += start[b];
    std::vector<int> cnode((size_t)start[nbk]), cinfo((size_t)start[nbk]);
    {
        std::vector<int> fill(start.begin(), start.end() - 1);
        // nodes come in ascending order, so every brick's copies are in box order
        each([&](size_t kb, int p, const int* c, int bx, int by, int bz) {
            const int li = c[0] - (bx * brick - 1), lj = c[1] - (by * brick - 1), lk = c[2] - (bz * brick - 1);
            const bool owned = c[0] / brick == bx && c[1] / brick == by && c[2] / brick == bz;
            const int at = fill[kb]++;
            cnode[at] = p;
            cinfo[at] = node_info(li + kNX * lj + kNXY * lk, mask[p], owned);
        });
    }
    // subdomains class by class, the largest class first (its blocks take an SM each)
    std::vector<size_t> order;
    for (size_t b = 0; b < nbk; ++b)
        if (start[b + 1] > start[b]) order.push_back(b);
    std::stable_sort(order.begin(), order.end(), [&](size_t x, size_t y) {
        return node_class(start[x + 1] - start[x]) > node_class(start[y + 1] - start[y]);
    });
    std::vector<int> slot;
    for (size_t b : order) {
        const int c0 = start[b], n = start[b + 1] - c0;
        const int cl = node_class(n);
        if (out.cls_count[cl] == 0) out.cls_first[cl] = (int)out.off.size();
        ++out.cls_count[cl];
        out.off.push_back((int)out.node.size());
        const int bx = (int)(b % nb[0]), by = (int)((b / nb[0]) % nb[1]), bz = (int)(b / ((size_t)nb[0] * nb[1]));
        out.org.insert(out.org.end(), {bx * brick - 1, by * brick - 1, bz * brick - 1});
        out.cls_copies[cl] += n;
        slot.resize(n);
        if (by_bank) {
            // Lanes of a warp in distinct shared-memory banks: the nodes sorted by
            // bank and dealt round-robin over the warps (every coupling sits at one
            // offset for all nodes).  A bank with more nodes than the subdomain has
            // warps still conflicts: 38% of the sweeps' load wavefronts on a 128^3
            // ellipsoid's fine level, 39 to 47% on the next, where box order takes two
            // to three passes for each load.
            const int ng = (n + 31) / 32;
            int cnt[33] = {};
            for (int i = 0; i < n; ++i) ++cnt[((cinfo[c0 + i] & 4095) & 31) + 1];
            for (int k = 0; k < 32; ++k) cnt[k + 1] += cnt[k];
            const size_t base = out.node.size();
            out.node.resize(base + 32 * (size_t)ng, -1);
            out.info.resize(base + 32 * (size_t)ng, 0);
            for (int i = 0; i < n; ++i) {
                const int rk = cnt[(cinfo[c0 + i] & 4095) & 31]++;
                const size_t at = base + (size_t)(rk % ng) * 32 + rk / ng;
                out.node[at] = cnode[c0 + i];
                out.info[at] = cinfo[c0 + i];
            }
        } else {
            out.node.insert(out.node.end(), cnode.begin() + c0, cnode.begin() + c0 + n);
            out.info.insert(out.info.end(), cinfo.begin() + c0, cinfo.begin() + c0 + n);
        }
    }
    out.off.push_back((int)out.node.size());
}

template <typename TC>
void band_node_vals(const int* node, const int* info, int ncopies, const Grid3& g, const int* tmap, const double* rows,
                    int nband, const double* invD, TC* vals, int* uidx, cudaStream_t s) {
    if (ncopies <= 0) return;
    launch("k_band_node_vals", k_band_node_vals<TC>, (ncopies + 127) / 128, 128, 0, s, ncopies, node, info, g.np, tmap,
           rows, nband, invD, vals, uidx);
}

namespace {


// A level with few subdomains goes in one launch shaped for its largest class:
// FP32, when they fit the SMs at one block each; FP64, when clusters of eight
// blocks for every subdomain still run at once.
bool one_launch(int nsub, bool wide) { return wide ? 8 * nsub <= 2 * kSMs : nsub <= kSMs; }

template <typename T, typename TC, int NT>
void launch_node(const char* name, double bytes, int first, int count, const NodeArgs<T, TC>& a, bool chain,
                 cudaStream_t s) {
    using C = typename Compute<T>::type;
    constexpr size_t smem = sizeof(C) * (2 * kNBuf + 3 * kXC);
    // above the 48 KB a kernel may use unasked; set on every call because the setting belongs to the current device
    DM_CUDA(cudaFuncSetAttribute(k_band_node<T, TC, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    if (chain) launch_chain(name, bytes, k_band_node<T, TC, NT>, count, NT, smem, s, first, a);
    else launch_b(name, bytes, k_band_node<T, TC, NT>, count, NT, smem, s, first, a);
}
template <int CS>
void launch_cluster(const char* name, double bytes, int first, int count, const NodeArgs<double, double>& a,
                    bool chain, cudaStream_t s) {
    constexpr size_t smem = sizeof(double) * 2 * kNBuf;
    // above the 48 KB a kernel may use unasked; set on every call because the setting belongs to the current device
    DM_CUDA(cudaFuncSetAttribute(k_band_node_cluster<double, double, CS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem));
    const auto kern = k_band_node_cluster<double, double, CS>;
    if (chain) launch_chain(name, bytes, kern, count * CS, kClusterThreads, smem, s, first, a);
    else launch_b(name, bytes, kern, count * CS, kClusterThreads, smem, s, first, a);
}

}  // namespace

// FP64 bricks of 4 and 5 nodes: by node while there is an SM for every subdomain, because a
// sweep then takes as long as a thread's chain (16^3 sphere, about a hundred
// subdomains of 4-node bricks: 0.22 ms a cycle against 0.29 by rows); with more of them the FP64 pipes are busy either way
// (4 nodes, 32^3 / 96^3 / nine-cell: 1.21 / 3.42 / 7.61 ms by node, 1.09 / 3.05 / 6.68 by rows;
// 5 nodes 1.18 / 2.97 / 6.03 and 1.15 / 2.88 / 6.37).
bool band_nodes_best(int brick, int prec, int nsub) { return prec != DM_PREC_F64 || brick >= 6 || nsub <= kSMs; }

bool band_nodes_fork(int nsub, const int cls_count[kNodeClasses], bool wide) {
    int nl = 0;
    for (int cl = 0; cl < kNodeClasses; ++cl) nl += cls_count[cl] > 0;
    return nl > 1 && !one_launch(nsub, wide);
}

template <typename T, typename TC>
void band_nodes(const BandNodes<TC>& bn, const Grid3& g, const int* band, int nband, const T* f, T* x, void* u_raw,
                double omega, int sweeps, bool fine, cudaStream_t s0, const Fork* fk) {
    using C = typename Compute<T>::type;
    if (nband <= 0 || bn.nsub <= 0 || sweeps <= 0) return;
    const char* name = stencil_name("band_schwarz", prec_index<T>(), ST_JACOBI, fine);
    C* u = static_cast<C*>(u_raw);
    const NodeArgs<T, TC> a{bn.off, bn.node, bn.info, bn.org, bn.vals, bn.ncopies, f, x, u, (C)omega, sweeps, g};
    // bytes: per node copy its 45 values and two words, x and f of its faces; the owners' corrections
    const double per = kNodeVals * sizeof(TC) + 8.0 + 6.0 * sizeof(T);
    const double owned = (double)nband * sizeof(C);
    constexpr bool wide = std::is_same<T, double>::value;
    int top = 0, nl = 0;
    for (int cl = 0; cl < kNodeClasses; ++cl)
        if (bn.cls_count[cl] > 0) {
            top = cl;
            ++nl;
        }
    const bool single = one_launch(bn.nsub, wide);
    if (single) nl = 1;
    const bool forked = fk && fk->naux > 0 && nl > 1;
    if (forked) {
        DM_CUDA(cudaEventRecord(fk->fork, s0));
        for (int k = 0; k < std::min(nl - 1, fk->naux); ++k) DM_CUDA(cudaStreamWaitEvent(fk->aux[k], fk->fork, 0));
    }
    int li = 0;
    for (int cl = kNodeClasses - 1; cl >= 0; --cl) {
        if (bn.cls_count[cl] == 0 || (single && cl != top)) continue;
        const int ai = li++;   // the first class stays on s0
        cudaStream_t s = (forked && ai > 0 && ai - 1 < fk->naux) ? fk->aux[ai - 1] : s0;
        // (the fork's event wait or another class's launch comes before the rest: those are ordered in full)
        const bool chain = ai == 0 && !forked;
        const int first = single ? 0 : bn.cls_first[cl], count = single ? bn.nsub : bn.cls_count[cl];
        const double bytes = (single ? bn.copies() : (double)bn.cls_copies[cl]) * per + owned / nl;
        if constexpr (wide) {
            if (single || cl >= 2) launch_cluster<8>(name, bytes, first, count, a, chain, s);
            else if (cl == 1) launch_cluster<4>(name, bytes, first, count, a, chain, s);
            else launch_cluster<2>(name, bytes, first, count, a, chain, s);
        } else {
            switch (cl) {
                case 0: launch_node<T, TC, 256>(name, bytes, first, count, a, chain, s); break;
                case 1: launch_node<T, TC, 512>(name, bytes, first, count, a, chain, s); break;
                case 2: launch_node<T, TC, 768>(name, bytes, first, count, a, chain, s); break;
                default: launch_node<T, TC, 1024>(name, bytes, first, count, a, chain, s);
            }
        }
    }
    if (forked)
        for (int k = 0; k < std::min(nl - 1, fk->naux); ++k) {
            DM_CUDA(cudaEventRecord(fk->join[k], fk->aux[k]));
            DM_CUDA(cudaStreamWaitEvent(s0, fk->join[k], 0));
        }
    const char* add = stencil_name("band_add", prec_index<T>(), ST_JACOBI, fine);
    const double add_bytes = (double)nband * (8.0 + sizeof(C) + 2.0 * sizeof(T));
    const int nb = (nband + 255) / 256;
    if (forked) launch_b(add, add_bytes, k_band_add_node<T>, nb, 256, 0, s0, band, bn.uidx, nband, (const C*)u, x);
    else launch_chain(add, add_bytes, k_band_add_node<T>, nb, 256, 0, s0, band, bn.uidx, nband, (const C*)u, x);
}

// rows per thread and block size of a class (R = 0: the shared-memory variant;
// FP64 rows hold twice the registers, so FP64 stops at R = 2)
template <typename T>
void class_shape(int cl, int& R, int& nt) {
    const bool wide = sizeof(typename Compute<T>::type) == 8;
    switch (cl) {
        case 0: R = 1; nt = 256; break;
        case 1: R = 1; nt = 512; break;
        case 2: R = 2; nt = 512; break;
        case 3: R = wide ? 0 : 4; nt = 512; break;
        default: R = 0; nt = 512;
    }
}

template <typename T, typename TC>
void band_schwarz(const BandSchwarz<TC>& bs, const TC* invD, const Grid3& g, const int* band, int nband, const T* f,
                  T* x, double* u, double omega, int sweeps, bool fine, cudaStream_t s0, const Fork* fk) {
    if (nband <= 0 || bs.nsub <= 0 || sweeps <= 0) return;
    const char* name = stencil_name("band_schwarz", prec_index<T>(), ST_JACOBI, fine);
    // a level whose subdomains fit in one wave goes in a single launch shaped for
    // its largest class; larger levels launch each class with its own shape
    int top = 0;
    for (int cl = 0; cl < kSchwarzClasses; ++cl)
        if (bs.cls_count[cl] > 0) top = cl;
    const bool single = bs.nsub <= kSingleLaunchSubdomains;
    // classes launched here, and the stream each takes
    int nl = 0;
    for (int cl = 0; cl < kSchwarzClasses; ++cl)
        if (bs.cls_count[cl] > 0 && !(single && cl != top)) ++nl;
    const bool forked = fk && fk->naux > 0 && nl > 1;
    if (forked) {
        DM_CUDA(cudaEventRecord(fk->fork, s0));
        for (int a = 0; a < std::min(nl - 1, fk->naux); ++a) DM_CUDA(cudaStreamWaitEvent(fk->aux[a], fk->fork, 0));
    }
    int li = 0;
    for (int cl = 0; cl < kSchwarzClasses; ++cl) {
        if (bs.cls_count[cl] == 0 || (single && cl != top)) continue;
        const int ai = li++;   // the first class stays on s0
        cudaStream_t s = (forked && ai > 0 && ai - 1 < fk->naux) ? fk->aux[ai - 1] : s0;
        int R, nt;
        class_shape<T>(single ? top : cl, R, nt);
        const int first = single ? 0 : bs.cls_first[cl];
        const int count = single ? bs.nsub : bs.cls_count[cl];
        const size_t smem = schwarz_smem<T>(bs.maxbox, bs.maxrows, R);
        // bytes: per row copy its 15 coefficients, copy and pos words, and the
        // row's x, f and 1/D (the slot gathers of x hit the row's neighbours,
        // which are other copies' rows); per owned copy the correction u
        long long copies = 0, owned = 0;
        for (int k = 0; k < kSchwarzClasses; ++k)
            if (single || k == cl) {
                copies += bs.cls_copies[k];
                owned += bs.cls_owned[k];
            }
        const double bytes = (double)copies * (16.0 * sizeof(TC) + 8.0 + 2.0 * sizeof(T)) + 8.0 * (double)owned;
#define DM_SCHWARZ(RV, NV)                                                                                         \
    launch_b(name, bytes, k_band_schwarz<T, TC, RV, NV>, count, NV, smem, s, first, bs.off, bs.copy, bs.pos,     \
             bs.dims, bs.org, bs.vals, bs.ncopies, band, invD, f, (const T*)x, u, omega, sweeps, g, bs.maxbox,     \
             bs.maxrows)
        if (nt == 256) DM_SCHWARZ(1, 256);
        else if (R == 1) DM_SCHWARZ(1, 512);
        else if (R == 2) DM_SCHWARZ(2, 512);
        else if (R == 4) DM_SCHWARZ(4, 512);
        else DM_SCHWARZ(0, 512);
#undef DM_SCHWARZ
    }
    if (forked)
        for (int a = 0; a < std::min(nl - 1, fk->naux); ++a) {
            DM_CUDA(cudaEventRecord(fk->join[a], fk->aux[a]));
            DM_CUDA(cudaStreamWaitEvent(s0, fk->join[a], 0));
        }
    launch_b(stencil_name("band_add", prec_index<T>(), ST_JACOBI, fine), (double)nband * (12.0 + 2.0 * sizeof(T)),
             k_band_add<T>, (nband + 255) / 256, 256, 0, s0, band, nband, (const double*)u, x);
}

// Allow each variant the device's opt-in shared memory less its static share;
// the largest subdomain box must fit in it.
template <typename K>
void allow_smem(K kernel, size_t need) {
    int dev = 0, optin = 0;
    DM_CUDA(cudaGetDevice(&dev));
    DM_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    cudaFuncAttributes fa{};
    DM_CUDA(cudaFuncGetAttributes(&fa, kernel));
    const long long limit = (long long)optin - (long long)fa.sharedSizeBytes;
    DM_REQUIRE((long long)need <= limit, DM_ERR_INVALID_ARG,
               "band brick too large: a subdomain's local box exceeds shared memory (use a smaller brick)");
    DM_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)limit));
}

template <typename T, typename TC>
void band_schwarz_prepare(const SchwarzLayout& sl) {
    for (int cl = 0; cl < kSchwarzClasses; ++cl) {
        if (sl.cls_count[cl] == 0) continue;
        int R, nt;
        class_shape<T>(cl, R, nt);
        const size_t need = schwarz_smem<T>(sl.maxbox, sl.maxrows, R);
        if (nt == 256) allow_smem(k_band_schwarz<T, TC, 1, 256>, need);
        else if (R == 1) allow_smem(k_band_schwarz<T, TC, 1, 512>, need);
        else if (R == 2) allow_smem(k_band_schwarz<T, TC, 2, 512>, need);
        else if (R == 4) allow_smem(k_band_schwarz<T, TC, 4, 512>, need);
        else allow_smem(k_band_schwarz<T, TC, 0, 512>, need);
    }
}

#define DM_INST(T, TC)                                                                                           \
    template void band_schwarz<T, TC>(const BandSchwarz<TC>&, const TC*, const Grid3&, const int*, int, const T*, \
                                      T*, double*, double, int, bool, cudaStream_t, const Fork*);                \
    template void band_schwarz_prepare<T, TC>(const SchwarzLayout&);                                             \
    template void band_nodes<T, TC>(const BandNodes<TC>&, const Grid3&, const int*, int, const T*, T*, void*,   \
                                    double, int, bool, cudaStream_t, const Fork*);
template void band_node_vals<double>(const int*, const int*, int, const Grid3&, const int*, const double*, int,
                                     const double*, double*, int*, cudaStream_t);
template void band_node_vals<float>(const int*, const int*, int, const Grid3&, const int*, const double*, int,
                                    const double*, float*, int*, cudaStream_t);
DM_INST(double, double)
DM_INST(float, float)
DM_INST(__nv_bfloat16, float)
#undef DM_INST

}  // namespace dm

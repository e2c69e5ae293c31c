// Grid transfers of the geometric V-cycles (a design of this library; the
// paper's multigrid was algebraic, Sec. 6).
//
// Face prolongation P (coarse -> fine, fine grid = 2x coarse), per component:
//   across the face plane: a fine face on a coarse plane copies it, a fine face
//   half-way takes the mean of the two coarse faces around it;
//   within the plane: bilinear, weight 3/4 towards the nearer coarse face
//   centre and 1/4 towards the farther one; at a domain wall the missing
//   neighbour's weight goes to the nearer face.
// The fine result is masked by the open fine faces.  Restriction R = P^T / 8
// is evaluated from the same per-axis weights, masked by the open coarse faces.
//
// The cell transfers are part of the scalar V-cycle's kernels (dm_stencil.cu).
#include "dm_common.cuh"

namespace dm {

namespace {

constexpr int BX = 32, BY = 4, BZ = 2;
const dim3 kBlock(BX, BY, BZ);

// Weights with which a coarse face (coarse index c along an axis) gathers the
// fine faces 2c - 1 .. 2c + 2 of P^T along that axis: along the face normal the
// planes 2c-1, 2c, 2c+1 (1/2, 1, 1/2); within the plane the cells 2c-1 .. 2c+2
// (1/4, 3/4, 3/4, 1/4, the wall rule moving a missing neighbour's 1/4 onto the
// nearer face).  Positions outside the grid get weight 0 and are ghosts (zero in
// every vector).
__device__ __forceinline__ void restrict_axis(bool normal, int c, int nc, int nf, float w[4]) {
    if (normal) {
        w[0] = c >= 1 ? 0.5f : 0.f;
        w[1] = 1.f;
        w[2] = 2 * c + 1 <= nf ? 0.5f : 0.f;
        w[3] = 0.f;
    } else {
        const bool lo = c >= 1, hi = c + 1 < nc;
        w[0] = lo ? 0.25f : 0.f;
        w[1] = lo ? 0.75f : 1.f;
        w[2] = hi ? 0.75f : 1.f;
        w[3] = hi ? 0.25f : 0.f;
    }
}

template <typename T, typename TC, bool SYM>
__global__ void k_face_restrict(Grid3 gf, Grid3 gc, const TC* __restrict__ Ac, const T* r_in,
                                T* __restrict__ fc, const int* __restrict__ tiles) {
    using C = typename Compute<T>::type;
    int I, J, K;
    block_node(gc, tiles, I, J, K);
    chain_wait();
    const T* __restrict__ r = after_wait(r_in);
    if (I > gc.nx || J > gc.ny || K > gc.nz) return;
    const int q = gc.idx(I, J, K);
    const int base = gf.idx(2 * I - 1, 2 * J - 1, 2 * K - 1);
#pragma unroll
    for (int comp = 0; comp < 3; ++comp) {
        const int oq = comp * gc.np + q;
        C acc = C(0);
        if ((C)Ac[oq] > C(0)) {
            float wx[4], wy[4], wz[4];
            restrict_axis(comp == 0, I, gc.nx, gf.nx, wx);
            restrict_axis(comp == 1, J, gc.ny, gf.ny, wy);
            restrict_axis(comp == 2, K, gc.nz, gf.nz, wz);
            const T* rc = r + comp * gf.np + base;
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                if (comp == 2 && a == 3) continue;
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    if (comp == 1 && b == 3) continue;
                    const float wab = wz[a] * wy[b];
                    const T* row = rc + a * gf.sxy + b * gf.sx;
#pragma unroll
                    for (int d = 0; d < 4; ++d) {
                        if (comp == 0 && d == 3) continue;
                        acc += C(wab * wx[d]) * (C)to_c(row[d]);
                    }
                }
            }
            acc *= C(0.125);
            if (SYM) acc *= sqrt((C)Ac[oq]);
        }
        fc[oq] = to_store<T>(acc);
    }
}

template <typename T, typename TC, bool SYM>
__global__ void k_face_prolong(Grid3 gf, Grid3 gc, const TC* __restrict__ Af, const T* ec_in,
                               T* x, const int* __restrict__ tiles) {
    using C = typename Compute<T>::type;
    int i, j, k;
    block_node(gf, tiles, i, j, k);
    chain_wait();
    const T* __restrict__ ec = after_wait(ec_in);
    if (i > gf.nx || j > gf.ny || k > gf.nz) return;
    const int p = gf.idx(i, j, k);
    // the coarse cell of the node, and per axis the offset and weights of the
    // other face: across the plane (n) and within it (t); an axis without one has
    // offset 0 and weight 0
    const int nc[3] = {gc.nx, gc.ny, gc.nz}, f[3] = {i, j, k}, st[3] = {1, gc.sx, gc.sxy};
    const int q = gc.idx(i >> 1, j >> 1, k >> 1);
    int on[3], ot[3];
    float wn[3][2], wt[3][2];
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        const int c = f[ax] >> 1;
        const bool odd = f[ax] & 1;
        const int nb = odd ? c + 1 : c - 1;
        const bool inside = nb >= 0 && nb < nc[ax];
        on[ax] = odd ? st[ax] : 0;
        wn[ax][0] = odd ? 0.5f : 1.f;
        wn[ax][1] = odd ? 0.5f : 0.f;
        ot[ax] = inside ? (odd ? st[ax] : -st[ax]) : 0;
        wt[ax][0] = inside ? 0.75f : 1.f;
        wt[ax][1] = inside ? 0.25f : 0.f;
    }
#pragma unroll
    for (int comp = 0; comp < 3; ++comp) {
        const int op = comp * gf.np + p;
        if (!((C)Af[op] > C(0))) continue;
        const T* e = ec + comp * gc.np + q;
        C acc = C(0);
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int b = 0; b < 2; ++b)
#pragma unroll
                for (int d = 0; d < 2; ++d) {
                    const float w = (comp == 2 ? wn[2][a] : wt[2][a]) * (comp == 1 ? wn[1][b] : wt[1][b]) *
                                    (comp == 0 ? wn[0][d] : wt[0][d]);
                    const int o = (d ? (comp == 0 ? on[0] : ot[0]) : 0) + (b ? (comp == 1 ? on[1] : ot[1]) : 0) +
                                  (a ? (comp == 2 ? on[2] : ot[2]) : 0);
                    acc += C(w) * (C)to_c(e[o]);
                }
        if (SYM) acc /= sqrt((C)Af[op]);
        x[op] = to_store<T>((C)to_c(x[op]) + acc);
    }
}

// x <- A^(-1/2) x (inverse) or A^(1/2) x on the open faces (closed: 0)
template <typename T, typename TC>
__global__ void k_scale_sqrt_a(Domain d, const TC* __restrict__ A, int inverse, T* __restrict__ x) {
    using C = typename Compute<T>::type;
    for_each_entry(d, [&](long long r) {
        const C a = (C)A[r];
        const C f = a > C(0) ? (inverse ? C(1) / sqrt(a) : sqrt(a)) : C(0);
        x[r] = to_store<T>((C)to_c(x[r]) * f);
    });
}

}  // namespace

template <typename T, typename TC>
void face_restrict(const Grid3& gf, const Grid3& gc, const TC* Ac, const T* r, T* fc, const int* tiles_c,
                   int ntiles_c, cudaStream_t s, bool sym) {
    // every open fine face's r once; per open coarse face its A and f_c
    const double bytes = (double)gf.nopen * sizeof(T) + (double)gc.nopen * (sizeof(T) + sizeof(TC));
    if (sym)
        launch_chain("k_face_restrict", bytes, k_face_restrict<T, TC, true>, tile_grid(gc, tiles_c, ntiles_c, 1), kBlock, 0,
                 s, gf, gc, Ac, r, fc, tiles_c);
    else
        launch_chain("k_face_restrict", bytes, k_face_restrict<T, TC, false>, tile_grid(gc, tiles_c, ntiles_c, 1), kBlock,
                 0, s, gf, gc, Ac, r, fc, tiles_c);
}
template <typename T, typename TC>
void face_prolong_add(const Grid3& gf, const Grid3& gc, const TC* Af, const T* ec, T* x, const int* tiles_f,
                      int ntiles_f, cudaStream_t s, bool sym) {
    // every open coarse face's e_c once; per open fine face its A and x read and written
    const double bytes = (double)gc.nopen * sizeof(T) + (double)gf.nopen * (2.0 * sizeof(T) + sizeof(TC));
    if (sym)
        launch_chain("k_face_prolong", bytes, k_face_prolong<T, TC, true>, tile_grid(gf, tiles_f, ntiles_f, 1), kBlock, 0,
                 s, gf, gc, Af, ec, x, tiles_f);
    else
        launch_chain("k_face_prolong", bytes, k_face_prolong<T, TC, false>, tile_grid(gf, tiles_f, ntiles_f, 1), kBlock, 0,
                 s, gf, gc, Af, ec, x, tiles_f);
}
template <typename T, typename TC>
void scale_sqrt_a(const Domain& d, const TC* A, bool inverse, T* x, cudaStream_t s) {
    launch_b("k_scale_sqrt_a", d.live() * (2.0 * sizeof(T) + sizeof(TC)), k_scale_sqrt_a<T, TC>,
             d.tiles ? std::max(d.ntiles, 1) : 1216, 256, 0, s, d, A, inverse ? 1 : 0, x);
}
#define DM_INST(T, TC)                                                                                   \
    template void face_restrict<T, TC>(const Grid3&, const Grid3&, const TC*, const T*, T*, const int*, int,  \
                                       cudaStream_t, bool);                                                \
    template void face_prolong_add<T, TC>(const Grid3&, const Grid3&, const TC*, const T*, T*, const int*, int, \
                                          cudaStream_t, bool);                                               \
    template void scale_sqrt_a<T, TC>(const Domain&, const TC*, bool, T*, cudaStream_t);
DM_INST(double, double)
DM_INST(float, float)
DM_INST(__nv_bfloat16, float)
#undef DM_INST

}  // namespace dm

// The FP64 cell pass with its contractions on the integer pipe (fixed64.cuh).
//
// As FP64 multiply-adds (one output node per thread, 3 (p + 1) of them plus the
// weights per real column, 2 per clock and SM) the degree-4 stiffness of 16
// columns on 12,144 cells took 1,080 us, with the FP64 pipe 92 % busy, against
// 30 us for the bytes.  Here a block works on whole cells:
//   1. gather (hanging points through C), largest exponent per cell and column;
//   2. every value as a 60-bit integer on that scale, and the pointwise part
//      m (V + E.r) u (+ m sum_q U_pq u_q) in FP64, once per node;
//   3. three sweeps over pencils (lines of p + 1 nodes): with D = W^-1 Khat,
//        (A_K u)_abc = h w_a w_b w_c (sum_j D_aj u_jbc + sum_j D_bj u_ajc
//                                     + sum_j D_cj u_abj),
//      so all three directions share one scale and their 63-bit sums add up as
//      integers in shared memory; a thread holds a pencil's values in registers
//      and reads D from constant memory (operands of the multiply-adds), 5
//      shared-memory accesses per node and sweep instead of 10 (p + 1) / 2 per
//      output;
//   4. the last sweep rounds to float64 once, adds the pointwise part and
//      scatters.
// A thread keeps one column (c = t % nc) through all of it and takes the nodes
// or pencils t / nc, + R, ..: with items divided by the run-time column count
// in every loop the kernel issued 560 instructions per node and column.
// Hanging nodes (constraint rows of 17 masters on average at degree 4) are
// listed and taken in loops of their own, which a warp runs for its listed
// nodes only; walked in place they cost every warp that held one.
// Per node and column: 9 (p + 1) IMAD.WIDE (31 per clock and SM), one
// int64 -> float64 conversion and one FP64 multiply-add.  The stiffness above
// takes 346 us; 9 columns at degree 3 on 4,164 cells 46 us instead of 120.  What
// bounds it now is instruction issue and the barriers between the sweeps.
// Each sum is exact to about 2^-57 of the cell column's largest |D| |u|.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "afem_internal.h"
#include "cell_common.cuh"
#include "fixed64.cuh"
#include "vec_common.cuh"

namespace afem {

// D = W^-1 Khat on its own scale (biased exponent e of its largest entry).
struct FxBasis {
    int h[kMaxP1 * kMaxP1], l[kMaxP1 * kMaxP1];
    int e;
    double w3[kMaxP1 * kMaxP1 * kMaxP1];   // w_a w_b w_c, rounded once
};

static FxBasis make_fx_basis(const Basis1D& b) {
    FxBasis f{};
    const int p1 = b.p + 1;
    long double D[kMaxP1 * kMaxP1], top = 0.0L;   // more than 60 bits of the quotient
    for (int i = 0; i < p1; ++i)
        for (int j = 0; j < p1; ++j) {
            D[i * p1 + j] = static_cast<long double>(b.K[i][j]) / b.w[i];
            top = std::max(top, std::fabs(D[i * p1 + j]));
        }
    f.e = std::ilogb(top) + 1023;
    for (int i = 0; i < p1 * p1; ++i) {
        const int64_t x = std::llrint(std::ldexp(D[i], 1082 - f.e));   // |x| < 2^60
        const int32_t l = int32_t(uint32_t(uint64_t(x) & 0xFFFFFFFFull));
        f.l[i] = l;
        f.h[i] = int((x - l) >> 32);
    }
    for (int c = 0; c < p1; ++c)
        for (int d = 0; d < p1; ++d)
            for (int i = 0; i < p1; ++i)
                f.w3[i + p1 * (d + p1 * c)] = double(static_cast<long double>(b.w[i]) * b.w[d] * b.w[c]);
    return f;
}

constexpr int kFxColumns = 16;   // real columns of a block at most

// Shared memory of cpb cells and nc columns.
static size_t cell_fx_smem(int nn, int cpb, int nc, bool pointwise) {
    return size_t(cpb) * nn * nc * (sizeof(double) + sizeof(int2) + (pointwise ? sizeof(double) : 0)) +
           size_t(cpb) * nn * 3 * sizeof(double) + size_t(cpb) * nc * sizeof(int) + size_t(cpb) * nn * 2 * sizeof(int) +
           size_t(cpb) * sizeof(double4);
}

// One component of acc + w u: the real (odd = 0) or the imaginary part.  The
// operands are selected, with the sign as a bit, so that lanes of both kinds
// share the two multiply-adds (as two expressions a warp ran all four: 3 complex
// orbitals at degree 3 on 4,164 cells took 82 us, now 66 us).
__device__ __forceinline__ double mean_field_part(double2 w, double2 u, int odd, double acc) {
    const double same = odd ? u.y : u.x, other = odd ? u.x : u.y;
    const double signed_other =
        __hiloint2double(__double2hiint(other) ^ (odd ? 0 : int(0x80000000u)), __double2loint(other));
    return fma(w.x, same, fma(w.y, signed_other, acc));
}

// PT 0: y += A x (real columns).  PT 1: y += H1~ x.  PT 2: the G cell pass, H1~ x
// plus the mean fields U (real columns 2p, 2p + 1: orbital p).  x, y: [N][ncol]
// doubles; blockIdx.y selects kFxColumns of them.
template <int P, int PT>
__global__ void __launch_bounds__(256, PT == 2 ? 5 : 1) cell_fx_kernel(const __grid_constant__ CellArgs a,
                                                      const __grid_constant__ FxBasis D, const double* __restrict__ x,
                                                      const double2* __restrict__ U, double* __restrict__ y, int ncol,
                                                      int cpb, int64_t ncell) {
    constexpr int P1 = P + 1, NN = P1 * P1 * P1, NP = P1 * P1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int c0 = blockIdx.y * kFxColumns, nc = min(ncol - c0, kFxColumns);
    const int64_t cell0 = int64_t(blockIdx.x) * cpb;
    const int nb = int(min(int64_t(cpb), ncell - cell0));   // cells of this block
    double4* s_g = reinterpret_cast<double4*>(smem_raw);                    // [cpb]
    double* s_u = reinterpret_cast<double*>(s_g + cpb);                     // [cpb][NN][nc] values, then sums
    long long* s_t = reinterpret_cast<long long*>(s_u);
    int2* s_i = reinterpret_cast<int2*>(s_u + cpb * NN * nc);               // [cpb][NN][nc] (l, h)
    double* s_pu = reinterpret_cast<double*>(s_i + cpb * NN * nc);          // [cpb][NN][nc] pointwise part (PT > 0)
    double* s_hw = s_pu + (PT ? cpb * NN * nc : 0);                         // [cpb][NN] c_kin h w_a w_b w_c
    double* s_pot = s_hw + cpb * NN;                                        // [cpb][NN] m (V + E.r)
    double* s_wq = s_pot + cpb * NN;                                        // [cpb][NN] m
    int* s_e = reinterpret_cast<int*>(s_wq + cpb * NN);                     // [cpb][nc]
    int* s_idx = s_e + cpb * nc;                                            // [cpb][NN]
    int* s_hl = s_idx + cpb * NN;                                           // [cpb][NN] the hanging nodes
    __shared__ int s_nh;
    const int tid = threadIdx.x, bs = blockDim.x;
    const int R = bs / nc;                       // rows of threads
    const int r0 = tid / nc, c = tid - r0 * nc;
    const bool on = r0 < R;
    if (tid == 0) s_nh = 0;
    __syncthreads();
    for (int i = tid; i < nb * NN; i += bs) {
        const int idx = a.cell_node[cell0 * NN + i];
        s_idx[i] = idx;
        if (idx < 0) s_hl[atomicAdd(&s_nh, 1)] = i;
    }
    for (int i = tid; i < nb; i += bs) s_g[i] = a.geom[cell0 + i];
    for (int i = tid; i < nb * nc; i += bs) s_e[i] = kFxMinExp;
    __syncthreads();
    const double* xc = x + c0 + c;
    double* yc = y + c0 + c;
    const int nodes = nb * NN, n_int = int(a.n_interior), nh = on ? s_nh : 0;
    for (int i0 = on ? r0 : nodes; i0 < nodes; i0 += 4 * R) {   // four values in flight
        double v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int i = i0 + q * R;
            v[q] = 0.0;
            if (i < nodes) {
                const int idx = s_idx[i];
                if (idx >= 0 && !(a.masked && idx >= n_int)) v[q] = xc[int64_t(idx) * ncol];
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int i = i0 + q * R;
            if (i >= nodes) break;
            if (s_idx[i] < 0) continue;
            s_u[i * nc + c] = v[q];
            const int e = int(fx_expbits(v[q]) >> 20);
            if (e > kFxMinExp) atomicMax(&s_e[(i / NN) * nc + c], e);
        }
    }
    for (int j = r0; j < nh; j += R) {
        const int i = s_hl[j];
        const double v = gather_value<double>(a, s_idx[i], x, ncol, c0 + c);
        s_u[i * nc + c] = v;
        const int e = int(fx_expbits(v) >> 20);
        if (e > kFxMinExp) atomicMax(&s_e[(i / NN) * nc + c], e);
    }
    for (int i = tid; i < nodes; i += bs) {
        const int cell = i / NN, n = i - cell * NN;
        const double4 g = s_g[cell];
        const double hw = g.w * D.w3[n];
        s_hw[i] = a.c_kin * hw;
        if constexpr (PT > 0) {
            const int idx = s_idx[i];
            const int ia = n % P1, ib = (n / P1) % P1, ic = n / NP;
            const double V = idx >= 0 ? a.v_master[idx] : a.v_hang[-idx - 1];
            const double px = g.x + g.w * a.B.xi[ia], py = g.y + g.w * a.B.xi[ib], pz = g.z + g.w * a.B.xi[ic];
            const double wq = hw * g.w * g.w;
            s_wq[i] = wq;
            s_pot[i] = wq * (V + a.E[0] * px + a.E[1] * py + a.E[2] * pz);
        }
    }
    __syncthreads();
    const int n = nc >> 1, nn2 = n * n, p = c >> 1;   // PT 2: orbitals
    for (int i = on ? r0 : nodes; i < nodes; i += R) {
        const int it = i * nc + c;
        const double v = s_u[it];
        const Fx f = fx_make(v, s_e[(i / NN) * nc + c]);
        s_i[it] = make_int2(f.l, f.h);
        if constexpr (PT == 1) s_pu[it] = s_pot[i] * v;
        if constexpr (PT == 2) {   // this column's part of m sum_q U_pq u_q
            const double2* su = reinterpret_cast<const double2*>(s_u) + i * n;
            const int idx = s_idx[i];
            const double2* row = idx >= 0 ? U + int64_t(idx) * nn2
                                          : a.u_hang ? a.u_hang + int64_t(-idx - 1) * nn2 : nullptr;
            double mf = 0.0;
            if (row) {
#pragma unroll 4
                for (int q = 0; q < n; ++q) mf = mean_field_part(row[p * n + q], su[q], c & 1, mf);
            } else {
                CellArgs au = a;
                au.masked = 0;   // the mean fields are defined on all masters
                for (int q = 0; q < n; ++q)
                    mf = mean_field_part(gather_value<double2>(au, idx, U, nn2, p * n + q), su[q], c & 1, mf);
            }
            s_pu[it] = fma(s_wq[i], mf, s_pot[i] * v);
        }
    }
    __syncthreads();
    const int pencils = nb * NP;
#pragma unroll
    for (int dir = 0; dir < 3; ++dir) {
        const int step = (dir == 0 ? 1 : dir == 1 ? P1 : NP) * nc;   // between a pencil's nodes
        for (int pc = on ? r0 : pencils; pc < pencils; pc += R) {
            const int cell = pc / NP, q = pc - cell * NP;
            const int qa = q % P1, qb = q / P1;
            const int n0 = cell * NN + (dir == 0 ? P1 * q : dir == 1 ? qa + NP * qb : q);
            const int base = n0 * nc + c;
            Fx u[P1];
#pragma unroll
            for (int j = 0; j < P1; ++j) {
                const int2 v = s_i[base + j * step];
                u[j] = Fx{v.y, v.x};
            }
            const int e = s_e[cell * nc + c];
#pragma unroll
            for (int i = 0; i < P1; ++i) {
                FxAcc acc{0, 0};
#pragma unroll
                for (int j = 0; j < P1; ++j) fx_mad_const(acc, Fx{D.h[i * P1 + j], D.l[i * P1 + j]}, u[j]);
                long long t = (acc.hh << 1) + (acc.x >> 31);
                const int o = base + i * step;
                if (dir > 0) t += s_t[o];
                if (dir < 2) {
                    s_t[o] = t;
                } else {
                    // t 2^(e + D.e - 2101), the power of two by the exponent field where
                    // its result is a normal number (t < 2^62)
                    double r = __ll2double_rn(t);
                    const int k = e + D.e - 2101;
                    if (k <= 2046 - 1086) r = t == 0 ? 0.0 : __hiloint2double(__double2hiint(r) + (k << 20), __double2loint(r));
                    else r = e == 0x7FF ? __hiloint2double(0x7FF80000, 0) : ldexp(r, k);
                    const int node = n0 + i * NP;
                    r = PT ? fma(r, s_hw[node], s_pu[o]) : r * s_hw[node];
                    const int idx = s_idx[node];
                    if (idx < 0) s_u[o] = r;   // (in place of this node's t)
                    else if (!(a.masked && idx >= n_int)) atomicAdd(yc + int64_t(idx) * ncol, r);
                }
            }
        }
        __syncthreads();
    }
    for (int j = r0; j < nh; j += R) {
        const int i = s_hl[j];
        scatter_value<double>(a, s_idx[i], y, ncol, c0 + c, s_u[i * nc + c]);
    }
}

template <int P, int PT>
static int launch_p(const afem_mesh* m, const CellArgs& a, const double* x, const double2* U, double* y, int ncol,
                    cudaStream_t s) {
    constexpr int P1 = P + 1, NN = P1 * P1 * P1;
    const int64_t ncell = m->dev.ncell;
    const int nc = std::min(ncol, kFxColumns);
    // whole cells per block: as many as give each thread one pencil per sweep
    const int per = P1 * P1 * nc, cpb = std::max(1, std::min(16, 256 / per));
    const int rounds = (cpb * per + 255) / 256;   // pencils of a thread
    const int rows = (cpb * P1 * P1 + rounds - 1) / rounds;
    const int block = std::min(256, (rows * nc + 31) / 32 * 32);
    const size_t smem = cell_fx_smem(NN, cpb, nc, PT > 0);
    AFEM_CUDA_TRY(allow_dyn_smem(cell_fx_kernel<P, PT>));
    const FxBasis D = make_fx_basis(m->basis);
    const dim3 grid(unsigned((ncell + cpb - 1) / cpb), unsigned((ncol + kFxColumns - 1) / kFxColumns));
    AFEM_LAUNCH((cell_fx_kernel<P, PT>), grid, block, smem, s, a, D, x, U, y, ncol, cpb, ncell);
    AFEM_CUDA_TRY(cudaGetLastError());
    return AFEM_OK;
}

template <int PT>
static int launch_pt(const afem_mesh* m, const CellArgs& a, const double* x, const double2* U, double* y, int ncol,
                     cudaStream_t s) {
    if (m->dev.ncell == 0) return AFEM_OK;
    switch (m->dev.p) {
        case 1: return launch_p<1, PT>(m, a, x, U, y, ncol, s);
        case 2: return launch_p<2, PT>(m, a, x, U, y, ncol, s);
        case 3: return launch_p<3, PT>(m, a, x, U, y, ncol, s);
        case 4: return launch_p<4, PT>(m, a, x, U, y, ncol, s);
    }
    return set_error(AFEM_EINVAL, "degree out of range");
}

// y += A x on ncol real columns, or (a.with_pot == 1, ncol = 2 n) y += H1~ x with
// the mean fields of the G pass when U is given; a as the FP64 cell kernels take it.
int launch_cell_fx(const afem_mesh* m, const CellArgs& a, const double* x, const double2* U, double* y, int ncol,
                   cudaStream_t s) {
    if (!a.with_pot) return launch_pt<0>(m, a, x, U, y, ncol, s);
    return U ? launch_pt<2>(m, a, x, U, y, ncol, s) : launch_pt<1>(m, a, x, U, y, ncol, s);
}

}  // namespace afem

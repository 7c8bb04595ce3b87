// The FP64 cell pass with its contractions on the integer pipe (fixed64.cuh).
//
// As FP64 multiply-adds (one output node per thread, 3 (p + 1) of them plus the
// weights per real column, 2 per clock and SM) the degree-4 stiffness of 16
// columns on 12,144 cells took 1,080 us, with the FP64 pipe 92 % busy, against
// 30 us for the bytes.  Here a block works on whole cells:
//   1. gather (hanging points through C) and, for G, the pointwise part
//      m (V + E.r) u + m sum_q U_pq u_q in FP64, once per node;
//   2. three sweeps over pencils (lines of p + 1 nodes): with D = W^-1 Khat,
//        (A_K u)_abc = h w_a w_b w_c (sum_j D_aj u_jbc + sum_j D_bj u_ajc
//                                     + sum_j D_cj u_abj);
//      a thread holds a pencil's values in registers, brings them to the scale of
//      the largest of them (60-bit integers) and reads D from constant memory
//      (operands of the multiply-adds), each row of D on its own scale.  The
//      63-bit sums of the three directions meet in shared memory, each with its
//      exponent, shifted to the larger of two when they are added;
//   3. the last sweep rounds to float64 once, adds the pointwise part and
//      scatters.
// What an output may be off by follows from its own three lines, as in FP64:
// one scale for all nodes of a cell took 346 us instead of 595 (46 instead of 61
// for the 9 columns below), but rounded small values on the scale of the cell's
// largest.  Each line's sum keeps 2^-60 of the largest |D||u| (degree 4 needs the
// products of the low words for that, its rows of D spanning 2^6); against a chain
// of FP64 multiply-adds the error over sum |D||u| is 0.05-0.7 of its size (rms,
// lines of equal, of single and of widely different values).  Lines with an
// infinity or NaN give what FP64 gives on that line; tiny ones are scaled up first.
// A thread keeps one column (c = t % nc) through all of it and takes the nodes
// or pencils t / nc, + R, ..: with items divided by the run-time column count
// in every loop the kernel issued 560 instructions per node and column.
// Hanging nodes (constraint rows of 17 masters on average at degree 4) are
// listed and taken in loops of their own, which a warp runs for its listed
// nodes only; walked in place they cost every warp that held one.
// Per node and column: 9 (p + 1) IMAD.WIDE (12 at degree 4; 31 per clock and SM),
// three conversions to integers, one back and one FP64 multiply-add.  The
// stiffness above takes 595 us; 9 columns at degree 3 on 4,164 cells 61 us instead
// of 120, with the mean fields of 3 orbitals 71 us instead of 106.  Counters of the
// first: 504 instructions per node and column, issue 53 %, multiply pipe 42 %, ALU
// 38 %, FP64 pipe 27 %, DRAM 6 %; warps wait for the barriers between sweeps, for
// instructions and for the multiply pipe.
// The sums of the directions as FP64 numbers took longer (622 and 81 us): the
// conversions run at 1.6 per clock and SM.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "afem_internal.h"
#include "cell_common.cuh"
#include "fixed64.cuh"
#include "vec_common.cuh"

namespace afem {

// D = W^-1 Khat, each row on the scale of its largest entry (biased exponent e).
template <int P>
struct FxBasis {
    static constexpr int P1 = P + 1;
    int h[P1 * P1], l[P1 * P1];
    int l8[P1 * P1];   // l / 8, for the products of low words
    int e[P1];
    double w3[P1 * P1 * P1], w3_lo[P1 * P1 * P1];   // w_a w_b w_c as a sum of two
};

// From the closed forms of the Gauss-Lobatto points and weights in long double, as
// D has 60 bits.  Error of the stiffness in norm on random columns, degrees 1 to 4:
// 1.1, 0.9, 0.9 and 0.8e-16 (with K and w rounded to float64 first 1.1, 2.5, 3.9 and
// 8.7e-16; as FP64 multiply-adds 1.1, 1.6, 4.3 and 8.6e-16).  H1 without potential:
// 1.2, 1.6, 1.8 and 1.0e-16 (FP64 multiply-adds 1.2, 1.3, 1.7 and 4.6e-16): what is
// left is the rounding of the lumped mass, the same in every cell of a size.
template <int P>
static FxBasis<P> make_fx_basis() {
    const long double z = P == 3 ? std::sqrt(0.2L) : std::sqrt(3.0L / 7.0L);   // the inner points on [-1, 1]
    constexpr int p = P, p1 = P + 1;
    long double x[kMaxP1] = {}, w[kMaxP1] = {};
    x[0] = -1.0L;
    x[p] = 1.0L;
    w[0] = w[p] = 1.0L / (p * p1);
    if (p == 2) w[1] = 2.0L / 3.0L;
    if (p >= 3) {
        x[1] = -z;
        x[p - 1] = z;
        w[1] = w[p - 1] = p == 3 ? 5.0L / 12.0L : 49.0L / 180.0L;
    }
    if (p == 4) w[2] = 16.0L / 45.0L;
    long double d[kMaxP1][kMaxP1];   // d[q][j] = L_j'(x_q) on [0, 1]
    for (int q = 0; q < p1; ++q) {
        d[q][q] = 0.0L;
        for (int j = 0; j < p1; ++j) {
            if (j == q) continue;
            long double r = 2.0L / (x[j] - x[q]);
            for (int k = 0; k < p1; ++k)
                if (k != q && k != j) r *= (x[q] - x[k]) / (x[j] - x[k]);
            d[q][j] = r;
            d[q][q] -= r;
        }
    }
    FxBasis<P> f{};
    for (int i = 0; i < p1; ++i) {
        long double D[kMaxP1], top = 0.0L;
        for (int j = 0; j < p1; ++j) {
            D[j] = 0.0L;
            for (int q = 0; q < p1; ++q) D[j] += w[q] * d[q][i] * d[q][j];
            D[j] /= w[i];
            top = std::max(top, std::fabs(D[j]));
        }
        f.e[i] = std::ilogb(top) + 1023;
        for (int j = 0; j < p1; ++j) {
            const int64_t v = std::llrint(std::ldexp(D[j], 1082 - f.e[i]));   // |v| < 2^60
            const int32_t l = int32_t(uint32_t(uint64_t(v) & 0xFFFFFFFFull));
            f.l[i * p1 + j] = l;
            f.l8[i * p1 + j] = l >> 3;
            f.h[i * p1 + j] = int((v - l) >> 32);
        }
    }
    for (int c = 0; c < p1; ++c)
        for (int e = 0; e < p1; ++e)
            for (int i = 0; i < p1; ++i) {
                const long double w3 = w[i] * w[e] * w[c];
                const int q = i + p1 * (e + p1 * c);
                f.w3[q] = double(w3);
                f.w3_lo[q] = double(w3 - f.w3[q]);
            }
    return f;
}

// Formed with the first launch of a degree (software arithmetic on an arm64 host).
template <int P>
static const FxBasis<P>& fx_basis() {
    static const FxBasis<P> f = make_fx_basis<P>();
    return f;
}

constexpr int kFxColumns = 16;   // real columns of a block at most

// Shared memory of cpb cells and nc columns (fields: with mean fields).
static size_t cell_fx_smem(int nn, int cpb, int nc, bool fields) {
    return size_t(cpb) * nn * nc * (2 * sizeof(double) + sizeof(short) + (fields ? sizeof(double) : 0)) +
           size_t(cpb) * nn * 3 * sizeof(double) + size_t(cpb) * nn * 2 * sizeof(int) + size_t(cpb) * sizeof(double4);
}

// Exponents of sums that are no number (above every other): sums of lines with
// an infinity or NaN.
constexpr int kSumInf = 0x7F00, kSumMinusInf = 0x7F01, kSumNan = 0x7F02;

// Row i of D on a line with an infinity or NaN: which of the three the sum is.
template <int P>
__device__ __noinline__ int non_finite_sum(const double* u, int step, const FxBasis<P>& D, int i) {
    double f = 0.0;
    for (int j = 0; j <= P; ++j)
        f = fma(fma(double(D.h[i * (P + 1) + j]), 4294967296.0, double(D.l[i * (P + 1) + j])), u[j * step], f);
    return f > 0.0 ? kSumInf : f < 0.0 ? kSumMinusInf : kSumNan;
}

// One component of acc + w u: the real (odd = 0) or the imaginary part.  The
// operands are selected, with the sign as a bit, so that lanes of both kinds
// share the two multiply-adds (as two expressions a warp ran all four: the pass on 3
// complex orbitals at degree 3 and 4,164 cells took 82 us in place of 66, in the
// form of one scale per cell).
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
__global__ void __launch_bounds__(256, PT == 2 ? 4 : 3) cell_fx_kernel(const __grid_constant__ CellArgs a,
                                                      const __grid_constant__ FxBasis<P> D, const double* __restrict__ x,
                                                      const double2* __restrict__ U, double* __restrict__ y, int ncol,
                                                      int cpb, int64_t ncell) {
    constexpr int P1 = P + 1, NN = P1 * P1 * P1, NP = P1 * P1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int c0 = blockIdx.y * kFxColumns, nc = min(ncol - c0, kFxColumns);
    const int64_t cell0 = int64_t(blockIdx.x) * cpb;
    const int nb = int(min(int64_t(cpb), ncell - cell0));   // cells of this block
    double4* s_g = reinterpret_cast<double4*>(smem_raw);                    // [cpb]
    double* s_u = reinterpret_cast<double*>(s_g + cpb);                     // [cpb][NN][nc] values
    long long* s_t = reinterpret_cast<long long*>(s_u + cpb * NN * nc);     // [cpb][NN][nc] running sums
    double* s_r = reinterpret_cast<double*>(s_t);                           // (and results of hanging nodes)
    double* s_pu = reinterpret_cast<double*>(s_t + cpb * NN * nc);          // [cpb][NN][nc] pointwise part (PT 2)
    double* s_hw = s_pu + (PT == 2 ? cpb * NN * nc : 0);                    // [cpb][NN] c_kin h w_a w_b w_c
    double* s_pot = s_hw + cpb * NN;                                        // [cpb][NN] m (V + E.r)
    double* s_wq = s_pot + cpb * NN;                                        // [cpb][NN] m
    int* s_idx = reinterpret_cast<int*>(s_wq + cpb * NN);                   // [cpb][NN]
    int* s_hl = s_idx + cpb * NN;                                           // [cpb][NN] the hanging nodes
    short* s_x = reinterpret_cast<short*>(s_hl + cpb * NN);                 // [cpb][NN][nc] exponents of the sums
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
        }
    }
    for (int j = r0; j < nh; j += R) {
        const int i = s_hl[j];
        s_u[i * nc + c] = gather_value<double>(a, s_idx[i], x, ncol, c0 + c);
    }
    for (int i = tid; i < nodes; i += bs) {
        const int cell = i / NN, n = i - cell * NN;
        const double4 g = s_g[cell];
        if constexpr (PT == 0) {
            s_hw[i] = a.c_kin * fma(g.w, D.w3[n], g.w * D.w3_lo[n]);   // rounded once
        } else {   // the weights as the lumped mass has them, which divides the result
            const int idx = s_idx[i];
            const int ia = n % P1, ib = (n / P1) % P1, ic = n / NP;
            const double V = idx >= 0 ? a.v_master[idx] : a.v_hang[-idx - 1];
            const double px = g.x + g.w * a.B.xi[ia], py = g.y + g.w * a.B.xi[ib], pz = g.z + g.w * a.B.xi[ic];
            const double wq = g.w * g.w * g.w * a.B.w[ia] * a.B.w[ib] * a.B.w[ic];
            s_hw[i] = a.c_kin * (g.w * a.B.w[ia] * a.B.w[ib] * a.B.w[ic]);
            s_wq[i] = wq;
            s_pot[i] = wq * (V + a.E[0] * px + a.E[1] * py + a.E[2] * pz);
        }
    }
    __syncthreads();
    if constexpr (PT == 2) {   // this column's part of m sum_q U_pq u_q
        const int n = nc >> 1, nn2 = n * n, p = c >> 1;   // orbitals
        for (int i = on ? r0 : nodes; i < nodes; i += R) {
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
            s_pu[i * nc + c] = fma(s_wq[i], mf, s_pot[i] * s_u[i * nc + c]);
        }
    }   // (each entry is read by a thread of the same column after the sweeps' barriers)
    const int pencils = nb * NP;
#pragma unroll
    for (int dir = 0; dir < 3; ++dir) {
        const int step = (dir == 0 ? 1 : dir == 1 ? P1 : NP) * nc;   // between a pencil's nodes
        for (int pc = on ? r0 : pencils; pc < pencils; pc += R) {
            const int cell = pc / NP, q = pc - cell * NP;
            const int qa = q % P1, qb = q / P1;
            const int n0 = cell * NN + (dir == 0 ? P1 * q : dir == 1 ? qa + NP * qb : q);
            const int base = n0 * nc + c;
            double v[P1];
            unsigned eb = 0u;
#pragma unroll
            for (int j = 0; j < P1; ++j) {
                v[j] = s_u[base + j * step];
                eb = max(eb, fx_expbits(v[j]));
            }
            int e = int(eb >> 20), off = 0;
            if (e < 2 * kFxMinExp) {   // zero, or too small for the integers: up by 2^600
                off = 600;
                eb = 0u;
#pragma unroll
                for (int j = 0; j < P1; ++j) {
                    v[j] *= __hiloint2double((1023 + 600) << 20, 0);
                    eb = max(eb, fx_expbits(v[j]));
                }
                e = int(eb >> 20);
            }
            Fx u[P1];
#pragma unroll
            for (int j = 0; j < P1; ++j) u[j] = fx_make(v[j], max(e, kFxMinExp));
#pragma unroll
            for (int i = 0; i < P1; ++i) {
                FxAcc acc{0, 0};
                long long low = 0;
#pragma unroll
                for (int j = 0; j < P1; ++j) {
                    fx_mad_const(acc, Fx{D.h[i * P1 + j], D.l[i * P1 + j]}, u[j]);
                    if constexpr (P == 4) low += static_cast<long long>(D.l8[i * P1 + j]) * u[j].l;
                }
                if constexpr (P == 4) acc.x += low >> 29;
                long long t = (acc.hh << 4) + (acc.x >> 28);
                int E = e ? e + D.e[i] - off : 0;   // the sum is t 2^(E - 2104)
                if (e == 0x7FF) E = non_finite_sum<P>(s_u + base, step, D, i);
                const int o = base + i * step;
                if (dir > 0) {
                    const int E1 = s_x[o], M = max(E, E1);
                    t = (t >> min(M - E, 63)) + (s_t[o] >> min(M - E1, 63));
                    E = (min(E, E1) >= kSumInf && E != E1) ? kSumNan : M;
                }
                if (dir < 2) {
                    s_t[o] = t;
                    s_x[o] = short(E);
                } else {
                    const int node = n0 + i * NP, idx = s_idx[node];
                    // the power of two by the exponent field where the result is a normal number (t < 2^63)
                    double r = __ll2double_rn(t);
                    const double pu = PT == 2 ? s_pu[o] : PT == 1 ? s_pot[node] * s_u[o] : 0.0;
                    const int k = t == 0 ? 0 : E - 2104;
                    if (unsigned(k + 1021) <= 1980u && E < kSumInf) {
                        r = t == 0 ? 0.0 : __hiloint2double(__double2hiint(r) + (k << 20), __double2loint(r));
                        r = PT ? fma(r, s_hw[node], pu) : r * s_hw[node];
                    } else {
                        r = E == kSumNan ? __hiloint2double(0x7FF80000, 0) : E == kSumInf ? __hiloint2double(0x7FF00000, 0)
                          : E == kSumMinusInf ? __hiloint2double(int(0xFFF00000), 0) : ldexp(r * s_hw[node], k);
                        r += pu;
                    }
                    if (idx < 0) s_r[o] = r;   // (in place of this node's sum)
                    else if (!(a.masked && idx >= n_int)) atomicAdd(yc + int64_t(idx) * ncol, r);
                }
            }
        }
        __syncthreads();
    }
    for (int j = r0; j < nh; j += R) {
        const int i = s_hl[j];
        scatter_value<double>(a, s_idx[i], y, ncol, c0 + c, s_r[i * nc + c]);
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
    const size_t smem = cell_fx_smem(NN, cpb, nc, PT == 2);
    if (smem > 48 * 1024) AFEM_CUDA_TRY(allow_dyn_smem(cell_fx_kernel<P, PT>));
    const dim3 grid(unsigned((ncell + cpb - 1) / cpb), unsigned((ncol + kFxColumns - 1) / kFxColumns));
    AFEM_LAUNCH((cell_fx_kernel<P, PT>), grid, block, smem, s, a, fx_basis<P>(), x, U, y, ncol, cpb,
                ncell);
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

// Short-iterative Arnoldi propagation of all orbitals at once (Sec. 3.2).
//
// With phi, the RDMs, the mean fields and the field frozen at t, the packed
// orbital equation (Eq. packed_orb_eom) is linear, i d(phi)/dt = G phi, and
// phi(t + dt) = exp(-i G dt) phi(t).  The Krylov space of G from phi is built
// by Arnoldi in the inner product <u, v> = sum_p u_p^H M_L v_p; then
// phi(t+dt) = beta V_m exp(-i dt H_m) e_1.
// G applied to the stacked orbitals v (Eqs. orb_eom / discretized_eom, X = 0):
//   z_p = H1~ v_p + C^T diag(m_f) sum_q (C U_pq) o (C v_q)      (one cell pass)
//   y_p = M_L^-1 z_p,   (G v)_p = y_p - sum_j phi_j (phi_j^H M_L y_p)
// and phi_j^H M_L y_p = phi_j^H z_p, so the projector needs no extra scaling.
//
// Orthogonalisation: classical Gram-Schmidt, one pass for all inner products
// (fused with the projector pass of G) and one for the update, plus a second
// pair of passes only when the update cancelled the vector to below 1e-2 of
// its norm (the Daniel-Gragg-Kaufman-Stewart test with a loose threshold).
// GB300 runs FP64 at about 1/64 of its FP32 rate, so the sums and products of
// these passes run on the integer pipe (fixed64.cuh) on a basis stored for it
// (KrylovBasis), and in the precision form the projector (part of applying G)
// runs in FP32.  The
// Hessenberg matrix and the norms stay on the device; the host waits once
// per substep, after the candidate substep exponentials are evaluated.
#include <algorithm>
#include <cmath>
#include <vector>

#include "afem_internal.h"
#include "arnoldi.cuh"
#include "fixed64.cuh"
#include "vec_common.cuh"

namespace afem {

// S[a][b] = sum_k w_k conj(A[k][a]) B[k][b] over rows k < n_rows (w_k = 1 when
// w is null), reduced in the same launch: partial rows of 2*kout doubles (re,
// im interleaved); the last block writes out[kout].  diag != 0: only a == b
// (kout = na), else all na*nb pairs (kout = na*nb <= 128).  On small meshes
// latency bounds it, so a thread has kDotRows rows in flight, the threads' sums
// meet in a tree, and row_blocks() leaves few rows to the last block: 3 x 3 pairs
// on 102,533 rows took 27 us with four blocks per SM and one row at a time, 19 us
// with two, 18 us with one.
constexpr int kDotRows = 4;
__global__ void __launch_bounds__(kRedThreads) cdot_fused_kernel(const double2* __restrict__ A, int na, const double2* __restrict__ B, int nb,
                                  const double* __restrict__ w, int64_t n_rows, int diag, double* __restrict__ partial,
                                  unsigned* __restrict__ counter, double2* __restrict__ out) {
    __shared__ double sx[kRedThreads], sy[kRedThreads];
    const int kout = diag ? na : na * nb;
    const int R = kRedThreads / kout, used = R * kout;
    const int t = threadIdx.x;
    double ax = 0.0, ay = 0.0;
    if (t < used) {
        const int o = t % kout, r = t / kout;
        const int ia = diag ? o : o / nb;
        const int ib = diag ? o : o - ia * nb;
        const int64_t step = int64_t(gridDim.x) * R;
        for (int64_t k0 = int64_t(blockIdx.x) * R + r; k0 < n_rows; k0 += kDotRows * step) {
            double2 u[kDotRows], v[kDotRows];
#pragma unroll
            for (int q = 0; q < kDotRows; ++q) {
                const int64_t k = k0 + q * step;
                u[q] = v[q] = make_double2(0.0, 0.0);
                if (k < n_rows) {
                    u[q] = A[k * na + ia];
                    v[q] = B[k * nb + ib];
                    if (w) {
                        const double wk = w[k];
                        u[q] = make_double2(wk * u[q].x, wk * u[q].y);
                    }
                }
            }
#pragma unroll
            for (int q = 0; q < kDotRows; ++q) {
                if (k0 + q * step >= n_rows) break;
                ax = fma(u[q].x, v[q].x, fma(u[q].y, v[q].y, ax));
                ay = fma(u[q].x, v[q].y, fma(-u[q].y, v[q].x, ay));
            }
        }
    }
    sx[t] = ax;
    sy[t] = ay;
    __syncthreads();
    for (int left = R; left > 1;) {   // tree over the rows of threads
        const int half = (left + 1) >> 1;
        if (t + half * kout < left * kout) {
            sx[t] += sx[t + half * kout];
            sy[t] += sy[t + half * kout];
        }
        __syncthreads();
        left = half;
    }
    if (t < kout) {
        partial[int64_t(blockIdx.x) * 2 * kout + 2 * t] = sx[t];
        partial[int64_t(blockIdx.x) * 2 * kout + 2 * t + 1] = sy[t];
    }
    if (!last_block_sum(partial, 2 * kout, counter, sx)) return;
    for (int o = t; o < kout; o += blockDim.x) out[o] = make_double2(sx[2 * o], sx[2 * o + 1]);
}

// Thread layout of the row-major [rows][n] vector kernels: thread t < n*R of a
// 256-thread block owns column p = t % n of rows r = t / n, r + R, ... within
// the block's row range (R = 256 / n), so consecutive threads touch
// consecutive elements and no element index is divided.
struct RowCol {
    int p, r, R;
    bool active;
    __device__ __forceinline__ RowCol(int n) {
        R = kRedThreads / n;
        active = int(threadIdx.x) < n * R;
        r = active ? int(threadIdx.x) / n : 0;
        p = active ? int(threadIdx.x) - r * n : 0;
    }
};

// Sums of v[0..cnt) over the block; the block's row partial[blockIdx][0..cnt)
// is written.  FP64 adds are the scarce resource on GB300, so for more than
// a few values the sums go through shared memory in chunks of 8 values
// (transposed: warp j sums value j of the chunk, 8 adds per lane and a 5-step
// shuffle) instead of a 5-step shuffle per value and thread: about 1.6 FP64
// adds per value and thread instead of 5.
template <int MAXV>
__device__ __forceinline__ void block_row_partial(double (&v)[MAXV], int cnt, double* __restrict__ partial) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if constexpr (MAXV < 4) {
        __shared__ double s_w[kRedThreads / 32][MAXV];
#pragma unroll
        for (int i = 0; i < MAXV; ++i) {
            if (i < cnt) {
                double x = v[i];
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
                if (lane == 0) s_w[warp][i] = x;
            }
        }
        __syncthreads();
        for (int i = threadIdx.x; i < cnt; i += blockDim.x) {
            double x = 0.0;
            for (int w = 0; w < kRedThreads / 32; ++w) x += s_w[w][i];
            partial[int64_t(blockIdx.x) * cnt + i] = x;
        }
    } else {
        static_assert(kRedThreads == 256, "the chunked block sum assumes 8 warps of 32");
        __shared__ double s_t[8][kRedThreads + 8];
        const int t = threadIdx.x;
#pragma unroll
        for (int c0 = 0; c0 < MAXV; c0 += 8) {
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (c0 + j < MAXV) s_t[j][t + (t >> 5)] = v[c0 + j];   // padded against bank conflicts
            __syncthreads();
            if (c0 + warp < cnt) {
                double x = 0.0;
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    const int src = lane * 8 + r;
                    x += s_t[warp][src + (src >> 5)];
                }
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
                if (lane == 0) partial[int64_t(blockIdx.x) * cnt + c0 + warp] = x;
            }
            __syncthreads();
        }
    }
}

// Projector overlaps of the precision form, S[a][b] = sum_k conj(A[k][a]) B[k][b]
// over interior rows from complex64 inputs (NO = n orbitals), added in FP64 into
// slot (block % kOvSlots) of slots[kOvSlots][2 NO^2] (re, im interleaved; the
// consumer sums the slots and clears them).  For even NO two threads share a
// row, each forming the products of half the rows a of S in FP32 registers
// (fewer registers, more rows in flight); the block sums its threads' values in
// FP32 over 8 segments of 32 threads (through shared memory, transposed) and
// the segment sums in FP64.  S is consumed in FP32 by the projector, and the
// FP64 work is per block, with no last-block pass.
constexpr int kOvSlots = 16;
template <int NO>
__global__ void __launch_bounds__(kRedThreads) overlap32_kernel(const float2* __restrict__ A,
                                                                const float2* __restrict__ B, int64_t n_rows,
                                                                double* __restrict__ slots) {
    constexpr int HS = NO % 2 == 0 ? 2 : 1;   // threads per row
    constexpr int NA = NO / HS;               // rows a of S per thread
    constexpr int CNT = 2 * NO * NO;          // values of S
    constexpr int CT = 2 * NA * NO;           // values per thread
    const int t = threadIdx.x;
    const int h = HS == 2 ? (t & 1) : 0;
    float f[CT];
#pragma unroll
    for (int i = 0; i < CT; ++i) f[i] = 0.f;
    const int rows_per_block = kRedThreads / HS;
#pragma unroll 2
    for (int64_t k = blockIdx.x * int64_t(rows_per_block) + t / HS; k < n_rows;
         k += int64_t(gridDim.x) * rows_per_block) {
        float2 a[NA], b[NO];
#pragma unroll
        for (int i = 0; i < NA; ++i) a[i] = A[k * NO + h * NA + i];
        if constexpr (NO % 2 == 0) {   // a row of B is NO/2 16-byte words
            const float4* B4 = reinterpret_cast<const float4*>(B + k * NO);
#pragma unroll
            for (int i = 0; i < NO / 2; ++i) {
                const float4 ub = B4[i];
                b[2 * i] = make_float2(ub.x, ub.y);
                b[2 * i + 1] = make_float2(ub.z, ub.w);
            }
        } else {
#pragma unroll
            for (int i = 0; i < NO; ++i) b[i] = B[k * NO + i];
        }
#pragma unroll
        for (int i = 0; i < NA; ++i)
#pragma unroll
            for (int j = 0; j < NO; ++j) {
                f[2 * (i * NO + j)] = fmaf(a[i].x, b[j].x, fmaf(a[i].y, b[j].y, f[2 * (i * NO + j)]));
                f[2 * (i * NO + j) + 1] = fmaf(a[i].x, b[j].y, fmaf(-a[i].y, b[j].x, f[2 * (i * NO + j) + 1]));
            }
    }
    static_assert(kRedThreads == 256, "the segment sums assume 8 warps of 32");
    __shared__ float s_t[32][kRedThreads + 1];   // a chunk of 32 values x 256 threads
    __shared__ float s_seg[8][32];
    const int lane = t & 31, seg = t >> 5;
    double* slot = slots + int64_t(blockIdx.x % kOvSlots) * CNT;
#pragma unroll
    for (int c0 = 0; c0 < CNT; c0 += 32) {
        // value c0 + j of S is this thread's f[c0 + j - h CT] when that index is its own
#pragma unroll
        for (int j = 0; j < 32; ++j) {
            if (c0 + j < CNT) {
                float v = 0.f;
                if (h == 0) {
                    if (c0 + j < CT) v = f[c0 + j < CT ? c0 + j : 0];
                } else {
                    if (c0 + j >= CT) v = f[c0 + j >= CT ? c0 + j - CT : 0];
                }
                s_t[j][t] = v;
            }
        }
        __syncthreads();
        if (c0 + lane < CNT) {   // value c0 + lane over the 32 threads of segment seg
            float x = 0.f;
#pragma unroll 8
            for (int r = 0; r < 32; ++r) x += s_t[lane][seg * 32 + r];
            s_seg[seg][lane] = x;
        }
        __syncthreads();
        if (t < 32 && c0 + t < CNT) {
            double x = 0.0;
#pragma unroll
            for (int g = 0; g < 8; ++g) x += widen_f32(s_seg[g][t]);
            atomicAdd(slot + c0 + t, x);
        }
        __syncthreads();
    }
}

// Krylov vectors are stored as integers (KrylovBasis below) and unscaled: V_0 is
// the substep's start vector and V_{i+1} the raw Gram-Schmidt remainder of the cell
// pass applied to V_i, with q_i = f[i] V_i, f[0] = 1 / beta, f[i] = f[i-1] / h_{i,i-1}
// (= 1 / |V_i|_M; 0 after a breakdown, h <= 1e-14 beta), so no pass over the basis
// only to scale it and no scaling of the new vector.  The pass that finishes
// V_i writes f[i] (and f[kScaleBeta] = beta); as a chain of float64 divisions by
// one thread of every block of every pass it took 6 us at 12 vectors.
constexpr int kScaleBeta = kMaxKrylov + 1;

// ------------------------------------------------- the Krylov basis in integers
// The Gram-Schmidt passes read every basis vector twice per new vector and are
// products and sums of float64 numbers, which run on the integer pipe
// (fixed64.cuh).  The vectors are therefore stored ready for it: per complex
// entry one exponent e (of its larger component) and per component the 64-bit
// integer X = v 2^(1082 - e), |X| < 2^60: 16 bytes, as the float64 pair was, and
// seven bits finer than float64 at the larger component.  Reading an entry then
// costs no conversion, only a shift to the scale of a sum: over the rows of a
// group (inner products, norms) that of the group's largest, over the vectors (a
// linear combination) that of the entry's own largest term, so that an entry
// is rounded on its own terms, as with float64, whatever its neighbours' size.
// Measured on 10 vectors of 775,009 x 4 (499 MB, 73 us at the copy rate): inner
// products with the projector 259 us as FP64 multiply-adds, 237 us converting
// from float64 on the way, 131 us stored as integers; the update 245 / 154 / 128
// us, the close of a substep 254 / 117 us.  (One exponent for the rows of a group
// took 127, 109 and 103 us, but rounded an entry on its group's largest.)
// Counters at 10 vectors of 508,385 x 4, two blocks of 256 threads per SM: inner
// products FP64 pipe 56 % busy (two conversions and two multiply-adds per group
// and vector), ALU 43 %, issue 46 %, DRAM 55 %, 72 instructions per entry and
// vector; update ALU 58 % (shifts, splits, carries), issue 54 %, DRAM 57 %, 85
// instructions.  No pipe is full: four warps a scheduler do not hide the latencies.

// Thread t < n R of a 256-thread block (R = 256 / n) owns column p = t % n and,
// in tile T, the rows T E R + r + R e (e < E, r = t / n): a group, the rows that
// one thread sums together, so that no thread waits for another's scale.  Storage
// follows the threads, not the rows: entry (T, e, t) of a vector, exponents (T, t),
// 16 bits each, the rows of a group in one or two words.  E (4, 2 or 1) is chosen per call so
// that the tiles fill the chip (krylov_rows).  Exponent 0: zero; 0x7FF: not finite.
constexpr int kFxNan = 0x7FF;
__host__ __device__ constexpr int exp_words(int E) { return (E + 1) / 2; }

__device__ __forceinline__ long long fx_re(int4 v) { return (static_cast<long long>(v.y) << 32) | unsigned(v.x); }
__device__ __forceinline__ long long fx_im(int4 v) { return (static_cast<long long>(v.w) << 32) | unsigned(v.z); }
__device__ __forceinline__ int4 fx_entry(long long re, long long im) {
    return make_int4(int(re), int(re >> 32), int(im), int(im >> 32));
}
// x 2^-d rounded down, for any d >= 0 (the instruction takes shifts beyond 63 as 64).
__device__ __forceinline__ long long shift_right(long long x, int d) {
    long long r;
    asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(d));
    return r;
}
// The exponents of a group's E rows.
template <int E>
__device__ __forceinline__ void read_exps(const int* p, int (&e)[E]) {
    if constexpr (E == 1) {
        e[0] = p[0];
    } else {
        int w[E / 2];
        if constexpr (E == 4) {
            const int2 v = *reinterpret_cast<const int2*>(p);
            w[0] = v.x;
            w[1] = v.y;
        } else {
            w[0] = p[0];
        }
#pragma unroll
        for (int r = 0; r < E; ++r) e[r] = (r & 1) ? int(unsigned(w[r / 2]) >> 16) : w[r / 2] & 0xFFFF;
    }
}
template <int E>
__device__ __forceinline__ void write_exps(int* p, const int (&e)[E]) {
    if constexpr (E == 4) *reinterpret_cast<int2*>(p) = make_int2(e[0] | (e[1] << 16), e[2] | (e[3] << 16));
    else if constexpr (E == 2) p[0] = e[0] | (e[1] << 16);
    else p[0] = e[0];
}
// An entry as float64.
__device__ __forceinline__ double2 fx_double2(int4 v, int e) {
    const double sc = e == kFxNan ? __hiloint2double(0x7FF80000, 0) : e == 0 ? 0.0 : ldexp(1.0, e - 1082);
    return make_double2(sc * double(fx_re(v)), sc * double(fx_im(v)));
}

struct TileRows {
    int p, r, R;
    bool active;
    __device__ __forceinline__ TileRows(int n) {
        R = kRedThreads / n;
        active = int(threadIdx.x) < n * R;
        r = active ? int(threadIdx.x) / n : 0;
        p = active ? int(threadIdx.x) - r * n : 0;
    }
};

// The basis vectors of a block's tiles as one stream of (tile, vector) items,
// item q = vector q % nv of the block's tile q / nv: each thread copies its own
// E rows of the item kStages - 1 ahead into its own slots of shared memory
// (cp.async, no barrier), so that about 50 KB per SM are in flight whatever the
// registers allow.  Loads into registers one vector ahead kept 32 KB in flight
// and ran at 4.5 TB/s.
__device__ __forceinline__ void copy16(void* smem_dst, const void* gmem_src) {
    const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(smem_dst));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gmem_src) : "memory");
}
template <int WORDS>
__device__ __forceinline__ void copy_exps(int* smem_dst, const int* gmem_src) {
    const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(smem_dst));
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(d), "l"(gmem_src), "n"(4 * WORDS) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int LEFT>
__device__ __forceinline__ void copy_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(LEFT) : "memory");
}

template <int E, int STAGES>
struct BasisStream {
    static constexpr int EW = exp_words(E);
    const int4* v;        // next item's first row
    const int* e;         // its exponents
    int4* slots;          // this thread's slots, [STAGES][E][kRedThreads]
    int* eslots;          // [STAGES][kRedThreads][EW] (STAGE_E)
    int64_t stride, estride, wrap, ewrap;   // to the next vector; from the last vector to the next tile's first
    int left, nv;         // tiles left, vectors
    int i, stage;
    __device__ __forceinline__ BasisStream(const KrylovBasis& B, int nv_, int4* sl, int* esl)
        : v(B.V + int64_t(blockIdx.x) * (E * kRedThreads) + threadIdx.x),
          e(B.e + (int64_t(blockIdx.x) * kRedThreads + threadIdx.x) * EW), slots(sl + threadIdx.x),
          eslots(esl + threadIdx.x * EW),
          stride(B.stride), estride(B.estride), wrap(int64_t(gridDim.x) * (E * kRedThreads) - (nv_ - 1) * B.stride),
          ewrap(int64_t(gridDim.x) * kRedThreads * EW - (nv_ - 1) * B.estride),
          left(int((B.tiles - blockIdx.x + gridDim.x - 1) / gridDim.x)), nv(nv_), i(0), stage(0) {}
    template <bool STAGE_E>
    __device__ __forceinline__ void issue() {
        if (left > 0) {
            int4* d = slots + stage * (E * kRedThreads);
#pragma unroll
            for (int r = 0; r < E; ++r) copy16(d + r * kRedThreads, v + r * kRedThreads);
            if (STAGE_E) copy_exps<EW>(eslots + stage * kRedThreads * EW, e);
            const bool last = ++i == nv;
            v += last ? wrap : stride;
            if (STAGE_E) e += last ? ewrap : estride;
            if (last) {
                i = 0;
                --left;
            }
        }
        copy_commit();
        stage = stage + 1 == STAGES ? 0 : stage + 1;
    }
};

// Gram-Schmidt inner products, with (MODE 1, 2) the projector pass of G in front:
//   MODE 0: w = V_nv, the stored remainder of the first pass (second pass;
//     skipped when gate && !*gate);
//   MODE 1: z is the FP64 cell pass applied to V_{nv-1}, and
//     w[k][p] = ML^-1[k] z[k][p] - sum_j phi[k][j] S[j][p] on interior rows
//     (0 on the others), which is G q_{nv-1} / s_f[nv-1], is written to wd;
//   MODE 2: the same for the precision form, the projector in FP32 from the
//     complex64 cell-pass output and orbitals; w is a complex64 vector (times
//     2^kv, see below) and replaces the cell pass's output in place.
// out[i] = s_f[i] fw sum_k m_k conj(V_i) w = <q_i, fw w>_M for i < nv with
// fw = s_f[nv-1], and out[nv] = (sum_i |out[i]|^2, 0), the squared norm of the
// part of fw w in the span of q_0..q_{nv-1}: by Pythagoras the norm before the
// update is this plus the norm that the update leaves, which is how the
// re-orthogonalisation test uses it.
//
// A thread forms m w of its E rows on their common scale and walks the basis
// vectors: E staged rows, shifted to the vector's largest of them, 12 E IMAD.WIDE
// and two float64 additions into its sums in shared memory.
struct GsDotsArgs {
    const double2* z;
    float2* z32;
    const double2* phi;
    const float2* phi32;
    const double2* S;
    double* S_slots;        // MODE 2: overlap32_kernel's slots (cleared by the last block), or null
    const double* ml_inv;
    const float* ml_inv32;
    const double* ml;
    int64_t n_int, N;
    int n;
    double2* wd;
    KrylovBasis B;
    int nv;
    const int* gate;
    const double* f;        // the basis's scales
    double* partial;
    unsigned* counter;
    double2* out;
};

template <int E, int MODE, int STAGES>
__global__ void __launch_bounds__(kRedThreads, 2) gs_dots_kernel(const __grid_constant__ GsDotsArgs a) {
    if (MODE == 0 && a.gate && *a.gate == 0) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double2* s_acc = reinterpret_cast<double2*>(smem_raw);                  // [nv][kRedThreads]
    int4* s_v = reinterpret_cast<int4*>(s_acc + a.nv * kRedThreads);       // [STAGES][E][kRedThreads]
    int* s_ve = reinterpret_cast<int*>(s_v + STAGES * E * kRedThreads);    // [STAGES][kRedThreads][EW]
    constexpr int EW = exp_words(E);
    __shared__ double s_f[kMaxKrylov];
    __shared__ double2 s_S[MODE == 1 ? kMaxOrbProj * kMaxOrbProj : 1];
    __shared__ float2 s_S32[MODE == 2 ? kMaxOrbProj * kMaxOrbProj : 1];
    const int nv = a.nv, n = a.n, tid = threadIdx.x;
    for (int i = 0; i < nv; ++i) s_acc[i * kRedThreads + tid] = make_double2(0.0, 0.0);
    if constexpr (MODE == 1)
        for (int i = tid; i < n * n; i += blockDim.x) s_S[i] = a.S[i];
    if constexpr (MODE == 2) {
        // the overlaps: the sum of overlap32_kernel's slots, or S itself (zero
        // without the projector)
        for (int i = tid; i < n * n; i += blockDim.x) {
            double2 v = make_double2(0.0, 0.0);
            if (a.S_slots) {
                for (int sl = 0; sl < kOvSlots; ++sl) {
                    v.x += a.S_slots[sl * 2 * n * n + 2 * i];
                    v.y += a.S_slots[sl * 2 * n * n + 2 * i + 1];
                }
            } else {
                v = a.S[i];
            }
            s_S32[i] = make_float2(narrow_f64(v.x), narrow_f64(v.y));
        }
    }
    if (tid < nv) s_f[tid] = a.f[tid];
    __syncthreads();
    // MODE 2: the complex64 input of the cell pass was 2^kv V_{nv-1}
    // (gs_combine_kernel's scaling; V_0 unscaled), so the raw vector is the
    // result times 2^-kv
    const int kv = (MODE == 2 && nv >= 2 && s_f[nv - 2] > 0.0) ? ilogb(s_f[nv - 2]) : 0;
    const TileRows rc(n);
    if (rc.active) {
        const int p = rc.p;
        BasisStream<E, STAGES> st(a.B, nv, s_v, s_ve);
#pragma unroll
        for (int q = 0; q < STAGES - 1; ++q) st.template issue<true>();
        int slot = 0;
        const int n_int = int(a.n_int);
        for (int64_t tile = blockIdx.x; tile < a.B.tiles; tile += gridDim.x) {
            const int k0 = int(tile) * (E * rc.R) + rc.r;
            double2 x[E];
            int kr[E];   // the rows (row 0 in place of those without a part in the sums, whose m w is 0)
            unsigned xe = 0u;
#pragma unroll
            for (int r = 0; r < E; ++r) {
                kr[r] = k0 + r * rc.R < n_int ? k0 + r * rc.R : 0;
                x[r] = make_double2(0.0, 0.0);
            }
            if constexpr (MODE == 0) {
                int e[E];
                read_exps<E>(a.B.e + nv * a.B.estride + (tile * kRedThreads + tid) * EW, e);
#pragma unroll
                for (int r = 0; r < E; ++r)
                    if (k0 + r * rc.R < n_int)
                        x[r] = fx_double2(a.B.V[nv * a.B.stride + (tile * E + r) * kRedThreads + tid], e[r]);
            }
            if constexpr (MODE == 1) {
                double2 zo[E];
                double s[E];
#pragma unroll
                for (int r = 0; r < E; ++r) {
                    s[r] = a.ml_inv[kr[r]];
                    zo[r] = a.z[unsigned(kr[r]) * unsigned(n) + unsigned(p)];
                }
#pragma unroll
                for (int r = 0; r < E; ++r) x[r] = make_double2(zo[r].x * s[r], zo[r].y * s[r]);
                for (int j = 0; j < n; ++j) {
                    const double2 c = s_S[j * n + p];
                    double2 f[E];
#pragma unroll
                    for (int r = 0; r < E; ++r) f[r] = a.phi[unsigned(kr[r]) * unsigned(n) + unsigned(j)];
#pragma unroll
                    for (int r = 0; r < E; ++r) {
                        x[r].x = fma(-f[r].x, c.x, fma(f[r].y, c.y, x[r].x));
                        x[r].y = fma(-f[r].x, c.y, fma(-f[r].y, c.x, x[r].y));
                    }
                }
            }
            if constexpr (MODE == 2) {
                float2 xf[E];
                float s[E];
                const float2* pr[E];
#pragma unroll
                for (int r = 0; r < E; ++r) {
                    s[r] = a.ml_inv32[kr[r]];
                    xf[r] = a.z32[unsigned(kr[r]) * unsigned(n) + unsigned(p)];
                    pr[r] = a.phi32 + unsigned(kr[r]) * unsigned(n);
                }
                float2 f[4][E];   // four orbitals of the rows in flight
#pragma unroll
                for (int j0 = 0; j0 < kMaxOrbProj; j0 += 4) {
                    if (j0 >= n) break;
#pragma unroll
                    for (int j = 0; j < 4; ++j)
#pragma unroll
                        for (int r = 0; r < E; ++r)
                            if (j0 + j < n) f[j][r] = pr[r][j0 + j];
                    if (j0 == 0) {
#pragma unroll
                        for (int r = 0; r < E; ++r) xf[r] = make_float2(xf[r].x * s[r], xf[r].y * s[r]);
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        if (j0 + j < n) {
                            const float2 c = s_S32[(j0 + j) * n + p];
#pragma unroll
                            for (int r = 0; r < E; ++r) {
                                xf[r].x = fmaf(-f[j][r].x, c.x, fmaf(f[j][r].y, c.y, xf[r].x));
                                xf[r].y = fmaf(-f[j][r].x, c.y, fmaf(-f[j][r].y, c.x, xf[r].y));
                            }
                        }
                    }
                }
#pragma unroll
                for (int r = 0; r < E; ++r) {
                    x[r] = make_double2(widen_f32_scaled(xf[r].x, -kv), widen_f32_scaled(xf[r].y, -kv));
                    if (k0 + r * rc.R < n_int) a.z32[unsigned(kr[r]) * unsigned(n) + unsigned(p)] = xf[r];
                }
            }
#pragma unroll
            for (int r = 0; r < E; ++r) {
                const int k = k0 + r * rc.R;
                const bool in = k < n_int;
                if (!in) x[r] = make_double2(0.0, 0.0);
                if (MODE == 1 && k < int(a.N)) a.wd[unsigned(k) * unsigned(n) + unsigned(p)] = x[r];
                const double m = in ? a.ml[k] : 0.0;
                x[r] = make_double2(m * x[r].x, m * x[r].y);
                xe = max(xe, max(fx_expbits(x[r].x), fx_expbits(x[r].y)));
            }
            const int ex = max(int(xe >> 20), kFxMinExp);
            Fx X[E], Y[E], nX[E];
#pragma unroll
            for (int r = 0; r < E; ++r) {
                X[r] = fx_make(x[r].x, ex);
                Y[r] = fx_make(x[r].y, ex);
                nX[r] = fx_neg(X[r]);
            }
            for (int i = 0; i < nv; ++i) {
                copy_wait<STAGES - 2>();
                int4 u[E];
#pragma unroll
                for (int r = 0; r < E; ++r) u[r] = s_v[(slot * E + r) * kRedThreads + tid];
                int er[E], eu = 0;
                read_exps<E>(s_ve + (slot * kRedThreads + tid) * EW, er);
                if (k0 + (E - 1) * rc.R >= n_int) {   // surface rows (m w = 0) may hold anything
#pragma unroll
                    for (int r = 0; r < E; ++r)
                        if (k0 + r * rc.R >= n_int) er[r] = 0;
                }
#pragma unroll
                for (int r = 0; r < E; ++r) eu = max(eu, er[r]);
                slot = slot + 1 == STAGES ? 0 : slot + 1;
                st.template issue<true>();
                FxAcc re{0, 0}, im{0, 0};
#pragma unroll
                for (int r = 0; r < E; ++r) {
                    const int d = eu - er[r];
                    const Fx ur = fx_split(shift_right(fx_re(u[r]), d)), ui = fx_split(shift_right(fx_im(u[r]), d));
                    fx_mad(re, ur, X[r]);
                    fx_mad(re, ui, Y[r]);
                    fx_mad(im, ur, Y[r]);
                    fx_mad(im, ui, nX[r]);
                }
                const double sc = fx_scale((eu == kFxNan || xe == kFxExpMask) ? 0x7FFFFF : eu + ex);
                double2 acc = s_acc[i * kRedThreads + tid];
                acc.x = fma(fx_value(re), sc, acc.x);
                acc.y = fma(fx_value(im), sc, acc.y);
                s_acc[i * kRedThreads + tid] = acc;
            }
        }
    }
    // block sums: warp j sums the 256 values of vectors j, j + 8, ..
    __syncthreads();
    {
        const int lane = tid & 31, warp = tid >> 5;
        for (int i = warp; i < nv; i += kRedThreads / 32) {
            double2 v = make_double2(0.0, 0.0);
#pragma unroll
            for (int r = 0; r < kRedThreads / 32; ++r) {
                const double2 t = s_acc[i * kRedThreads + 32 * r + lane];
                v.x += t.x;
                v.y += t.y;
            }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                v.x += __shfl_xor_sync(0xffffffffu, v.x, off);
                v.y += __shfl_xor_sync(0xffffffffu, v.y, off);
            }
            if (lane == 0) {
                a.partial[int64_t(blockIdx.x) * 2 * nv + 2 * i] = v.x;
                a.partial[int64_t(blockIdx.x) * 2 * nv + 2 * i + 1] = v.y;
            }
        }
    }
    __shared__ double s_sum[kRedThreads];
    if (!last_block_sum(a.partial, 2 * nv, a.counter, s_sum)) return;
    const double fw = s_f[nv - 1];
    if (tid < 32) {
        double nn = 0.0;
        if (tid < nv) {
            const double f = s_f[tid] * fw;
            const double2 o = make_double2(f * s_sum[2 * tid], f * s_sum[2 * tid + 1]);
            a.out[tid] = o;
            nn = o.x * o.x + o.y * o.y;
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) nn += __shfl_xor_sync(0xffffffffu, nn, off);
        if (tid == 0) a.out[nv] = make_double2(nn, 0.0);
    }
    if (MODE == 2 && a.S_slots)
        for (int o = tid; o < kOvSlots * 2 * n * n; o += blockDim.x) a.S_slots[o] = 0.0;
}

// Linear combinations of the basis, x = base + sum_{i<nv} c_i V_i, stored as a
// basis vector with its norm:
//   KIND 0 opens the first substep: x = src, to V_0;
//   KIND 1 closes a substep and opens the next: x = scale sum y_i q_i, to out
//     (phi after the substep; when non-null) and V_0;
//   KIND 2 is the Gram-Schmidt update of the raw vector w of gs_dots_kernel (the
//     true vector is fw w with fw = s_f[nv-1]): fw w -= sum c_i q_i, i.e.
//     w -= sum (c_i s_f[i] / fw) V_i on interior rows (0 on the others), to V_nv;
//   KIND 4 is the same in the precision form, from the complex64 raw vector;
//   KIND 3 is the second such pass, on V_nv itself (skipped when !*gate).
// vd (FP64 form) and v32 (precision form) receive the float64 / complex64 copy
// of x that the next cell pass reads.  The last block writes beta2_out =
// |x|_M^2 over interior rows (KIND 0, 1), or the Hessenberg column (KIND 2..4):
// Hcol[i] = c_i (KIND 3: += c_i), Hcol[nv] = fw |w|_M, and (KIND 2, 4) *reorth = 1
// when the pass left |fw w|^2 < eta2 (c[nv] + |fw w|^2), the squared norm before
// it (c[nv] is its part in the span of the basis), and the new scale (every block
// reads the scales at its start, the last block writes after all others have
// finished); V_0 is written tile by tile after the tile's reads.
//
// A thread brings each of its rows to the scale of the row's largest term c_i e_i
// by shifting the entries; an entry then costs its 16 bytes and 12 IMAD.WIDE per
// vector, against 4 FP64 multiply-add slots of 64 lanes before.  The result keeps
// 58 bits below its largest term or the base and is shifted to its own exponent;
// its squares for the norm are integer products too, on the scale of the group's
// largest, rounded to float64 once per row.
struct GsCombineArgs {
    KrylovBasis B;
    int nv;
    const double2* c;       // KIND 1: y; KIND 2, 3: inner products
    double scale;           // KIND 1
    const double2* src;     // KIND 0
    const double2* wd;      // KIND 2: the raw vector, float64 form
    const float2* w32;      // KIND 4: the raw vector times 2^kv, precision form
    const double* ml;
    int64_t n_int, N;
    int n;
    const int* gate;
    double eta2;
    int* reorth;
    double* f;              // the basis's scales
    double2* out;
    double2* vd;
    float2* v32;
    double* partial;
    unsigned* counter;
    double2* Hcol;
    double2* beta2_out;
};

// f 2^32 times its own scale over 2^s: the 24-bit significand at bit 32, shifted
// right by s - e (e the biased exponent of f), with its sign.
__device__ __forceinline__ long long float_int(float f, int s) {
    const unsigned u = __float_as_uint(f);
    const int e = int((u >> 23) & 0xFFu);
    const unsigned long long m = e == 0 ? 0ull : static_cast<unsigned long long>((u & 0x7FFFFFu) | 0x800000u) << 32;
    const unsigned long long v = m >> min(s - e, 63);
    return int(u) < 0 ? -static_cast<long long>(v) : static_cast<long long>(v);
}

template <int E, int KIND, int STAGES>
__global__ void __launch_bounds__(kRedThreads, 2) gs_combine_kernel(const __grid_constant__ GsCombineArgs a) {
    if (KIND == 3 && *a.gate == 0) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int4* s_v = reinterpret_cast<int4*>(smem_raw);                                   // [stages][E][kRedThreads]
    int* s_ge = reinterpret_cast<int*>(s_v + STAGES * E * kRedThreads);     // [2][nv][kRedThreads][EW]
    constexpr int EW = exp_words(E);
    __shared__ double s_f[kMaxKrylov];
    __shared__ double2 s_c[kMaxKrylov + 1];
    __shared__ int4 s_ci[kMaxKrylov];        // coefficients, integers on their own scale (re l, re h, im l, im h)
    __shared__ int s_ce[kMaxKrylov];         // their biased exponents
    __shared__ int s_low;                    // smallest admissible term exponent (kFxMaxSum + 1: NaN)
    const int nv = a.nv, n = a.n, tid = threadIdx.x;
    double fw = 1.0;
    int kw = 0, kv = 0;
    if constexpr (KIND != 0) {
        if (tid < nv) s_f[tid] = a.f[tid];
        if (tid <= (KIND == 1 ? nv - 1 : nv)) s_c[tid] = a.c[tid];
        __syncthreads();
        if constexpr (KIND >= 2) {
            fw = s_f[nv - 1];
            // the complex64 copy holds 2^kw w with 2^kw ~ fw, i.e. about the true
            // vector fw w (whose size is the Hessenberg entry): the raw vectors
            // grow like the operator norm to the power of their index and would
            // leave the binary32 range (gs_dots_kernel undoes the factor)
            kw = fw > 0.0 ? ilogb(fw) : 0;
            if (nv >= 2 && s_f[nv - 2] > 0.0) kv = ilogb(s_f[nv - 2]);   // the cell pass's factor 2^kv in w32
        }
        if (tid < nv) {
            const double f = KIND == 1 ? a.scale * s_f[tid] : fw > 0.0 ? -s_f[tid] / fw : 0.0;
            const double2 c = make_double2(f * s_c[tid].x, f * s_c[tid].y);
            const int e = int(max(fx_expbits(c.x), fx_expbits(c.y)) >> 20);
            s_ce[tid] = e;
            const Fx re = fx_split(e ? fx_int(c.x, e) : 0), im = fx_split(e ? fx_int(c.y, e) : 0);
            s_ci[tid] = make_int4(re.l, re.h, im.l, im.h);
        }
        __syncthreads();
        if (tid == 0) {
            int m = 1023;
            bool bad = false;
            for (int i = 0; i < nv; ++i) {
                m = max(m, s_ce[i]);
                bad = bad || s_ce[i] == 0x7FF;
            }
            s_low = bad ? kFxMaxSum + 1 : m + kFxMinExp;
        }
        __syncthreads();
    }
    const TileRows rc(n);
    const int p = rc.p;
    double nrm[1] = {0.0};
    // the exponents of this and the next tile, staged like the vectors
    auto copy_e = [&](int64_t tile, int par) {
        if (tile < a.B.tiles)
            for (int i = 0; i < nv; ++i)
                copy_exps<EW>(s_ge + ((par * nv + i) * kRedThreads + tid) * EW,
                              a.B.e + i * a.B.estride + (tile * kRedThreads + tid) * EW);
    };
    BasisStream<E, STAGES> st(a.B, nv, s_v, s_ge);
    if (KIND != 0 && rc.active) {
        copy_e(blockIdx.x, 0);   // complete with the first item
#pragma unroll
        for (int q = 0; q < STAGES - 1; ++q) st.template issue<false>();
    }
    int slot = 0, par = 0;
    const int N = int(a.N), n_int = int(a.n_int);
    const int rows = KIND >= 2 ? n_int : N;   // rows of the result; zero beyond
    for (int64_t tile = blockIdx.x; rc.active && tile < a.B.tiles; tile += gridDim.x, par ^= 1) {
        int* eg = a.B.e + (tile * kRedThreads + tid) * EW;
        const int k0 = int(tile) * (E * rc.R) + rc.r;
        unsigned o[E];
        long long tx[E], ty[E];
        float2 bf[E];    // the base and the masses: loaded ahead of the walk
        double mass[E];
#pragma unroll
        for (int r = 0; r < E; ++r) {
            const int k = k0 + r * rc.R;
            o[r] = unsigned(k < N ? k : 0) * unsigned(n) + unsigned(p);
            tx[r] = ty[r] = 0;
            mass[r] = k < n_int ? a.ml[k] : 0.0;
            bf[r] = make_float2(0.f, 0.f);
            if (KIND == 4 && k < n_int) bf[r] = a.w32[o[r]];
        }
        int EM[E];       // the rows' scales
#pragma unroll
        for (int r = 0; r < E; ++r) EM[r] = KIND == 0 ? 1023 + kFxMinExp : s_low;
        if constexpr (KIND != 0) {
            // this tile's exponents came with an item at least nv before its own
            if (tile == blockIdx.x) copy_wait<STAGES - 2>();
            else if (nv < STAGES) copy_wait<0>();
            const int* ge = s_ge + (par * nv * kRedThreads + tid) * EW;
            unsigned bad = 0u;
#pragma unroll 4
            for (int i = 0; i < nv; ++i) {
                int e[E];
                read_exps<E>(ge + i * kRedThreads * EW, e);
                const int ce = s_ce[i];
#pragma unroll
                for (int r = 0; r < E; ++r) {
                    if (e[r] == kFxNan) bad |= 1u << r;
                    EM[r] = max(EM[r], e[r] + ce);
                }
            }
            copy_e(tile + gridDim.x, par ^ 1);   // in the next item's group
            FxAcc ax[E], ay[E];
#pragma unroll
            for (int r = 0; r < E; ++r) ax[r] = ay[r] = FxAcc{0, 0};
            for (int i = 0; i < nv; ++i) {
                int e[E];
                read_exps<E>(ge + i * kRedThreads * EW, e);
                const int ce = s_ce[i];
                const int4 c4 = s_ci[i];
                const Fx re{c4.y, c4.x}, im{c4.w, c4.z}, nim = fx_neg(im);
                copy_wait<STAGES - 2>();
                int4 u[E];
#pragma unroll
                for (int r = 0; r < E; ++r) u[r] = s_v[(slot * E + r) * kRedThreads + tid];
                slot = slot + 1 == STAGES ? 0 : slot + 1;
                st.template issue<false>();
#pragma unroll
                for (int r = 0; r < E; ++r) {
                    const int sh = EM[r] - e[r] - ce;
                    const Fx ur = fx_split(shift_right(fx_re(u[r]), sh)), ui = fx_split(shift_right(fx_im(u[r]), sh));
                    fx_mad(ax[r], re, ur);
                    fx_mad(ax[r], nim, ui);
                    fx_mad(ay[r], re, ui);
                    fx_mad(ay[r], im, ur);
                }
                if (i & 1) {   // two vectors (4 products) between carries
#pragma unroll
                    for (int r = 0; r < E; ++r) {
                        fx_carry(ax[r]);
                        fx_carry(ay[r]);
                    }
                }
            }
#pragma unroll
            for (int r = 0; r < E; ++r) {
                if (bad & (1u << r)) EM[r] = kFxMaxSum + 1;
                tx[r] = (ax[r].hh << 1) + (ax[r].x >> 31);
                ty[r] = (ay[r].hh << 1) + (ay[r].x >> 31);
            }
        }
        if constexpr (KIND == 4) {   // the base: 24 bits at 2^56 of the scale EM
#pragma unroll
            for (int r = 0; r < E; ++r) {
                const unsigned be = max(__float_as_uint(bf[r].x) & 0x7F800000u, __float_as_uint(bf[r].y) & 0x7F800000u);
                const int eb = max(int(be >> 23) + 896 - kv, kFxMinExp);
                const int up = max(EM[r], eb + 1023), d = min(up - EM[r], 63);
                tx[r] = (tx[r] >> d) + float_int(bf[r].x, up - 1919 + kv);
                ty[r] = (ty[r] >> d) + float_int(bf[r].y, up - 1919 + kv);
                EM[r] = (EM[r] > kFxMaxSum || be == 0x7F800000u || eb >= kFxNan) ? kFxMaxSum + 1 : up;
            }
        } else if constexpr (KIND != 1) {   // the base: 53 bits at 2^56 of the scale EM
            double2 b[E];
            int e3[E];
            if constexpr (KIND == 3) read_exps<E>(eg + nv * a.B.estride, e3);
#pragma unroll
            for (int r = 0; r < E; ++r) {
                b[r] = make_double2(0.0, 0.0);
                if (k0 + r * rc.R < rows) {
                    if constexpr (KIND == 0) b[r] = a.src[o[r]];
                    if constexpr (KIND == 2) b[r] = a.wd[o[r]];
                    if constexpr (KIND == 3)
                        b[r] = fx_double2(a.B.V[nv * a.B.stride + (tile * E + r) * kRedThreads + tid], e3[r]);
                }
            }
#pragma unroll
            for (int r = 0; r < E; ++r) {
                const unsigned be = max(fx_expbits(b[r].x), fx_expbits(b[r].y));
                const int eb = max(int(be >> 20), kFxMinExp);
                const int up = max(EM[r], eb + 1023), d = min(up - EM[r], 63);
                const int es = min(up - 1023, 8000);   // b 2^(2101 - up) = (b 2^(1082 - es)) / 16 for es = up - 1023
                tx[r] = (tx[r] >> d) + (fx_int(b[r].x, es) >> 4);
                ty[r] = (ty[r] >> d) + (fx_int(b[r].y, es) >> 4);
                EM[r] = (EM[r] > kFxMaxSum || be == kFxExpMask) ? kFxMaxSum + 1 : up;
            }
        }
        const int dst = KIND <= 1 ? 0 : nv;
        int eo[E], top = 0;   // the rows' new exponents, the group's largest
        double n2 = 0.0;
#pragma unroll
        for (int r = 0; r < E; ++r) {
            if (k0 + r * rc.R >= rows) tx[r] = ty[r] = 0;
            const int bits = 64 - __clzll(static_cast<long long>((tx[r] ^ (tx[r] >> 63)) | (ty[r] ^ (ty[r] >> 63))));
            // |x| <= 2^(bits + EM - 2101) (t = -1 alone: bits = 0)
            eo[r] = bits ? bits + EM[r] - 1079 : 0;
            if (EM[r] > kFxMaxSum || eo[r] > kFxNan) eo[r] = kFxNan;
            if (eo[r] < kFxMinExp) eo[r] = 0;
            if (k0 + r * rc.R < n_int) top = max(top, eo[r]);   // (surface rows have no part in the norm)
            // t 2^(EM - 2101) = X 2^(eo - 1082), X = t 2^(60 - bits)
            const long long vx = eo[r] != 0 ? (tx[r] << (63 - bits)) >> 3 : 0, vy = eo[r] != 0 ? (ty[r] << (63 - bits)) >> 3 : 0;
            if (k0 + r * rc.R < N) {
                a.B.V[dst * a.B.stride + (tile * E + r) * kRedThreads + tid] = fx_entry(vx, vy);
                if ((KIND == 1 && a.out) || a.vd) {
                    const double sc = fx_scale(EM[r]);
                    const double2 v = make_double2(__ll2double_rn(tx[r]) * sc, __ll2double_rn(ty[r]) * sc);
                    if (KIND == 1 && a.out) a.out[o[r]] = v;
                    if (a.vd) a.vd[o[r]] = v;
                }
                if (a.v32) a.v32[o[r]] = make_float2(fx_to_f32(vx, eo[r] - 1082 + kw), fx_to_f32(vy, eo[r] - 1082 + kw));
            }
            tx[r] = vx;
            ty[r] = vy;
        }
        write_exps<E>(eg + dst * a.B.estride, eo);
#pragma unroll
        for (int r = 0; r < E; ++r) {
            const int d = min(max(top - eo[r], 0), 63);
            const Fx fx = fx_split(tx[r] >> d), fy = fx_split(ty[r] >> d);
            FxAcc sq{0, 0};
            fx_mad(sq, fx, fx);
            fx_mad(sq, fy, fy);
            n2 = fma(mass[r], fx_value(sq), n2);
        }
        nrm[0] = fma(n2, top == kFxNan ? __hiloint2double(0x7FF80000, 0) : fx_scale(2 * top), nrm[0]);
    }
    __syncthreads();
    block_row_partial<1>(nrm, 1, a.partial);
    __shared__ double s_sum[kRedThreads];
    if (!last_block_sum(a.partial, 1, a.counter, s_sum)) return;
    if (tid == 0) {
        if constexpr (KIND <= 1) {
            const double b2 = fmax(s_sum[0], 0.0), beta = sqrt(b2);
            *a.beta2_out = make_double2(b2, 0.0);
            a.f[0] = beta > 0.0 ? 1.0 / beta : 0.0;
            a.f[kScaleBeta] = beta;
        } else {
            for (int i = 0; i < nv; ++i) {
                const double2 h = KIND == 3 ? make_double2(a.Hcol[i].x + s_c[i].x, a.Hcol[i].y + s_c[i].y) : s_c[i];
                a.Hcol[i] = h;
            }
            const double nn = fw * fw * fmax(s_sum[0], 0.0);   // |fw w|^2
            const double h = sqrt(nn);
            a.Hcol[nv] = make_double2(h, 0.0);
            a.f[nv] = (h > 1e-14 * a.f[kScaleBeta] && h > 0.0) ? fw / h : 0.0;
            // |fw w|^2 before the update = in-span part (c[nv]) + what is left (nn)
            if (KIND != 3) *a.reorth = nn < a.eta2 * (s_c[nv].x + nn) ? 1 : 0;
        }
    }
}

// exp(-i dt H) (imag: exp(-dt H), the imaginary-time step) for an m x m
// complex matrix (m <= kMaxKrylov) by one block: scaling and squaring with a
// truncated Taylor series (the scaled matrix has 1-norm <= 1/2; the remainder
// after 16 terms is below 0.5^17 / 17! ~ 2e-20 relative, under the FP64
// rounding of the squarings).  The series is summed by powers of A^4
// (Paterson and Stockmeyer): 6 matrix products instead of 16, of which each
// takes about 2 m^3 clocks of the SM's FP64 pipe, and two threads share an
// entry's sum.  One ladder of 64 candidates: 68 us at m = 10 and 96 us at m = 12
// term by term; now 28 and 39 us.
constexpr int kTaylorTerms = 16;
constexpr int kExpmThreads = 2 * kMaxKrylov * kMaxKrylov;

// O = X Y + add (add may be null) by pairs of threads; the caller synchronises
// before O is read and before X, Y change.  O may alias add but not X or Y.
__device__ __forceinline__ void block_matmul(const double2* X, const double2* Y, double2* O, const double2* add, int m) {
    const int t = threadIdx.x, o = t >> 1, half = t & 1;
    double x = 0.0, y = 0.0;
    if (o < m * m) {
        const int i = o % m, j = o / m;
#pragma unroll 4
        for (int l = half; l < m; l += 2) {
            const double2 a = X[l * m + i], b = Y[j * m + l];
            x = fma(a.x, b.x, fma(-a.y, b.y, x));
            y = fma(a.x, b.y, fma(a.y, b.x, y));
        }
    }
    x += __shfl_xor_sync(0xffffffffu, x, 1);
    y += __shfl_xor_sync(0xffffffffu, y, 1);
    if (o < m * m && half == 0) {
        if (add) {
            x += add[o].x;
            y += add[o].y;
        }
        O[o] = make_double2(x, y);
    }
}

// H: column-major with leading dimension ldh.  Returns the matrix of the result
// (S or T).  A, A2, A3, A4, S, T: m x m in shared memory.
__device__ double2* block_expm(const double2* __restrict__ H, int ldh, int m, double dt, int imag, double2* A,
                               double2* A2, double2* A3, double2* A4, double2* S, double2* T) {
    __shared__ int s_sq;
    const int t = threadIdx.x;
    const int mm = m * m;
    for (int o = t; o < mm; o += blockDim.x) {
        const int i = o % m, j = o / m;
        const double2 h = H[j * ldh + i];
        A[o] = imag ? make_double2(-dt * h.x, -dt * h.y)    // -dt h
                    : make_double2(dt * h.y, -dt * h.x);    // -i dt h
    }
    __syncthreads();
    // 1-norm: column sums by m threads (each in row order), then their maximum
    __shared__ double s_col[kMaxKrylov];
    if (t < m) {
        double c = 0.0;
        for (int i = 0; i < m; ++i) c += hypot(A[t * m + i].x, A[t * m + i].y);
        s_col[t] = c;
    }
    __syncthreads();
    if (t == 0) {
        double nrm = 0.0;
        for (int j = 0; j < m; ++j) nrm = fmax(nrm, s_col[j]);
        int sq = 0;
        while (nrm > 0.5 && sq < 60) {
            nrm *= 0.5;
            ++sq;
        }
        s_sq = sq;
    }
    __syncthreads();
    const double sc = ldexp(1.0, -s_sq);
    for (int o = t; o < mm; o += blockDim.x) {
        A[o].x *= sc;
        A[o].y *= sc;
    }
    __syncthreads();
    block_matmul(A, A, A2, nullptr, m);
    __syncthreads();
    block_matmul(A2, A, A3, nullptr, m);
    block_matmul(A2, A2, A4, nullptr, m);
    __syncthreads();
    // S = sum_{k<=16} A^k / k! = B0 + A4 (B1 + A4 (B2 + A4 (B3 + A4 / 16!))),
    // B_q = sum_{r<4} A^r / (4 q + r)!
    double f[kTaylorTerms + 1];
    f[0] = 1.0;
#pragma unroll
    for (int k = 1; k <= kTaylorTerms; ++k) f[k] = f[k - 1] / k;
    auto block_poly = [&](int q, double2* out, bool top) {   // B_q (+ A4 / 16! for the top one)
        for (int o = t; o < mm; o += blockDim.x) {
            const double2 a = A[o], a2 = A2[o], a3 = A3[o], a4 = A4[o];
            double2 v = make_double2(fma(f[4 * q + 1], a.x, fma(f[4 * q + 2], a2.x, f[4 * q + 3] * a3.x)),
                                     fma(f[4 * q + 1], a.y, fma(f[4 * q + 2], a2.y, f[4 * q + 3] * a3.y)));
            if (top) {
                v.x = fma(f[16], a4.x, v.x);
                v.y = fma(f[16], a4.y, v.y);
            }
            if (o % m == o / m) v.x += f[4 * q];
            out[o] = v;
        }
    };
    double2 *P = S, *Q = T;
    block_poly(3, P, true);
#pragma unroll
    for (int q = 2; q >= 0; --q) {
        block_poly(q, Q, false);
        __syncthreads();
        block_matmul(A4, P, Q, Q, m);
        __syncthreads();
        double2* n = P;
        P = Q;
        Q = n;
    }
    for (int q = 0; q < s_sq; ++q) {
        block_matmul(P, P, Q, nullptr, m);
        __syncthreads();
        double2* n = P;
        P = Q;
        Q = n;
    }
    return P;
}

struct TauLadder {
    double tau[kLadder];
};

// Block c evaluates E_c = exp(-i tau_c H_m) (imag: exp(-tau_c H_m)): writes
// its first column to col[c][0..m) and err[c].x = |h_{m+1,m}| |E_c[m-1][0]|
// (the error estimate divided by beta; 0 when exact is set, i.e. after a
// breakdown).
__global__ void __launch_bounds__(kExpmThreads) expm_ladder_kernel(const double2* __restrict__ H, int ldh, int m, TauLadder taus, int exact,
                                   int imag, double2* __restrict__ col, double2* __restrict__ err) {
    __shared__ double2 s_m[6][kMaxKrylov * kMaxKrylov];
    const int c = blockIdx.x;
    const double2* S = block_expm(H, ldh, m, taus.tau[c], imag, s_m[0], s_m[1], s_m[2], s_m[3], s_m[4], s_m[5]);
    for (int i = threadIdx.x; i < m; i += blockDim.x) col[c * kMaxKrylov + i] = S[i];
    if (threadIdx.x == 0) {
        const double2 hs = H[(m - 1) * ldh + m];
        const double2 e = S[m - 1];
        err[c] = make_double2(exact ? 0.0 : hypot(hs.x, hs.y) * hypot(e.x, e.y), 0.0);
    }
}

// ------------------------------------------------------------------- host
int launch_g_cell(const afem_mesh* m, const double* E, const double2* v, const double2* U, double2* z, int n,
                  cudaStream_t s, int velocity, const double2* U_hang = nullptr);

// The frozen mean fields at the hanging points, Uh[h] = sum_e w_e U[master_e]
// (the constraint rows C; the same products in the same order as the cell
// passes' own gather, so the cell pass gives the same bits either way), formed
// once per propagation instead of in every cell pass of every Krylov vector.
__global__ void hang_rows64_kernel(const double2* __restrict__ U, const int32_t* __restrict__ hp,
                                   const int32_t* __restrict__ hm, const double* __restrict__ hw, int64_t nh, int k,
                                   double2* __restrict__ Uh) {
    const int64_t n = nh * k;
    for (int64_t o = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; o < n; o += int64_t(gridDim.x) * blockDim.x) {
        const int64_t h = o / k;
        const int c = int(o - h * k);
        double2 v = make_double2(0.0, 0.0);
        for (int e = hp[h]; e < hp[h + 1]; ++e) {
            const double2 u = U[int64_t(hm[e]) * k + c];
            v.x = fma(hw[e], u.x, v.x);
            v.y = fma(hw[e], u.y, v.y);
        }
        Uh[o] = v;
    }
}

__global__ void hang_rows32_kernel(const float2* __restrict__ U, const int32_t* __restrict__ hp,
                                   const int32_t* __restrict__ hm, const float* __restrict__ hw, int64_t nh, int k,
                                   float2* __restrict__ Uh) {
    const int64_t n = nh * k;
    for (int64_t o = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; o < n; o += int64_t(gridDim.x) * blockDim.x) {
        const int64_t h = o / k;
        const int c = int(o - h * k);
        float2 v = make_float2(0.0f, 0.0f);
        for (int e = hp[h]; e < hp[h + 1]; ++e) {
            const float2 u = U[int64_t(hm[e]) * k + c];
            v.x = fmaf(hw[e], u.x, v.x);
            v.y = fmaf(hw[e], u.y, v.y);
        }
        Uh[o] = v;
    }
}

int cdot(const double2* A, int na, const double2* B, int nb, const double* w, int64_t rows, int diag,
         double2* partial, double2* out, unsigned* counter, cudaStream_t s) {
    AFEM_LAUNCH((cdot_fused_kernel), row_blocks(rows, diag ? na : na * nb), kRedThreads, 0, s, A, na, B, nb, w, rows, diag,
                reinterpret_cast<double*>(partial), counter, out);
    AFEM_CUDA_TRY(cudaGetLastError());
    return AFEM_OK;
}

__global__ void to_c64_kernel(const double2* __restrict__ x, float2* __restrict__ y, int64_t n) {
    for (int64_t o = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; o < n; o += int64_t(gridDim.x) * blockDim.x)
        y[o] = make_float2(narrow_f64(x[o].x), narrow_f64(x[o].y));
}

__global__ void narrow_kernel(const double* __restrict__ x, float* __restrict__ y, int64_t n) {
    for (int64_t o = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; o < n; o += int64_t(gridDim.x) * blockDim.x)
        y[o] = narrow_f64(x[o]);
}

__global__ void widen_kernel(const float* __restrict__ x, double* __restrict__ y, int64_t n) {
    for (int64_t o = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; o < n; o += int64_t(gridDim.x) * blockDim.x)
        y[o] = widen_f32(x[o]);
}

int convert_f64_f32(const double* x, float* y, int64_t n, cudaStream_t s) {
    if (n <= 0) return AFEM_OK;
    AFEM_LAUNCH((narrow_kernel), grid_for(n), 256, 0, s, x, y, n);
    AFEM_CUDA_TRY(cudaGetLastError());
    return AFEM_OK;
}

int convert_f32_f64(const float* x, double* y, int64_t n, cudaStream_t s) {
    if (n <= 0) return AFEM_OK;
    AFEM_LAUNCH((widen_kernel), grid_for(n), 256, 0, s, x, y, n);
    AFEM_CUDA_TRY(cudaGetLastError());
    return AFEM_OK;
}

int to_c64(const double2* x, float2* y, int64_t n, cudaStream_t s) {
    AFEM_LAUNCH((to_c64_kernel), grid_for(n), 256, 0, s, x, y, n);
    AFEM_CUDA_TRY(cudaGetLastError());
    return AFEM_OK;
}

int launch_g_cell32(const afem_mesh* m, const double* E, const float2* v, const float2* U, float2* z, int n,
                    cudaStream_t s, int velocity, const float2* U_hang = nullptr,
                    CellForm form = CellForm::kNode);

// Blocks of kernel K for `tiles` tiles: one resident wave at most (every block
// then takes several tiles and adds one row of partial sums).
template <auto K>
static unsigned wave_grid(int64_t tiles, size_t smem) {
    static const int per_sm = [smem] {
        int b = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, K, kRedThreads, smem) != cudaSuccess || b < 1) b = 1;
        return b;
    }();
    const int64_t cap = std::min<int64_t>(int64_t(device_sms()) * per_sm, red_blocks());
    return unsigned(std::max<int64_t>(1, std::min(tiles, cap)));
}

// Rows of a tile per thread: as many as leave each SM a tile.  The two float64
// additions of a group and vector serve all its rows, so fewer rows cost more
// than idle warps: one orbital on 78,761 points with one row per thread (four
// tiles per SM) took 24.5 us per inner-product pass, with two rows 17.4 us.
static int krylov_rows(int64_t N, int n) {
    const int64_t R = kRedThreads / n;
    for (int E = 4; E > 1; E >>= 1)
        if ((N + E * R - 1) / (E * R) >= device_sms()) return E;
    return 1;
}

template <int E, int MODE, int STAGES>
static int launch_gs_dots_s(const GsDotsArgs& a, cudaStream_t s) {
    constexpr size_t kStage = size_t(STAGES) * kRedThreads * (E * sizeof(int4) + exp_words(E) * sizeof(int));
    AFEM_CUDA_TRY(allow_dyn_smem(gs_dots_kernel<E, MODE, STAGES>));
    const unsigned g = wave_grid<gs_dots_kernel<E, MODE, STAGES>>(
        a.B.tiles, (STAGES == 4 ? 9 : STAGES == 3 ? 13 : 16) * kRedThreads * sizeof(double2) + kStage);
    AFEM_LAUNCH((gs_dots_kernel<E, MODE, STAGES>), g, kRedThreads, a.nv * kRedThreads * sizeof(double2) + kStage, s, a);
    AFEM_CUDA_TRY(cudaGetLastError());
    return AFEM_OK;
}
template <int E, int MODE>
static int launch_gs_dots_e(const GsDotsArgs& a, cudaStream_t s) {
    // (the sums of nv vectors beside the ring: its depth leaves two blocks per SM)
    return a.nv <= 9 ? launch_gs_dots_s<E, MODE, 4>(a, s) : a.nv <= 13 ? launch_gs_dots_s<E, MODE, 3>(a, s)
                                                                       : launch_gs_dots_s<E, MODE, 2>(a, s);
}
template <int MODE>
static int launch_gs_dots(int E, const GsDotsArgs& a, cudaStream_t s) {
    if (a.nv < 1 || a.nv > kMaxKrylov) return set_error(AFEM_EINVAL, "arnoldi: Krylov vector count out of range");
    return E == 4 ? launch_gs_dots_e<4, MODE>(a, s) : E == 2 ? launch_gs_dots_e<2, MODE>(a, s)
                                                            : launch_gs_dots_e<1, MODE>(a, s);
}

template <int E, int KIND, int STAGES, int NV>   // NV: most vectors of this ring depth
static int launch_gs_combine_s(const GsCombineArgs& a, cudaStream_t s) {
    constexpr size_t kStage = KIND == 0 ? 0 : size_t(STAGES) * kRedThreads * E * sizeof(int4);
    constexpr size_t kExp = KIND == 0 ? 0 : 2 * kRedThreads * exp_words(E) * sizeof(int);   // per vector
    AFEM_CUDA_TRY(allow_dyn_smem(gs_combine_kernel<E, KIND, STAGES>));
    const unsigned g = wave_grid<gs_combine_kernel<E, KIND, STAGES>>(a.B.tiles, kStage + NV * kExp);
    AFEM_LAUNCH((gs_combine_kernel<E, KIND, STAGES>), g, kRedThreads, kStage + a.nv * kExp, s, a);
    AFEM_CUDA_TRY(cudaGetLastError());
    return AFEM_OK;
}
// With four rows the exponents of 16 vectors take 64 KB beside the ring: its
// depth leaves two blocks per SM.
template <int E, int KIND>
static int launch_gs_combine_e(const GsCombineArgs& a, cudaStream_t s) {
    if constexpr (E == 4 && KIND != 0) {
        if (a.nv > 14) return launch_gs_combine_s<E, KIND, 2, kMaxKrylov>(a, s);
        if (a.nv > 11) return launch_gs_combine_s<E, KIND, 3, 14>(a, s);
        return launch_gs_combine_s<E, KIND, 4, 11>(a, s);
    } else {
        return launch_gs_combine_s<E, KIND, 4, kMaxKrylov>(a, s);
    }
}
template <int KIND>
static int launch_gs_combine(int E, const GsCombineArgs& a, cudaStream_t s) {
    if (a.nv < (KIND == 0 ? 0 : 1) || a.nv > kMaxKrylov)
        return set_error(AFEM_EINVAL, "arnoldi: Krylov vector count out of range");
    return E == 4 ? launch_gs_combine_e<4, KIND>(a, s) : E == 2 ? launch_gs_combine_e<2, KIND>(a, s)
                                                               : launch_gs_combine_e<1, KIND>(a, s);
}

// The cell pass of G and the projector overlaps S[j][p] = phi_j^H z_p (equal to
// phi_j^H M_L y_p); the projector itself runs fused with the first
// Gram-Schmidt pass.  Precision form: the cell pass in complex64 from v32 (the
// complex64 copy of the vector) and the overlaps from phi32.
static int g_cell_overlaps32(afem_mesh* m, const double* E, const float2* phi32, const float2* U32, int n,
                             const float2* v32, ArnoldiWork& w, cudaStream_t s, int velocity) {
    const DeviceMesh& D = m->dev;
    int rc;
    {   // algorithmic bytes: read v, U (n^2 fields), write z, complex64
        ProfScope ps(AFEM_PROF_GCELL32, s, double(D.n_master) * 8.0 * n * (2 + n));
        rc = w.gb ? launch_g_cell32_blocks(m, v32, w.gb, w.z32, n, w.bulk_err, w.vh32, s)
                  : launch_g_cell32(m, E, v32, U32, w.z32, n, s, velocity, w.uh32);
        if (rc) return rc;
    }
    auto* part = reinterpret_cast<double*>(w.cpartial);
    switch (n) {
#define AFEM_OV_CASE(NO)                                                                                        \
    case NO:                                                                                                    \
        AFEM_LAUNCH((overlap32_kernel<NO>), red_blocks(), kRedThreads, 0, s, phi32, w.z32, D.n_interior,         \
                    w.Sslots);                                                                                  \
        break;
        AFEM_OV_CASE(1)
        AFEM_OV_CASE(2)
        AFEM_OV_CASE(3)
        AFEM_OV_CASE(4)
        AFEM_OV_CASE(5)
        AFEM_OV_CASE(6)
        AFEM_OV_CASE(7)
        AFEM_OV_CASE(8)
#undef AFEM_OV_CASE
        default:
            return set_error(AFEM_EINVAL, "arnoldi: orbital count out of range");
    }
    AFEM_CUDA_TRY(cudaGetLastError());
    return AFEM_OK;
}

static int g_cell_overlaps(afem_mesh* m, const double* E, const double2* phi, const double2* U, int n,
                           const double2* v, ArnoldiWork& w, cudaStream_t s, int velocity) {
    const DeviceMesh& D = m->dev;
    int rc;
    {
        const int p1 = D.p + 1;
        ProfScope ps(AFEM_PROF_CELL64, s, double(D.ncell) * p1 * p1 * p1 * 2.0 * n * (3.0 * p1 * 2.0 + 6.0));
        rc = launch_g_cell(m, E, v, U, w.z, n, s, velocity, w.uh);
    }
    if (rc) return rc;
    return cdot(phi, n, w.z, n, nullptr, D.n_interior, 0, w.cpartial, w.S, w.counters, s);
}

int arnoldi_reserve(afem_mesh* m, int n, int mk, ArnoldiWork& w) {
    const size_t NV = size_t(m->dev.n_master) * n;
    w.rows = krylov_rows(m->dev.n_master, n);
    const int64_t tile = int64_t(w.rows) * (kRedThreads / n);
    w.B.tiles = (m->dev.n_master + tile - 1) / tile;
    w.B.stride = w.B.tiles * w.rows * kRedThreads;
    w.B.estride = w.B.tiles * kRedThreads * exp_words(w.rows);
    auto carve = [&](Carver& cv) {
        w.B.V = cv.take<int4>(size_t(mk + 1) * w.B.stride);
        w.B.e = cv.take<int>(size_t(mk + 1) * w.B.estride);
        w.vd = cv.take<double2>(NV);
        w.z = cv.take<double2>(NV);
        w.cpartial = cv.take<double2>(size_t(kRedBlocksMax) * 256);
        w.S = cv.take<double2>(kMaxOrbProj * kMaxOrbProj);
        w.Sslots = cv.take<double>(size_t(kOvSlots) * 2 * kMaxOrbProj * kMaxOrbProj);
        w.res = cv.take<double2>(kResSize);
        w.c1 = cv.take<double2>(kMaxKrylov + 1);
        w.c2 = cv.take<double2>(kMaxKrylov + 1);
        w.f = cv.take<double>(kScaleBeta + 1);
        w.v32 = cv.take<float2>(NV);
        w.z32 = cv.take<float2>(NV);
        w.phi32 = cv.take<float2>(NV);
        w.U32 = cv.take<float2>(NV * n);
        w.Uh = cv.take<double2>(size_t(m->dev.n_hanging) * n * n);
        w.Uh32 = cv.take<float2>(size_t(m->dev.n_hanging) * n * n);
        w.vh32 = reinterpret_cast<float4*>(cv.take<float2>(size_t(m->dev.n_hanging) * n + 2));
        w.counters = cv.take<unsigned>(4);
        w.flag = cv.take<int>(4);
    };
    Carver measure(nullptr);
    carve(measure);
    int rc = m->ws_arnoldi.reserve(measure.size());
    if (rc) return rc;
    Carver cv(m->ws_arnoldi.ptr);
    carve(cv);
    w.H = w.res + kResH;
    w.beta2 = w.res + kResBeta2;
    w.col = w.res + kResCol;
    w.err = w.res + kResErr;
    w.bulk_err = reinterpret_cast<double*>(w.res + kResFlag);
    w.gb = nullptr;
    return AFEM_OK;
}

// Candidate substep lengths of one ladder: tau_max * 2^(-c/8), c = 0..K-1.
static TauLadder make_ladder(double tau_max, int K) {
    TauLadder L{};
    for (int c = 0; c < kLadder; ++c) L.tau[c] = c < K ? tau_max * std::pow(2.0, -kLadderLog2 * c) : 0.0;
    return L;
}

// Propagates phi by exp(-i G dt) with G frozen at phi (projector), U and E.
// tol <= 0: one Krylov step of dimension mk over the whole dt.  tol > 0:
// substeps from fresh Krylov spaces of the same G, each as long as the error
// estimate beta |h_{m+1,m}| |e_m^T exp(-i tau H_m) e_1| <= tol * beta allows
// among the candidates tau_max 2^(-c/8), c = 0..63, where tau_max is the
// remainder for the first substep and min(remainder, 2 tau_previous) after
// it; when no candidate passes, the ladder continues below the smallest one
// (the paper fixes the Krylov accuracy by such an estimate; here the
// dimension is fixed and the substep adapts).
int arnoldi_step(afem_mesh* m, const double* E, const double2* phi, const double2* U, const float2* U32, int n,
                 int mk, double dt, int mixed, double tol, double2* phi_out, double* err_est, int* m_used_out,
                 int* breakdown_out, int* substeps_out, cudaStream_t s, int flags, int adaptive_steps,
                 int* dim_sum_out, int* unmet_out) {
    const DeviceMesh& D = m->dev;
    if (mk < 1 || mk > kMaxKrylov) return set_error(AFEM_EINVAL, "arnoldi: krylov_m out of range");
    if (n < 1 || n > kMaxOrbProj) return set_error(AFEM_EINVAL, "arnoldi: orbital count out of range");
    if (adaptive_steps < 0 || (adaptive_steps > 0 && !(tol > 0.0)))
        return set_error(AFEM_EINVAL, "arnoldi: the adaptive dimension needs steps >= 1 and a threshold > 0");
    const int imag = (flags & kArnImaginary) ? 1 : 0;
    const int velocity = (flags & kArnVelocity) ? 1 : 0;   // E holds the vector potential A
    const bool adaptive = adaptive_steps > 0;
    const double tau_fixed = adaptive ? dt / adaptive_steps : 0.0;
    ArnoldiWork w{};
    int rc = arnoldi_reserve(m, n, mk, w);
    if (rc) return rc;
    const int64_t NV = D.n_master * n;
    const bool projector = !(flags & kArnNoProjector);
    // candidate exponentials exp(-i tau H_m), or exp(+i tau H_m) propagating backward
    auto signed_ladder = [&](double tm, int K) {
        TauLadder L = make_ladder(tm, K);
        if (flags & kArnBackward)
            for (int c = 0; c < kLadder; ++c) L.tau[c] = -L.tau[c];
        return L;
    };
    if (!projector) AFEM_CUDA_TRY(cudaMemsetAsync(w.S, 0, sizeof(double2) * kMaxOrbProj * kMaxOrbProj, s));
    if (mixed) {
        if (U && !U32) {
            if ((rc = to_c64(U, w.U32, D.n_master * n * n, s))) return rc;
            U32 = w.U32;
        }
        if ((rc = to_c64(phi, w.phi32, NV, s))) return rc;
    }
    w.uh = nullptr;
    w.uh32 = nullptr;
    if (D.n_hanging > 0 && (mixed ? U32 != nullptr : U != nullptr)) {
        const int64_t nh = D.n_hanging;
        const int k = n * n;
        if (mixed) {
            AFEM_LAUNCH((hang_rows32_kernel), grid_for(nh * k), 256, 0, s, U32, D.hang_ptr, D.hang_master,
                        D.hang_w32, nh, k, w.Uh32);
            w.uh32 = w.Uh32;
        } else {
            AFEM_LAUNCH((hang_rows64_kernel), grid_for(nh * k), 256, 0, s, U, D.hang_ptr, D.hang_master, D.hang_w,
                        nh, k, w.Uh);
            w.uh = w.Uh;
        }
        AFEM_CUDA_TRY(cudaGetLastError());
    }
    w.gb = nullptr;
    if (mixed && U32 && gcell_blocks_apply(m, n, velocity)) {
        // the frozen pointwise part of G, one contiguous block per cell, staged by
        // the cell pass with one bulk copy (formed once for all substeps)
        if ((rc = m->ws_gblocks.reserve(gcell_blocks_bytes(m, n)))) return rc;
        auto* B = static_cast<float4*>(m->ws_gblocks.ptr);
        if ((rc = build_gcell_blocks32(m, E, U32, w.uh32, n, B, s))) return rc;
        w.gb = B;
        AFEM_CUDA_TRY(cudaMemsetAsync(w.bulk_err, 0, sizeof(double), s));
    }
    AFEM_CUDA_TRY(cudaMemsetAsync(w.counters, 0, 4 * sizeof(unsigned), s));
    AFEM_CUDA_TRY(cudaMemsetAsync(w.flag, 0, 4 * sizeof(int), s));
    AFEM_CUDA_TRY(cudaMemsetAsync(w.Sslots, 0, sizeof(double) * kOvSlots * 2 * kMaxOrbProj * kMaxOrbProj, s));
    const int ldh = kMaxKrylov + 1;
    double* part = reinterpret_cast<double*>(w.cpartial);
    unsigned* cnt = w.counters + 1;
    const double eta2 = 1e-4;   // second pass when the update left less than 1e-2 of the norm
    double remaining = dt, tau_prev = 0.0;
    double err_sum = 0.0;
    int substeps = 0, m_used = mk, brk = 0, dim_max = 0, dim_sum = 0, unmet = 0;
    std::vector<double2> res(kResSize);
    auto fetch = [&]() -> int {
        AFEM_CUDA_TRY(cudaMemcpyAsync(res.data(), w.res, kResSize * sizeof(double2), cudaMemcpyDeviceToHost, s));
        AFEM_CUDA_TRY(cudaStreamSynchronize(s));
        if (w.gb && res[kResFlag].x != 0.0)
            return set_error(AFEM_ECUDA, "arnoldi: a G cell pass gave up waiting for a per-cell block copy");
        return AFEM_OK;
    };
    GsDotsArgs da{};
    da.z = w.z;
    da.z32 = w.z32;
    da.phi = phi;
    da.phi32 = w.phi32;
    da.S = w.S;
    da.S_slots = (mixed && projector) ? w.Sslots : nullptr;
    da.ml_inv = D.ml_inv;
    da.ml_inv32 = D.ml_inv32;
    da.ml = D.ml;
    da.n_int = D.n_interior;
    da.N = D.n_master;
    da.n = n;
    da.wd = w.vd;
    da.B = w.B;
    da.f = w.f;
    da.partial = part;
    da.counter = cnt;
    GsCombineArgs ca{};
    ca.B = w.B;
    ca.src = phi;
    ca.wd = w.vd;
    ca.w32 = mixed ? w.z32 : nullptr;
    ca.ml = D.ml;
    ca.n_int = D.n_interior;
    ca.N = D.n_master;
    ca.n = n;
    ca.gate = w.flag;
    ca.eta2 = eta2;
    ca.reorth = w.flag;
    ca.f = w.f;
    ca.vd = mixed ? nullptr : w.vd;
    ca.v32 = mixed ? w.v32 : nullptr;
    ca.partial = part;
    ca.counter = cnt;
    ca.beta2_out = w.beta2;
    // V_0 = phi (unscaled), the cell pass's copy of it and beta^2 = <phi, phi>_M;
    // later substeps get theirs from the closing pass of the previous one
    if ((rc = launch_gs_combine<0>(w.rows, ca, s))) return rc;
    // closes a substep with the coefficients y = beta exp(..) e_1; phi_out is
    // written by the last one alone
    auto close = [&](int mu, const double2* y, double beta, bool last) -> int {
        ca.nv = mu;
        ca.c = y;
        ca.scale = beta;
        ca.out = last ? phi_out : nullptr;
        return launch_gs_combine<1>(w.rows, ca, s);
    };
    while (remaining > 0.0) {
        if (substeps >= 4096) return set_error(AFEM_EINVAL, "arnoldi: more than 4096 substeps (tolerance too tight)");
        AFEM_CUDA_TRY(cudaMemsetAsync(w.H, 0, sizeof(double2) * ldh * kMaxKrylov, s));
        for (int j = 0; j < mk; ++j) {
            double2* Hcol = w.H + j * ldh;
            // w = G q_j (the cell pass on the stored V_j, scaled in the projector
            // pass) with the inner products against q_0..q_j, the update (which
            // leaves V_{j+1} = h_{j+1,j} q_{j+1}), and a second pass when the
            // update cancelled most of w
            if (!projector) {   // the cell pass alone; S stays zero
                if (mixed) {
                    rc = w.gb ? launch_g_cell32_blocks(m, w.v32, w.gb, w.z32, n, w.bulk_err, w.vh32, s)
                              : launch_g_cell32(m, E, w.v32, U32, w.z32, n, s, velocity, w.uh32);
                    if (rc) return rc;
                } else {
                    if ((rc = launch_g_cell(m, E, w.vd, U, w.z, n, s, velocity, w.uh))) return rc;
                }
            } else if (mixed) {
                if ((rc = g_cell_overlaps32(m, E, w.phi32, U32, n, w.v32, w, s, velocity))) return rc;
            } else {
                if ((rc = g_cell_overlaps(m, E, phi, U, n, w.vd, w, s, velocity))) return rc;
            }
            // algorithmic FP64 flops per element: 8 per basis vector in each pass
            // (one complex multiply-add), plus 4 for the new norm in the update
            const double gs_flops = double(D.n_interior) * n * 8.0 * (j + 1);
            {
                ProfScope ps(AFEM_PROF_GS, s, gs_flops);
                da.nv = j + 1;
                da.gate = nullptr;
                da.out = w.c1;
                rc = mixed ? launch_gs_dots<2>(w.rows, da, s) : launch_gs_dots<1>(w.rows, da, s);
            }
            ca.nv = j + 1;
            ca.c = w.c1;
            ca.Hcol = Hcol;
            if (!rc) {
                ProfScope ps(AFEM_PROF_GS, s, gs_flops + double(D.n_interior) * n * 4.0);
                rc = mixed ? launch_gs_combine<4>(w.rows, ca, s) : launch_gs_combine<2>(w.rows, ca, s);
            }
            da.gate = w.flag;
            da.out = w.c2;
            ca.c = w.c2;
            if (rc || (rc = launch_gs_dots<0>(w.rows, da, s)) || (rc = launch_gs_combine<3>(w.rows, ca, s))) return rc;
            if (adaptive) {
                // Sec. 3.2's rule: the estimate of dimension j + 1 at the fixed step;
                // the first dimension that meets the threshold (or breaks down) ends
                // the process
                AFEM_LAUNCH((expm_ladder_kernel), 1, kExpmThreads, 0, s, w.H, ldh, j + 1, signed_ladder(tau_fixed, 1), 0,
                            imag, w.col, w.err);
                AFEM_CUDA_TRY(cudaGetLastError());
                if ((rc = fetch())) return rc;
                const double b = std::sqrt(res[kResBeta2].x);
                const double hn = res[kResH + j * ldh + j + 1].x;
                if (!(b > 0.0) || !std::isfinite(b) || !std::isfinite(hn))
                    return set_error(AFEM_ENAN, "arnoldi: zero or non-finite Krylov vector");
                m_used = j + 1;
                brk = hn < 1e-14 * b ? 1 : 0;
                if (brk || res[kResErr].x <= tol) break;
            }
        }
        double tau, err;
        int pick = 0;
        if (adaptive) {
            const double beta = std::sqrt(res[kResBeta2].x);
            tau = tau_fixed;
            err = brk ? 0.0 : beta * res[kResErr].x;
            if (!brk && res[kResErr].x > tol) ++unmet;
            if ((rc = close(m_used, w.col, beta, substeps + 1 >= adaptive_steps || !(remaining - tau > 0.0)))) return rc;
            err_sum += err;
            ++substeps;
            dim_max = std::max(dim_max, m_used);
            dim_sum += m_used;
            tau_prev = tau;
            remaining = substeps >= adaptive_steps ? 0.0 : remaining - tau;
            continue;
        }
        // candidate substeps, one block each; a single host wait per ladder
        double tau_max = (tol <= 0.0 || substeps == 0) ? remaining : std::fmin(remaining, 2.0 * tau_prev);
        int K = tol <= 0.0 ? 1 : kLadder;
        int exact = 0;
        AFEM_LAUNCH((expm_ladder_kernel), K, kExpmThreads, 0, s, w.H, ldh, mk, signed_ladder(tau_max, K), 0, imag, w.col,
                    w.err);
        AFEM_CUDA_TRY(cudaGetLastError());
        if ((rc = fetch())) return rc;
        const double beta = std::sqrt(res[kResBeta2].x);
        if (!(beta > 0.0) || !std::isfinite(beta)) return set_error(AFEM_ENAN, "arnoldi: zero or non-finite norm");
        m_used = mk;
        brk = 0;
        for (int j = 0; j < mk; ++j) {
            const double hn = res[kResH + j * ldh + j + 1].x;
            if (!std::isfinite(hn)) return set_error(AFEM_ENAN, "arnoldi: non-finite Krylov vector");
            if (hn < 1e-14 * beta) {
                m_used = j + 1;
                brk = 1;
                break;
            }
        }
        if (brk) {   // invariant subspace: the projected exponential is exact
            tau_max = remaining;
            K = 1;
            exact = 1;
            AFEM_LAUNCH((expm_ladder_kernel), 1, kExpmThreads, 0, s, w.H, ldh, m_used, signed_ladder(tau_max, 1), 1, imag,
                        w.col, w.err);
            AFEM_CUDA_TRY(cudaGetLastError());
            if ((rc = fetch())) return rc;
        }
        pick = -1;
        for (int round = 0;; ++round) {
            for (int c = 0; c < K; ++c) {
                if (exact || tol <= 0.0 || res[kResErr + c].x <= tol) {
                    pick = c;
                    break;
                }
            }
            if (pick >= 0) break;
            if (round >= 8) {   // accept the smallest candidate
                pick = K - 1;
                break;
            }
            tau_max *= std::pow(2.0, -kLadderLog2 * K);
            AFEM_LAUNCH((expm_ladder_kernel), K, kExpmThreads, 0, s, w.H, ldh, m_used, signed_ladder(tau_max, K), 0, imag,
                        w.col, w.err);
            AFEM_CUDA_TRY(cudaGetLastError());
            if ((rc = fetch())) return rc;
        }
        tau = make_ladder(tau_max, K).tau[pick];
        err = beta * res[kResErr + pick].x;
        // phi_out = beta V_m exp(-i tau H_m) e_1, which also opens the next substep
        if ((rc = close(m_used, w.col + pick * kMaxKrylov, beta, tau >= remaining || !(remaining - tau > 0.0))))
            return rc;
        err_sum += err;
        ++substeps;
        dim_max = std::max(dim_max, m_used);
        dim_sum += m_used;
        tau_prev = tau;
        remaining = (tau >= remaining) ? 0.0 : remaining - tau;
    }
    AFEM_CUDA_TRY(cudaStreamSynchronize(s));
    if (err_est) *err_est = err_sum;
    if (m_used_out) *m_used_out = adaptive ? dim_max : m_used;
    if (dim_sum_out) *dim_sum_out = dim_sum;
    if (unmet_out) *unmet_out = unmet;
    if (breakdown_out) *breakdown_out = brk;
    if (substeps_out) *substeps_out = substeps;
    return AFEM_OK;
}

}  // namespace afem

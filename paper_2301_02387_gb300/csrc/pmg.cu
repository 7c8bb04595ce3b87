// Geometric multigrid preconditioner for the batched Poisson solves of the
// mean fields (Sec. 3.1, Eq. mean-field: the paper solves them by CG with an
// algebraic multigrid preconditioner; this is its geometric counterpart on the
// octree the library already holds).
//
// Levels, fine to coarse: the mesh itself (degree p); the same leaves at
// degree p/2, ..., 1 (p-coarsening); then degree 1 on the octree truncated at
// levels L-1, ..., 0 (h-coarsening: every leaf finer than the cap replaced by
// its ancestor there; the last is the uniform coarse grid).  Every leaf of a
// level has an ancestor-or-self leaf on the next coarser octree, whatever rule
// refined the mesh, and the coarse finite-element space is a
// subspace of the fine one, so the prolongation P is exact interpolation: the
// value of the coarse function at each interior fine master, evaluated in one
// "owner" cell that holds the master as a node (the lowest-index such cell).
// The restriction is R = P^T (the owner's interpolation weights, transposed,
// then the coarse constraints C^T), so the V-cycle is a symmetric operator.
// Smoothing: Chebyshev polynomials in D^-1 A (D the diagonal of the
// constrained stiffness) on [lambda_max / 15, 1.15 lambda_max], degree 3 before
// and after the coarse correction; lambda_max by power iteration at set-up;
// the coarsest level gets a degree-30 Chebyshev polynomial on
// [lambda_max / 400, 1.15 lambda_max].  All levels act on the Dirichlet
// interior (surface rows zero), every column of the batch at once.
//
// Solvers built on it: CG in float64 preconditioned by the float64 V-cycle (the
// FP64 form), and float64 defect correction whose corrections are float32 CG
// iterations preconditioned by the float32 V-cycle (the precision form).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <new>
#include <tuple>
#include <type_traits>
#include <unordered_set>
#include <vector>

#include "afem_internal.h"
#include "vec_common.cuh"

namespace afem {

int launch_stiffness32(const afem_mesh* m, const float* x, float* y, int nv, int masked, cudaStream_t s,
                       double* pap_slots, bool y_zero = false, CellForm form = CellForm::kBySize);
int poisson_rhs_bc(afem_mesh* m, const double2* phi, int n, double* W, double* b, double* qpart, double* q,
                   cudaStream_t s);
int mom_blocks_count();
constexpr int kPmgMaxP1 = kMaxP1;
constexpr int kPmgPreDegree = 3;      // Chebyshev degree of each smoothing
constexpr int kPmgCoarseDegree = 30;  // Chebyshev degree on the coarsest level
constexpr double kPmgSmoothRange = 15.0;
constexpr double kPmgCoarseRange = 400.0;
constexpr double kPmgLambdaSafety = 1.15;
constexpr int kPmgPowerIters = 40;

struct PmgLevel {
    afem_mesh* mesh = nullptr;   // level 0: the caller's mesh (not owned)
    bool owned = false;
    // transfer from the next coarser level to this one, per cell of this level
    int32_t* coarse_cell = nullptr;   // [ncell] the coarse ancestor-or-self leaf
    float4* xform = nullptr;          // [ncell] (offset x, y, z, scale) in the coarse cell's unit cube
    int32_t* own_node = nullptr;      // [ncell][(p+1)^3] the interior master whose value this (cell, node) holds, or -1
    double lam_max = 0.0;             // largest eigenvalue of D^-1 A_II
    // the coarsest level: interior master of each interior grid node, x fastest
    int32_t* grid_map = nullptr;      // [grid_n^3]
    int grid_n = 0;                   // 0: not a uniform degree-1 grid
};

}  // namespace afem

struct afem_pmg {
    std::vector<afem::PmgLevel> lv;
    afem::Workspace ws;   // level vectors of the current solve
};

namespace afem {

// ------------------------------------------------------------- set-up (host)
static void free_level(PmgLevel& L) {
    cudaFree(L.coarse_cell);
    cudaFree(L.xform);
    cudaFree(L.own_node);
    cudaFree(L.grid_map);
    L.grid_map = nullptr;
    L.grid_n = 0;
    L.coarse_cell = nullptr;
    L.xform = nullptr;
    L.own_node = nullptr;
    if (L.owned && L.mesh) afem_mesh_destroy(L.mesh);
    L.mesh = nullptr;
}

void pmg_free(afem_pmg* g) {
    if (!g) return;
    for (auto& L : g->lv) free_level(L);
    g->ws.release();
    delete g;
}

template <typename T>
static int upload(T*& dst, const std::vector<T>& v) {
    dst = nullptr;
    if (v.empty()) return AFEM_OK;
    cudaError_t e = cudaMalloc(&dst, v.size() * sizeof(T));
    if (e != cudaSuccess) return set_error(AFEM_ENOMEM, "multigrid set-up: cudaMalloc failed");
    AFEM_CUDA_TRY(cudaMemcpy(dst, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice));
    return AFEM_OK;
}

// Ancestor map and owner flags of fine level `f` over coarse level `c`.
static int build_transfer(const HostMesh& F, const HostMesh& C, PmgLevel& L) {
    const int64_t nf = int64_t(F.lev.size());
    std::map<std::tuple<int, int, int, int>, int32_t> key;
    for (int32_t c = 0; c < int32_t(C.lev.size()); ++c) key[{C.lev[c], C.ci[c], C.cj[c], C.ck[c]}] = c;
    std::vector<int32_t> cc(nf);
    std::vector<float4> xf(nf);
    for (int64_t f = 0; f < nf; ++f) {
        int l = F.lev[f], i = F.ci[f], j = F.cj[f], k = F.ck[f];
        int found = -1, lc = l;
        for (; lc >= 0; --lc) {
            const int sh = l - lc;
            auto it = key.find({lc, i >> sh, j >> sh, k >> sh});
            if (it != key.end()) {
                found = it->second;
                break;
            }
        }
        if (found < 0) return set_error(AFEM_EMESH, "multigrid set-up: a leaf has no coarse ancestor");
        const int sh = l - lc;
        const float sc = std::ldexp(1.0f, -sh);
        cc[f] = found;
        xf[f] = make_float4(float(i - ((i >> sh) << sh)) * sc, float(j - ((j >> sh) << sh)) * sc,
                            float(k - ((k >> sh) << sh)) * sc, sc);
    }
    const int nn = (F.p + 1) * (F.p + 1) * (F.p + 1);
    std::vector<int32_t> own(size_t(nf) * nn, -1);
    std::vector<uint8_t> seen(size_t(F.n_master), 0);
    for (int64_t f = 0; f < nf; ++f)
        for (int i = 0; i < nn; ++i) {
            const int32_t idx = F.cell_node[size_t(f) * nn + i];
            if (idx < 0 || idx >= F.n_interior || seen[idx]) continue;
            seen[idx] = 1;
            own[size_t(f) * nn + i] = idx;
        }
    int rc;
    if ((rc = upload(L.coarse_cell, cc))) return rc;
    if ((rc = upload(L.xform, xf))) return rc;
    return upload(L.own_node, own);
}

// Interior master of every interior node of a uniform degree-1 grid (grid_n
// stays 0 for any other mesh).
static int build_grid_map(PmgLevel& L) {
    const HostMesh& H = L.mesh->host;
    const int n = H.n_coarse - 1;
    if (H.p != 1 || H.max_level != 0 || H.n_hanging != 0 || n < 1 || H.n_interior != int64_t(n) * n * n) return AFEM_OK;
    std::vector<int32_t> map(size_t(n) * n * n, -1);
    for (size_t c = 0; c < H.lev.size(); ++c)
        for (int q = 0; q < 8; ++q) {
            const int x = H.ci[c] + (q & 1) - 1, y = H.cj[c] + ((q >> 1) & 1) - 1, z = H.ck[c] + (q >> 2) - 1;
            if (x >= 0 && x < n && y >= 0 && y < n && z >= 0 && z < n)
                map[size_t(x) + size_t(n) * (y + size_t(n) * z)] = H.cell_node[c * 8 + q];
        }
    for (int32_t i : map)
        if (i < 0 || i >= H.n_interior) return AFEM_OK;
    const int rc = upload(L.grid_map, map);
    if (rc == AFEM_OK) L.grid_n = n;
    return rc;
}

// ------------------------------------------------------------------ kernels
// The vectors are [rows][k].  A thread owns one group of VEC columns (a 16-byte
// word where k allows it) and walks rows: no division of an element index by
// the run-time column count, column scalars formed once per thread.  With
// element indices divided in every element these kernels ran at 10-25 % of the
// copy rate (12.4 M float elements: update of x and r 218 us, of p 184 us,
// Chebyshev step 76 us; now 44, 29 and 40 us, 75-85 % of it).
template <typename T, int VEC>
struct alignas(sizeof(T) * VEC) Pack {
    T v[VEC];
};

struct ColGroup {
    int q, r, R;   // column group, first row within the block, rows per block
    bool on;
    __device__ __forceinline__ explicit ColGroup(int groups) {
        R = 256 / groups;
        r = int(threadIdx.x) / groups;
        q = int(threadIdx.x) - r * groups;
        on = r < R;
    }
};
template <typename T, int VEC>
__device__ __forceinline__ Pack<T, VEC> load_pack(const T* x, int64_t row, int groups, int q) {
    return reinterpret_cast<const Pack<T, VEC>*>(x)[row * groups + q];
}
template <typename T, int VEC>
__device__ __forceinline__ void store_pack(T* x, int64_t row, int groups, int q, const Pack<T, VEC>& p) {
    reinterpret_cast<Pack<T, VEC>*>(x)[row * groups + q] = p;
}

// Lagrange basis of degree pc (1 or 2) on its GLL nodes {0, 1} / {0, 1/2, 1}.
__device__ __forceinline__ float lagrange_c(int pc, int j, float t) {
    if (pc == 1) return j == 0 ? 1.0f - t : t;
    if (j == 0) return 2.0f * (t - 0.5f) * (t - 1.0f);
    if (j == 1) return -4.0f * t * (t - 1.0f);
    return 2.0f * t * (t - 0.5f);
}

struct XferArgs {
    // fine level
    const int32_t* own_node;  // [ncell][(pf+1)^3] the interior master this cell owns there, or -1
    const int32_t* coarse_cell;
    const float4* xform;
    int64_t ncell;
    float xi_f[kPmgMaxP1];
    // coarse level
    const int32_t* c_node;    // [ncell_c][(pc+1)^3]
    const int32_t* c_hp;
    const int32_t* c_hm;
    const double* c_hw;
    int64_t c_ni;             // coarse interior masters
    int k;                    // columns
};

// Cells of a transfer block: as many as give each thread of 256 one fine node
// (and column group).
__host__ __device__ constexpr int xfer_cells(int pf, int groups) {
    return (pf + 1) * (pf + 1) * (pf + 1) * groups >= 256 ? 1 : 256 / ((pf + 1) * (pf + 1) * (pf + 1) * groups);
}

// The (pf+1) x (pc+1) interpolation tables of the block's cells, per direction.
template <int PF, int PC>
__device__ __forceinline__ void xfer_tables(const XferArgs& a, int64_t f0, int cells, float (*tab)[PF + 1][PC + 1]) {
    constexpr int NT = 3 * (PF + 1) * (PC + 1);
    for (int t = threadIdx.x; t < cells * NT; t += blockDim.x) {
        const int cell = t / NT, u = t - cell * NT;
        const int d = u / ((PF + 1) * (PC + 1)), r = u - d * (PF + 1) * (PC + 1);
        const int i = r / (PC + 1), j = r - i * (PC + 1);
        const float4 x = a.xform[f0 + cell];
        tab[3 * cell + d][i][j] = lagrange_c(PC, j, (d == 0 ? x.x : d == 1 ? x.y : x.z) + x.w * a.xi_f[i]);
    }
}

// Coarse values of the block's cells: one (cell, coarse node, column group) per
// item, hanging points through the coarse constraints.
template <typename T, int VEC>
__device__ __forceinline__ Pack<T, VEC> coarse_value(const XferArgs& a, int idx, const T* __restrict__ xc, int groups,
                                                     int q) {
    Pack<T, VEC> v{};
    if (idx >= 0) {
        if (idx < a.c_ni) v = load_pack<T, VEC>(xc, idx, groups, q);
        return v;
    }
    const int h = -idx - 1;
    for (int e = a.c_hp[h]; e < a.c_hp[h + 1]; ++e) {
        const int mm = a.c_hm[e];
        if (mm >= a.c_ni) continue;
        const T w = T(a.c_hw[e]);
        const Pack<T, VEC> u = load_pack<T, VEC>(xc, mm, groups, q);
#pragma unroll
        for (int s = 0; s < VEC; ++s) v.v[s] += w * u.v[s];
    }
    return v;
}

// y_f += P x_c: every interior fine master gets the coarse function's value at
// its position, evaluated in its owner cell, one direction at a time (pc + 1
// products per value and direction instead of (pc + 1)^3 per fine node).
template <typename T, int VEC, int PF, int PC>
__global__ void __launch_bounds__(256) pmg_prolong_kernel(const __grid_constant__ XferArgs a,
                                                          const T* __restrict__ xc, T* __restrict__ yf, int cpb) {
    constexpr int F1 = PF + 1, C1 = PC + 1, NF = F1 * F1 * F1, NC = C1 * C1 * C1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int groups = a.k / VEC;
    const int64_t f0 = int64_t(blockIdx.x) * cpb;
    const int cells = int(min(int64_t(cpb), a.ncell - f0));
    using P = Pack<T, VEC>;
    P* s_a = reinterpret_cast<P*>(smem_raw);             // [cpb][NC] coarse; then [cpb][C1][F1][F1]
    P* s_b = s_a + cpb * C1 * F1 * F1 * groups;          // [cpb][C1][C1][F1]
    float(*tab)[F1][C1] = reinterpret_cast<float(*)[F1][C1]>(s_b + cpb * C1 * C1 * F1 * groups);
    xfer_tables<PF, PC>(a, f0, cells, tab);
    const ColGroup g(groups);
    for (int it = g.on ? g.r : cells * NC; it < cells * NC; it += g.R) {
        const int cell = it / NC;
        s_a[it * groups + g.q] =
            coarse_value<T, VEC>(a, a.c_node[int64_t(a.coarse_cell[f0 + cell]) * NC + it - cell * NC], xc, groups, g.q);
    }
    __syncthreads();
    // x: [c][c][c] -> [c][c][f]
    for (int it = g.on ? g.r : cells * C1 * C1 * F1; it < cells * C1 * C1 * F1; it += g.R) {
        const int ia = it % F1, row = it / F1, cell = row / (C1 * C1);
        P v{};
#pragma unroll
        for (int j = 0; j < C1; ++j) {
            const T w = T(tab[3 * cell][ia][j]);
            const P u = s_a[(row * C1 + j) * groups + g.q];
#pragma unroll
            for (int s = 0; s < VEC; ++s) v.v[s] += w * u.v[s];
        }
        s_b[it * groups + g.q] = v;
    }
    __syncthreads();
    // y: -> [c][f][f]
    for (int it = g.on ? g.r : cells * C1 * F1 * F1; it < cells * C1 * F1 * F1; it += g.R) {
        const int ia = it % F1, ib = (it / F1) % F1, row = it / (F1 * F1), cell = row / C1;
        P v{};
#pragma unroll
        for (int j = 0; j < C1; ++j) {
            const T w = T(tab[3 * cell + 1][ib][j]);
            const P u = s_b[((row * C1 + j) * F1 + ia) * groups + g.q];
#pragma unroll
            for (int s = 0; s < VEC; ++s) v.v[s] += w * u.v[s];
        }
        s_a[it * groups + g.q] = v;
    }
    __syncthreads();
    // z, at the owned nodes
    for (int it = g.on ? g.r : cells * NF; it < cells * NF; it += g.R) {
        const int row = a.own_node[f0 * NF + it];
        if (row < 0) continue;
        const int cell = it / NF, n = it - cell * NF, ic = n / (F1 * F1), ab = n - ic * F1 * F1;
        P v = load_pack<T, VEC>(yf, row, groups, g.q);
#pragma unroll
        for (int j = 0; j < C1; ++j) {
            const T w = T(tab[3 * cell + 2][ic][j]);
            const P u = s_a[((cell * C1 + j) * F1 * F1 + ab) * groups + g.q];
#pragma unroll
            for (int s = 0; s < VEC; ++s) v.v[s] += w * u.v[s];
        }
        store_pack<T, VEC>(yf, row, groups, g.q, v);
    }
}

// yc += R (b - ax) = P^T (b - ax) (yc zeroed by the caller), ax cleared for the
// next operator application: the owned interior fine residuals times the
// interpolation weights, one direction at a time, then spread through the
// coarse constraints to interior coarse masters.  With (pf + 1)^3 products per
// coarse node the finest transfer took 1,163 us for 16 columns, with the
// residual's own pass 1,183 us; now 46 us.
template <typename T, int VEC, int PF, int PC>
__global__ void __launch_bounds__(256) pmg_restrict_kernel(const __grid_constant__ XferArgs a,
                                                           const T* __restrict__ b, T* __restrict__ ax,
                                                           T* __restrict__ yc, int cpb, int clear) {
    constexpr int F1 = PF + 1, C1 = PC + 1, NF = F1 * F1 * F1, NC = C1 * C1 * C1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int groups = a.k / VEC;
    const int64_t f0 = int64_t(blockIdx.x) * cpb;
    const int cells = int(min(int64_t(cpb), a.ncell - f0));
    using P = Pack<T, VEC>;
    P* s_a = reinterpret_cast<P*>(smem_raw);            // [cpb][NF] residuals; then [cpb][C1][C1][F1]
    P* s_b = s_a + cpb * NF * groups;                   // [cpb][C1][F1][F1]
    float(*tab)[F1][C1] = reinterpret_cast<float(*)[F1][C1]>(s_b + cpb * C1 * F1 * F1 * groups);
    xfer_tables<PF, PC>(a, f0, cells, tab);
    const ColGroup g(groups);
    for (int it0 = g.on ? g.r : cells * NF; it0 < cells * NF; it0 += 2 * g.R) {   // two rows in flight
        P v[2], u[2];
        int row[2];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int it = it0 + r * g.R;
            row[r] = it < cells * NF ? a.own_node[f0 * NF + it] : -1;
            v[r] = u[r] = P{};
        }
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            if (row[r] < 0) continue;
            v[r] = load_pack<T, VEC>(b, row[r], groups, g.q);
            u[r] = load_pack<T, VEC>(ax, row[r], groups, g.q);
        }
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int it = it0 + r * g.R;
            if (it >= cells * NF) break;
            if (clear && row[r] >= 0) store_pack<T, VEC>(ax, row[r], groups, g.q, P{});
#pragma unroll
            for (int s = 0; s < VEC; ++s) v[r].v[s] -= u[r].v[s];
            s_a[it * groups + g.q] = v[r];
        }
    }
    __syncthreads();
    // z: [f][f][f] -> [c][f][f]
    for (int it = g.on ? g.r : cells * C1 * F1 * F1; it < cells * C1 * F1 * F1; it += g.R) {
        const int ab = it % (F1 * F1), row = it / (F1 * F1), jc = row % C1, cell = row / C1;
        P v{};
#pragma unroll
        for (int i = 0; i < F1; ++i) {
            const T w = T(tab[3 * cell + 2][i][jc]);
            const P u = s_a[(cell * NF + i * F1 * F1 + ab) * groups + g.q];
#pragma unroll
            for (int s = 0; s < VEC; ++s) v.v[s] += w * u.v[s];
        }
        s_b[it * groups + g.q] = v;
    }
    __syncthreads();
    // y: -> [c][c][f]
    for (int it = g.on ? g.r : cells * C1 * C1 * F1; it < cells * C1 * C1 * F1; it += g.R) {
        const int ia = it % F1, row = it / F1, jb = row % C1, cc = row / C1, cell = cc / C1;
        P v{};
#pragma unroll
        for (int i = 0; i < F1; ++i) {
            const T w = T(tab[3 * cell + 1][i][jb]);
            const P u = s_b[((cc * F1 + i) * F1 + ia) * groups + g.q];
#pragma unroll
            for (int s = 0; s < VEC; ++s) v.v[s] += w * u.v[s];
        }
        s_a[it * groups + g.q] = v;
    }
    __syncthreads();
    // x, and into the coarse level
    for (int it = g.on ? g.r : cells * NC; it < cells * NC; it += g.R) {
        const int ja = it % C1, row = it / C1, cell = it / NC;
        P v{};
#pragma unroll
        for (int i = 0; i < F1; ++i) {
            const T w = T(tab[3 * cell][i][ja]);
            const P u = s_a[(row * F1 + i) * groups + g.q];
#pragma unroll
            for (int s = 0; s < VEC; ++s) v.v[s] += w * u.v[s];
        }
        const int idx = a.c_node[int64_t(a.coarse_cell[f0 + cell]) * NC + it - cell * NC];
        auto add = [&](int64_t m, T w) {
            T* y = yc + (m * groups + g.q) * VEC;
            if constexpr (VEC == 4 && sizeof(T) == 4) {
                atomicAdd(reinterpret_cast<float4*>(y), make_float4(w * v.v[0], w * v.v[1], w * v.v[2], w * v.v[3]));
            } else {
#pragma unroll
                for (int s = 0; s < VEC; ++s) atomicAdd(y + s, w * v.v[s]);
            }
        };
        if (idx >= 0) {
            if (idx < a.c_ni) add(idx, T(1));
        } else {
            const int h = -idx - 1;
            for (int e = a.c_hp[h]; e < a.c_hp[h + 1]; ++e)
                if (a.c_hm[e] < a.c_ni) add(a.c_hm[e], T(a.c_hw[e]));
        }
    }
}

// One Chebyshev step on the interior rows: res = b - A x (ax = A x, cleared for
// the next operator application; x = 0 when ax is null), d = c1 d + c2 D^-1 res,
// x += d.  first: d = c2 D^-1 res (d is not read: on the first step it holds
// whatever the workspace held).
template <typename T, int VEC>
__global__ void __launch_bounds__(256) pmg_cheb_kernel(T* __restrict__ x, T* __restrict__ d, const T* __restrict__ b,
                                                       T* __restrict__ ax, const T* __restrict__ dinv, int64_t ni,
                                                       int groups, T c1, T c2, int first, int clear) {
    const ColGroup g(groups);
    if (!g.on) return;
    using P = Pack<T, VEC>;
    for (int64_t row = int64_t(blockIdx.x) * g.R + g.r; row < ni; row += int64_t(gridDim.x) * g.R) {
        // all loads of a row before its stores (which the compiler may not pass)
        const T w = c2 * dinv[row];
        P res = load_pack<T, VEC>(b, row, groups, g.q), t{}, dn{}, xn{};
        if (ax) {
            t = load_pack<T, VEC>(ax, row, groups, g.q);
            xn = load_pack<T, VEC>(x, row, groups, g.q);
        }
        if (!first) dn = load_pack<T, VEC>(d, row, groups, g.q);
#pragma unroll
        for (int s = 0; s < VEC; ++s) {
            dn.v[s] = (first ? T(0) : c1 * dn.v[s]) + w * (res.v[s] - t.v[s]);
            xn.v[s] = ax ? xn.v[s] + dn.v[s] : dn.v[s];
        }
        if (clear) store_pack<T, VEC>(ax, row, groups, g.q, P{});
        store_pack<T, VEC>(d, row, groups, g.q, dn);
        store_pack<T, VEC>(x, row, groups, g.q, xn);
    }
}

// The coarsest level in one launch: degree 1 on the uniform grid of n^3 interior
// nodes, where (quadrature at the nodes) A x = h (6 x - sum of the 6 neighbours)
// and D = 6 h, so a Chebyshev step needs the neighbours only.  One block per
// column keeps x in shared memory (with a ring of zeros, the Dirichlet surface)
// and d, b in registers through all `steps` steps: 30 steps as memset, cell
// pass and update took 30 x 14 us on 6,859 nodes of 16 columns; now 84 us, bound
// by the block's barriers and shared-memory reads (one SM per column).
// steps[2 s], steps[2 s + 1]: c1 and c2 of step s; hd = 1 / (6 h); x0 = 0.
constexpr int kPmgCoarseThreads = 1024;
struct ChebSteps {
    double c[2 * kPmgCoarseDegree];
};
template <typename T, int NPT>
__global__ void __launch_bounds__(kPmgCoarseThreads) pmg_coarse_kernel(const int32_t* __restrict__ map, int n,
                                                                       const T* __restrict__ b, T* __restrict__ x,
                                                                       int k, T hd, const __grid_constant__ ChebSteps st) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* s_x = reinterpret_cast<T*>(smem_raw);   // [(n+2)^3]
    const int np = n + 2, total = n * n * n, col = blockIdx.x;
    for (int i = threadIdx.x; i < np * np * np; i += kPmgCoarseThreads) s_x[i] = T(0);
    T rb[NPT], d[NPT];
    int at[NPT];
#pragma unroll
    for (int j = 0; j < NPT; ++j) {
        const int i = int(threadIdx.x) + j * kPmgCoarseThreads;
        at[j] = -1;
        rb[j] = d[j] = T(0);
        if (i < total) {
            const int ix = i % n, iy = (i / n) % n, iz = i / (n * n);
            at[j] = (ix + 1) + np * ((iy + 1) + np * (iz + 1));
            rb[j] = hd * b[int64_t(map[i]) * k + col];   // D^-1 b
        }
    }
    __syncthreads();
    for (int s = 0; s < kPmgCoarseDegree; ++s) {
        const T c1 = T(st.c[2 * s]), c2 = T(st.c[2 * s + 1]);
#pragma unroll
        for (int j = 0; j < NPT; ++j) {
            if (at[j] < 0) continue;
            const T* q = s_x + at[j];
            const T xc = q[0];
            const T nb = ((q[-1] + q[1]) + (q[-np] + q[np])) + (q[-np * np] + q[np * np]);
            const T res = rb[j] - (xc - nb * T(1.0 / 6.0));   // D^-1 (b - A x)
            d[j] = c1 * d[j] + c2 * res;
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < NPT; ++j)
            if (at[j] >= 0) s_x[at[j]] += d[j];
        __syncthreads();
    }
#pragma unroll
    for (int j = 0; j < NPT; ++j)
        if (at[j] >= 0) x[int64_t(map[int(threadIdx.x) + j * kPmgCoarseThreads]) * k + col] = s_x[at[j]];
}

__device__ __forceinline__ double as_f64(float v) { return widen_f32(v); }
__device__ __forceinline__ double as_f64(double v) { return v; }

// out[c] += sum over interior rows of x[row][c] y[row][c] (FP64 accumulation)
template <typename T, int VEC>
__global__ void __launch_bounds__(256) pmg_coldot_kernel(const T* __restrict__ x, const T* __restrict__ y, int64_t ni,
                                                         int groups, double* __restrict__ out) {
    __shared__ double s[256 * VEC];
    const ColGroup g(groups);
    double acc[VEC];
#pragma unroll
    for (int v = 0; v < VEC; ++v) acc[v] = 0.0;
    if (g.on) {
        for (int64_t row = int64_t(blockIdx.x) * g.R + g.r; row < ni; row += int64_t(gridDim.x) * g.R) {
            const Pack<T, VEC> a = load_pack<T, VEC>(x, row, groups, g.q), b = load_pack<T, VEC>(y, row, groups, g.q);
#pragma unroll
            for (int v = 0; v < VEC; ++v) acc[v] = fma(as_f64(a.v[v]), as_f64(b.v[v]), acc[v]);
        }
    }
#pragma unroll
    for (int v = 0; v < VEC; ++v) s[threadIdx.x * VEC + v] = acc[v];
    __syncthreads();
    const int k = groups * VEC;
    for (int left = g.R; left > 1;) {   // tree over the rows of threads
        const int half = (left + 1) >> 1;
        for (int i = threadIdx.x; i + half * k < left * k; i += blockDim.x) s[i] += s[i + half * k];
        __syncthreads();
        left = half;
    }
    for (int c = threadIdx.x; c < k; c += blockDim.x) atomicAdd(&out[c], s[c]);
}

// p = z + beta p with beta = rz / rz_old per column (0 when rz_old = 0);
// first: p = z (p is not read).
template <typename T, int VEC>
__global__ void __launch_bounds__(256) pmg_pupdate_kernel(T* __restrict__ p, const T* __restrict__ z,
                                                          const double* __restrict__ rz,
                                                          const double* __restrict__ rz_old, int64_t ni, int groups,
                                                          int first) {
    const ColGroup g(groups);
    if (!g.on) return;
    T beta[VEC];
    bool keep[VEC];
#pragma unroll
    for (int v = 0; v < VEC; ++v) {
        const double ro = rz_old[g.q * VEC + v];
        keep[v] = !first && ro > 0.0;
        beta[v] = keep[v] ? T(rz[g.q * VEC + v] / ro) : T(0);
    }
    for (int64_t row = int64_t(blockIdx.x) * g.R + g.r; row < ni; row += int64_t(gridDim.x) * g.R) {
        Pack<T, VEC> zz = load_pack<T, VEC>(z, row, groups, g.q);
        if (!first) {
            const Pack<T, VEC> pp = load_pack<T, VEC>(p, row, groups, g.q);
#pragma unroll
            for (int v = 0; v < VEC; ++v)
                if (keep[v]) zz.v[v] = zz.v[v] + beta[v] * pp.v[v];
        }
        store_pack<T, VEC>(p, row, groups, g.q, zz);
    }
}

// x += alpha p, r -= alpha q with alpha = rz / pq per column (0 when pq <= 0).
template <typename T, int VEC>
__global__ void __launch_bounds__(256) pmg_xr_kernel(T* __restrict__ x, T* __restrict__ r, const T* __restrict__ p,
                                                     const T* __restrict__ q, const double* __restrict__ rz,
                                                     const double* __restrict__ pq, int64_t ni, int groups) {
    const ColGroup g(groups);
    if (!g.on) return;
    T al[VEC];
#pragma unroll
    for (int v = 0; v < VEC; ++v) {
        const double den = pq[g.q * VEC + v];
        al[v] = T(den > 0.0 ? rz[g.q * VEC + v] / den : 0.0);
    }
    for (int64_t row = int64_t(blockIdx.x) * g.R + g.r; row < ni; row += int64_t(gridDim.x) * g.R) {
        Pack<T, VEC> xx = load_pack<T, VEC>(x, row, groups, g.q), rr = load_pack<T, VEC>(r, row, groups, g.q);
        const Pack<T, VEC> pp = load_pack<T, VEC>(p, row, groups, g.q), qq = load_pack<T, VEC>(q, row, groups, g.q);
#pragma unroll
        for (int v = 0; v < VEC; ++v) {
            xx.v[v] += al[v] * pp.v[v];
            rr.v[v] -= al[v] * qq.v[v];
        }
        store_pack<T, VEC>(x, row, groups, g.q, xx);
        store_pack<T, VEC>(r, row, groups, g.q, rr);
    }
}

// W += e on the interior rows (the float32 correction into the float64 solution)
__global__ void pmg_add_f32_kernel(double* __restrict__ W, const float* __restrict__ e, int64_t n) {
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
        W[i] += double(e[i]);
}

// deterministic start vector of the power iteration (interior rows)
__global__ void pmg_seed_kernel(double* __restrict__ x, int64_t ni) {
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < ni; i += int64_t(gridDim.x) * blockDim.x) {
        uint64_t h = uint64_t(i) * 0x9E3779B97F4A7C15ull + 0x632BE59BD9B4E019ull;
        h ^= h >> 31;
        h *= 0xBF58476D1CE4E5B9ull;
        h ^= h >> 29;
        x[i] = 0.5 + double(h >> 11) * (1.0 / 9007199254740992.0);
    }
}

// y = D^-1 y on the interior rows, one column
__global__ void pmg_jacobi_scale_kernel(double* __restrict__ y, const double* __restrict__ dinv, int64_t ni,
                                        double s) {
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < ni; i += int64_t(gridDim.x) * blockDim.x)
        y[i] = s * dinv[i] * y[i];
}

__global__ void pmg_f64_to_f32_kernel(const double* __restrict__ x, float* __restrict__ y, int64_t n) {
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
        y[i] = float(x[i]);
}

// r = b - t - ax on the interior rows (FP64 residual of the full system with
// the surface data: t = A g_ext, ax = A_II W_I)
__global__ void pmg_residual64_kernel(double* __restrict__ r, const double* __restrict__ b,
                                      const double* __restrict__ t, const double* __restrict__ ax, int64_t ni,
                                      int k) {
    const int64_t n = ni * k;
    for (int64_t o = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; o < n; o += int64_t(gridDim.x) * blockDim.x)
        r[o] = b[o] - t[o] - ax[o];
}

// --------------------------------------------------------------- host parts
// Whether the consumers of A x clear it for the next application (one launch
// less; the vectors of a small level stay in L2) or the application does: with
// 50 MB vectors a Chebyshev step that also clears takes 145-172 us instead of
// 40 and a memset of 12, so the line is drawn at 8 MB.
template <typename T>
static bool clear_in_pass(const afem_mesh* m, int k) {
    return size_t(m->dev.n_master) * k * sizeof(T) <= (size_t(8) << 20);
}
// y = A x on the interior
template <typename T>
static int stiff(const afem_mesh* m, const T* x, T* y, int k, cudaStream_t s);
template <>
int stiff<double>(const afem_mesh* m, const double* x, double* y, int k, cudaStream_t s) {
    return launch_stiffness(m, x, y, k, 1, s, clear_in_pass<double>(m, k));
}
template <>
int stiff<float>(const afem_mesh* m, const float* x, float* y, int k, cudaStream_t s) {
    return launch_stiffness32(m, x, y, k, 1, s, nullptr, clear_in_pass<float>(m, k));
}
// Columns per thread of the vector kernels: a 16-byte word where k allows it.
template <typename T>
static bool packed(int k) {
    return k % int(16 / sizeof(T)) == 0;
}
template <typename T, typename F>
static auto with_pack(int k, F&& f) {
    return packed<T>(k) ? f(std::integral_constant<int, int(16 / sizeof(T))>()) : f(std::integral_constant<int, 1>());
}
// Blocks of a vector kernel over `rows` rows of `groups` column groups.
static unsigned rows_grid(int64_t rows, int groups, int per_sm = 8) {
    const int R = 256 / groups;
    const int64_t g = (rows + R - 1) / R;
    return unsigned(std::max<int64_t>(1, std::min<int64_t>(g, int64_t(per_sm) * device_sms())));
}
template <typename T>
static void coldot(const T* x, const T* y, int64_t ni, int k, double* out, cudaStream_t s) {
    with_pack<T>(k, [&](auto V) {
        constexpr int VEC = decltype(V)::value;
        AFEM_LAUNCH((pmg_coldot_kernel<T, VEC>), rows_grid(ni, k / VEC, 4), 256, 0, s, x, y, ni, k / VEC, out);
        return 0;
    });
}
template <typename T>
static void pupdate(T* p, const T* z, const double* rz, const double* rz_old, int64_t ni, int k, int first,
                    cudaStream_t s) {
    with_pack<T>(k, [&](auto V) {
        constexpr int VEC = decltype(V)::value;
        AFEM_LAUNCH((pmg_pupdate_kernel<T, VEC>), rows_grid(ni, k / VEC), 256, 0, s, p, z, rz, rz_old, ni, k / VEC,
                    first);
        return 0;
    });
}
template <typename T>
static void xr_update(T* x, T* r, const T* p, const T* q, const double* rz, const double* pq, int64_t ni, int k,
                      cudaStream_t s) {
    // (x is the caller's array in the FP64 form: any 8-byte alignment)
    with_pack<T>((reinterpret_cast<uintptr_t>(x) & 15) == 0 ? k : 1, [&](auto V) {
        constexpr int VEC = decltype(V)::value;
        AFEM_LAUNCH((pmg_xr_kernel<T, VEC>), rows_grid(ni, k / VEC), 256, 0, s, x, r, p, q, rz, pq, ni, k / VEC);
        return 0;
    });
}
template <typename T>
static const T* dinv_of(const afem_mesh* m);
template <>
const double* dinv_of<double>(const afem_mesh* m) {
    return m->dev.stiff_dinv;
}
template <>
const float* dinv_of<float>(const afem_mesh* m) {
    return m->dev.stiff_dinv32;
}

static XferArgs xfer_args(const PmgLevel& F, const PmgLevel& C, int k) {
    XferArgs a{};
    const DeviceMesh& fd = F.mesh->dev;
    const DeviceMesh& cd = C.mesh->dev;
    a.coarse_cell = F.coarse_cell;
    a.xform = F.xform;
    a.own_node = F.own_node;
    a.ncell = fd.ncell;
    for (int i = 0; i <= fd.p; ++i) a.xi_f[i] = float(F.mesh->basis.xi[i]);
    a.c_node = cd.cell_node;
    a.c_hp = cd.hang_ptr;
    a.c_hm = cd.hang_master;
    a.c_hw = cd.hang_w;
    a.c_ni = cd.n_interior;
    a.k = k;
    return a;
}

// Vectors of one level: x (solution), b (right-hand side), t (A x; zero
// between its uses), d (Chebyshev direction).
template <typename T>
struct LevelVec {
    T *x, *t, *d;
    T* b;
};

// c1, c2 of `deg` Chebyshev steps on [lo, hi].
static void cheb_steps(double lo, double hi, int deg, double* c) {
    const double theta = 0.5 * (hi + lo), delta = 0.5 * (hi - lo), sigma = theta / delta;
    double rho = 1.0 / sigma;
    for (int it = 0; it < deg; ++it) {
        if (it == 0) {
            c[0] = 0.0;
            c[1] = 1.0 / theta;
        } else {
            const double rho_new = 1.0 / (2.0 * sigma - rho);
            c[2 * it] = rho_new * rho;
            c[2 * it + 1] = 2.0 * rho_new / delta;
            rho = rho_new;
        }
    }
}

// Chebyshev smoothing of A x = b on [lo, hi] (eigenvalues of D^-1 A), `deg`
// steps, from x = 0 (zero_start) or the current x.
template <typename T>
static int chebyshev(const afem_mesh* m, LevelVec<T>& v, int k, double lo, double hi, int deg, bool zero_start,
                     cudaStream_t s) {
    const int64_t ni = m->dev.n_interior;
    if (ni == 0) return AFEM_OK;
    const T* dinv = dinv_of<T>(m);
    double c[2 * kPmgCoarseDegree];
    cheb_steps(lo, hi, deg, c);
    int rc;
    for (int it = 0; it < deg; ++it) {
        const bool x_zero = zero_start && it == 0;
        if (!x_zero && (rc = stiff<T>(m, v.x, v.t, k, s))) return rc;
        with_pack<T>(k, [&](auto V) {
            constexpr int VEC = decltype(V)::value;
            AFEM_LAUNCH((pmg_cheb_kernel<T, VEC>), rows_grid(ni, k / VEC), 256, 0, s, v.x, v.d, v.b,
                        x_zero ? static_cast<T*>(nullptr) : v.t, dinv, ni, k / VEC, T(c[2 * it]), T(c[2 * it + 1]),
                        it == 0 ? 1 : 0, (!x_zero && clear_in_pass<T>(m, k)) ? 1 : 0);
            return 0;
        });
    }
    AFEM_CUDA_TRY(cudaGetLastError());
    return AFEM_OK;
}

// The coarsest level's polynomial in one launch, where its grid fits a block.
template <typename T, int NPT>
static int coarse_solve_npt(const PmgLevel& L, LevelVec<T>& v, int k, const ChebSteps& st, cudaStream_t s) {
    const int n = L.grid_n;
    const double h = (L.mesh->desc.hi - L.mesh->desc.lo) / (n + 1);
    AFEM_CUDA_TRY(allow_dyn_smem(pmg_coarse_kernel<T, NPT>));
    AFEM_LAUNCH((pmg_coarse_kernel<T, NPT>), unsigned(k), kPmgCoarseThreads,
                size_t(n + 2) * (n + 2) * (n + 2) * sizeof(T), s, L.grid_map, n, v.b, v.x, k, T(1.0 / (6.0 * h)), st);
    AFEM_CUDA_TRY(cudaGetLastError());
    return AFEM_OK;
}
template <typename T>
static bool coarse_fits(const PmgLevel& L) {   // 16 (float) or 8 (double) nodes a thread keep to 64 registers
    return L.grid_n > 0 && L.grid_n * L.grid_n * L.grid_n <= kPmgCoarseThreads * (sizeof(T) == 4 ? 16 : 8);
}
template <typename T>
static int coarse_solve(const PmgLevel& L, LevelVec<T>& v, int k, double lo, double hi, cudaStream_t s) {
    ChebSteps st;
    cheb_steps(lo, hi, kPmgCoarseDegree, st.c);
    const int total = L.grid_n * L.grid_n * L.grid_n;
    if (total <= kPmgCoarseThreads) return coarse_solve_npt<T, 1>(L, v, k, st, s);
    if (total <= 8 * kPmgCoarseThreads) return coarse_solve_npt<T, 8>(L, v, k, st, s);
    if constexpr (sizeof(T) == 4) return coarse_solve_npt<T, 16>(L, v, k, st, s);
    return set_error(AFEM_EINVAL, "multigrid: coarse grid out of range");
}

// Transfers between level F (degree PF) and the next coarser level (degree PC).
template <typename T, int PF, int PC>
static int restrict_to(const PmgLevel& F, const PmgLevel& C, const T* b, T* ax, T* yc, int k, cudaStream_t s) {
    const XferArgs a = xfer_args(F, C, k);
    return with_pack<T>(k, [&](auto V) -> int {
        constexpr int VEC = decltype(V)::value, F1 = PF + 1, C1 = PC + 1;
        const int groups = k / VEC, cpb = xfer_cells(PF, groups);
        const size_t smem = size_t(cpb) * groups * (F1 * F1 * F1 + C1 * F1 * F1) * sizeof(T) * VEC +
                            size_t(cpb) * 3 * F1 * C1 * sizeof(float);
        AFEM_CUDA_TRY(allow_dyn_smem(pmg_restrict_kernel<T, VEC, PF, PC>));
        AFEM_LAUNCH((pmg_restrict_kernel<T, VEC, PF, PC>), unsigned((a.ncell + cpb - 1) / cpb), 256, smem, s, a, b, ax,
                    yc, cpb, clear_in_pass<T>(F.mesh, k) ? 1 : 0);
        AFEM_CUDA_TRY(cudaGetLastError());
        return AFEM_OK;
    });
}
template <typename T, int PF, int PC>
static int prolong_from(const PmgLevel& F, const PmgLevel& C, const T* xc, T* yf, int k, cudaStream_t s) {
    const XferArgs a = xfer_args(F, C, k);
    return with_pack<T>(k, [&](auto V) -> int {
        constexpr int VEC = decltype(V)::value, F1 = PF + 1, C1 = PC + 1;
        const int groups = k / VEC, cpb = xfer_cells(PF, groups);
        const size_t smem = size_t(cpb) * groups * (C1 * F1 * F1 + C1 * C1 * F1) * sizeof(T) * VEC +
                            size_t(cpb) * 3 * F1 * C1 * sizeof(float);
        AFEM_CUDA_TRY(allow_dyn_smem(pmg_prolong_kernel<T, VEC, PF, PC>));
        AFEM_LAUNCH((pmg_prolong_kernel<T, VEC, PF, PC>), unsigned((a.ncell + cpb - 1) / cpb), 256, smem, s, a, xc, yf,
                    cpb);
        AFEM_CUDA_TRY(cudaGetLastError());
        return AFEM_OK;
    });
}
// The degree pairs of the hierarchy (4 -> 2 -> 1, 3 -> 1, 2 -> 1, 1 -> 1).
#define AFEM_XFER(FN, T, F, C, ...)                                                          \
    ((F).mesh->dev.p == 4 ? FN<T, 4, 2>(F, C, __VA_ARGS__)                                   \
     : (F).mesh->dev.p == 3 ? FN<T, 3, 1>(F, C, __VA_ARGS__)                                 \
     : (F).mesh->dev.p == 2 ? FN<T, 2, 1>(F, C, __VA_ARGS__) : FN<T, 1, 1>(F, C, __VA_ARGS__))

// z = V(l) b on level l (v[l].b holds b; the result is left in v[l].x).
template <typename T>
static int vcycle(afem_pmg* g, std::vector<LevelVec<T>>& v, int l, int k, cudaStream_t s) {
    PmgLevel& L = g->lv[l];
    const afem_mesh* m = L.mesh;
    int rc;
    if (l + 1 == int(g->lv.size())) {
        const double hi = L.lam_max * kPmgLambdaSafety, lo = hi / kPmgCoarseRange;
        if (coarse_fits<T>(L)) return coarse_solve<T>(L, v[l], k, lo, hi, s);
        return chebyshev<T>(m, v[l], k, lo, hi, kPmgCoarseDegree, true, s);
    }
    const double hi = L.lam_max * kPmgLambdaSafety, lo = hi / kPmgSmoothRange;
    if ((rc = chebyshev<T>(m, v[l], k, lo, hi, kPmgPreDegree, true, s))) return rc;
    // coarse right-hand side R (b - A x)
    if ((rc = stiff<T>(m, v[l].x, v[l].t, k, s))) return rc;
    PmgLevel& C = g->lv[l + 1];
    AFEM_CUDA_TRY(cudaMemsetAsync(v[l + 1].b, 0, size_t(C.mesh->dev.n_master) * k * sizeof(T), s));
    if ((rc = AFEM_XFER(restrict_to, T, L, C, v[l].b, v[l].t, v[l + 1].b, k, s))) return rc;
    if ((rc = vcycle<T>(g, v, l + 1, k, s))) return rc;
    if ((rc = AFEM_XFER(prolong_from, T, L, C, v[l + 1].x, v[l].x, k, s))) return rc;
    return chebyshev<T>(m, v[l], k, lo, hi, kPmgPreDegree, false, s);
}

// Largest eigenvalue of D^-1 A_II of a level by power iteration (FP64, one
// column): x_hat = x / ||x||, x <- D^-1 A x_hat, lambda ~ ||x||.
static int estimate_lambda(afem_mesh* m, double* lam, cudaStream_t s) {
    const int64_t N = m->dev.n_master, ni = m->dev.n_interior;
    *lam = 1.0;
    if (ni == 0) return AFEM_OK;
    double *x = nullptr, *y = nullptr, *acc = nullptr;
    cudaError_t e = cudaMalloc(&x, N * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc(&y, N * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc(&acc, sizeof(double));
    int rc = e == cudaSuccess ? AFEM_OK : set_error(AFEM_ENOMEM, "multigrid set-up: cudaMalloc failed");
    auto norm = [&](const double* v, double* out) -> int {
        AFEM_CUDA_TRY(cudaMemsetAsync(acc, 0, sizeof(double), s));
        coldot<double>(v, v, ni, 1, acc, s);
        double h = 0.0;
        AFEM_CUDA_TRY(cudaMemcpyAsync(&h, acc, sizeof(double), cudaMemcpyDeviceToHost, s));
        AFEM_CUDA_TRY(cudaStreamSynchronize(s));
        *out = std::sqrt(h);
        return AFEM_OK;
    };
    double nx = 0.0, est = 0.0;
    if (rc == AFEM_OK) {
        if (cudaMemsetAsync(x, 0, N * sizeof(double), s) != cudaSuccess) rc = set_error(AFEM_ECUDA, "memset");
        else {
            AFEM_LAUNCH((pmg_seed_kernel), grid_for(ni), 256, 0, s, x, ni);
            rc = norm(x, &nx);
        }
    }
    for (int it = 0; rc == AFEM_OK && it < kPmgPowerIters && nx > 0.0 && std::isfinite(nx); ++it) {
        if ((rc = launch_stiffness(m, x, y, 1, 1, s))) break;
        AFEM_LAUNCH((pmg_jacobi_scale_kernel), grid_for(ni), 256, 0, s, y, m->dev.stiff_dinv, ni, 1.0 / nx);
        if ((rc = norm(y, &est))) break;
        std::swap(x, y);
        nx = est;
    }
    if (rc == AFEM_OK && est > 0.0 && std::isfinite(est)) *lam = est;
    cudaFree(x);
    cudaFree(y);
    cudaFree(acc);
    return rc;
}

// Builds the level hierarchy of mesh m (once).
static int pmg_setup(afem_mesh* m, cudaStream_t s) {
    if (m->pmg) return AFEM_OK;
    auto* g = new (std::nothrow) afem_pmg();
    if (!g) return set_error(AFEM_ENOMEM, "multigrid set-up: out of host memory");
    PmgLevel top;
    top.mesh = m;
    g->lv.push_back(top);
    int rc = AFEM_OK;
    // p-coarsening on the same leaves, then degree 1 on the leaves truncated at
    // levels Lf-1, ..., 0 (every leaf finer than the cap replaced by its
    // ancestor at the cap): each level's octree coarsens the previous one
    const HostMesh& F = m->host;
    const int Lf = F.max_level;
    std::vector<int> degrees;
    for (int p = m->desc.degree; p > 1;) {
        p = p >= 4 ? p / 2 : 1;
        degrees.push_back(p);
    }
    auto add_level = [&](int degree, int cap) -> int {
        afem_mesh_desc e = m->desc;
        e.degree = degree;
        std::vector<int32_t> lev, ci, cj, ck;
        std::unordered_set<uint64_t> seen;
        for (size_t q = 0; q < F.lev.size(); ++q) {
            const int sh = F.lev[q] > cap ? F.lev[q] - cap : 0;
            const int32_t l = F.lev[q] - sh, i = F.ci[q] >> sh, j = F.cj[q] >> sh, k = F.ck[q] >> sh;
            const uint64_t key = (uint64_t(l) << 60) | (uint64_t(i) << 40) | (uint64_t(j) << 20) | uint64_t(k);
            if (!seen.insert(key).second) continue;
            lev.push_back(l);
            ci.push_back(i);
            cj.push_back(j);
            ck.push_back(k);
        }
        afem_mesh* lm = nullptr;
        int r = create_mesh_from_cells(e, lev, ci, cj, ck, &lm);
        if (r) return r;
        PmgLevel L;
        L.mesh = lm;
        L.owned = true;
        g->lv.push_back(L);
        return AFEM_OK;
    };
    for (int p : degrees)
        if (rc == AFEM_OK) rc = add_level(p, Lf);
    for (int cap = Lf - 1; rc == AFEM_OK && cap >= 0; --cap) rc = add_level(1, cap);
    for (size_t l = 0; rc == AFEM_OK && l + 1 < g->lv.size(); ++l)
        rc = build_transfer(g->lv[l].mesh->host, g->lv[l + 1].mesh->host, g->lv[l]);
    if (rc == AFEM_OK) rc = build_grid_map(g->lv.back());
    for (size_t l = 0; rc == AFEM_OK && l < g->lv.size(); ++l) rc = estimate_lambda(g->lv[l].mesh, &g->lv[l].lam_max, s);
    if (rc) {
        pmg_free(g);
        return rc;
    }
    m->pmg = g;
    return AFEM_OK;
}

template <typename T>
static int carve_levels(afem_pmg* g, int k, std::vector<LevelVec<T>>& v, Carver& cv) {
    v.resize(g->lv.size());
    for (size_t l = 0; l < g->lv.size(); ++l) {
        const size_t NK = size_t(g->lv[l].mesh->dev.n_master) * k;
        v[l].x = cv.take<T>(NK);
        v[l].b = l > 0 ? cv.take<T>(NK) : nullptr;   // the finest level's is the caller's residual
        v[l].t = cv.take<T>(NK);
        v[l].d = cv.take<T>(NK);
    }
    return AFEM_OK;
}
// A x of every level cleared (its users clear it again).
template <typename T>
static int clear_levels(afem_pmg* g, int k, std::vector<LevelVec<T>>& v, cudaStream_t s) {
    for (size_t l = 0; l < g->lv.size(); ++l)
        AFEM_CUDA_TRY(cudaMemsetAsync(v[l].t, 0, size_t(g->lv[l].mesh->dev.n_master) * k * sizeof(T), s));
    return AFEM_OK;
}

}  // namespace afem

namespace afem {

// The batched Poisson solve with the multigrid preconditioner.  mixed = 0:
// CG in float64 with the float64 V-cycle; mixed = 1: float64 defect
// correction, each correction `inner` float32 CG iterations with the float32
// V-cycle.  Stopping test per column: ||b - A_IB g - A_II W_I|| <= rtol ||b - A_IB g||.
int poisson_batch_mg(afem_mesh* m, const double2* phi, int n, double* W, double rtol, int max_it, int warm, int mixed,
                     int* iters_out, int* outer_out, double* relres_out, cudaStream_t s) {
    int rc = pmg_setup(m, s);
    if (rc) return rc;
    afem_pmg* g = m->pmg;
    const DeviceMesh& D = m->dev;
    const int k = n * n;
    const int64_t N = D.n_master, Ni = D.n_interior;
    const size_t NK = size_t(N) * k;
    const int nq = kMultipoleTerms;
    double *b, *t, *r, *z64, *p64, *q64, *qpart, *q, *red;
    float *r32, *e32, *p32, *q32;
    std::vector<LevelVec<double>> v64;
    std::vector<LevelVec<float>> v32;
    const int mb = mom_blocks_count();
    auto carve = [&](Carver& cv) {
        b = cv.take<double>(NK);
        t = cv.take<double>(NK);
        r = cv.take<double>(NK);
        z64 = cv.take<double>(NK);
        p64 = cv.take<double>(mixed ? 0 : NK);
        q64 = cv.take<double>(mixed ? 0 : NK);
        qpart = cv.take<double>(size_t(mb) * nq * k);
        q = cv.take<double>(size_t(nq) * k);
        red = cv.take<double>(size_t(8) * k);
        r32 = cv.take<float>(mixed ? NK : 0);
        e32 = cv.take<float>(mixed ? NK : 0);
        p32 = cv.take<float>(mixed ? NK : 0);
        q32 = cv.take<float>(mixed ? NK : 0);
        if (mixed) carve_levels<float>(g, k, v32, cv);
        else carve_levels<double>(g, k, v64, cv);
    };
    Carver measure(nullptr);
    carve(measure);
    if ((rc = g->ws.reserve(measure.size()))) return rc;
    Carver cv(g->ws.ptr);
    carve(cv);
    double* rz = red;            // r.z
    double* rz_old = red + k;
    double* pq = red + 2 * k;
    double* rr = red + 3 * k;    // r.r
    double* bb = red + 4 * k;    // ||b - A_IB g||^2
    const unsigned gk = grid_for(Ni * k);

    if (!warm) AFEM_CUDA_TRY(cudaMemsetAsync(W, 0, NK * sizeof(double), s));
    if ((rc = poisson_rhs_bc(m, phi, n, W, b, qpart, q, s))) return rc;
    // t = A g_ext (the surface data alone): W with its interior rows cleared
    AFEM_CUDA_TRY(cudaMemcpyAsync(z64, W, NK * sizeof(double), cudaMemcpyDeviceToDevice, s));
    AFEM_CUDA_TRY(cudaMemsetAsync(z64, 0, size_t(Ni) * k * sizeof(double), s));
    if ((rc = launch_stiffness(m, z64, t, k, 0, s))) return rc;
    // ||b - A_IB g||^2 per column (r as scratch)
    AFEM_CUDA_TRY(cudaMemsetAsync(z64, 0, NK * sizeof(double), s));
    AFEM_LAUNCH((pmg_residual64_kernel), gk, 256, 0, s, r, b, t, z64, Ni, k);
    AFEM_CUDA_TRY(cudaMemsetAsync(red, 0, size_t(8) * k * sizeof(double), s));
    coldot<double>(r, r, Ni, k, bb, s);
    std::vector<double> hb(k), hr(k);
    AFEM_CUDA_TRY(cudaMemcpyAsync(hb.data(), bb, k * sizeof(double), cudaMemcpyDeviceToHost, s));
    AFEM_CUDA_TRY(cudaStreamSynchronize(s));

    // FP64 residual r of the current W, its squared norms into hr, the columns above rtol into active
    int active = 0;
    auto count_active = [&]() {
        active = 0;
        for (int c = 0; c < k; ++c)
            if (hr[c] > rtol * rtol * hb[c]) ++active;
    };
    auto residual = [&]() -> int {
        int r_;
        if ((r_ = launch_stiffness(m, W, z64, k, 1, s))) return r_;
        AFEM_LAUNCH((pmg_residual64_kernel), gk, 256, 0, s, r, b, t, z64, Ni, k);
        AFEM_CUDA_TRY(cudaMemsetAsync(rr, 0, k * sizeof(double), s));
        coldot<double>(r, r, Ni, k, rr, s);
        AFEM_CUDA_TRY(cudaMemcpyAsync(hr.data(), rr, k * sizeof(double), cudaMemcpyDeviceToHost, s));
        AFEM_CUDA_TRY(cudaStreamSynchronize(s));
        count_active();
        return AFEM_OK;
    };
    int it = 0, outer = 0;
    if ((rc = residual())) return rc;
    const int inner = 6;   // float32 CG iterations per correction
    if (!mixed) {
        // float64 CG with the float64 V-cycle; restarted from the true residual
        // whenever the recursively updated one meets rtol (or after 64 iterations)
        std::vector<LevelVec<double>>& v = v64;
        v[0].b = r;
        if ((rc = clear_levels<double>(g, k, v, s))) return rc;
        while (active > 0 && it < max_it) {
            ++outer;
            for (int j = 0; j < 64 && active > 0 && it < max_it; ++j, ++it) {
                if ((rc = vcycle<double>(g, v, 0, k, s))) return rc;
                AFEM_CUDA_TRY(cudaMemcpyAsync(rz_old, rz, k * sizeof(double), cudaMemcpyDeviceToDevice, s));
                AFEM_CUDA_TRY(cudaMemsetAsync(rz, 0, k * sizeof(double), s));
                coldot<double>(r, v[0].x, Ni, k, rz, s);
                pupdate<double>(p64, v[0].x, rz, rz_old, Ni, k, j == 0 ? 1 : 0, s);
                if ((rc = launch_stiffness(m, p64, q64, k, 1, s))) return rc;
                AFEM_CUDA_TRY(cudaMemsetAsync(pq, 0, k * sizeof(double), s));
                coldot<double>(p64, q64, Ni, k, pq, s);
                xr_update<double>(W, r, p64, q64, rz, pq, Ni, k, s);
                AFEM_CUDA_TRY(cudaMemsetAsync(rr, 0, k * sizeof(double), s));
                coldot<double>(r, r, Ni, k, rr, s);
                AFEM_CUDA_TRY(cudaMemcpyAsync(hr.data(), rr, k * sizeof(double), cudaMemcpyDeviceToHost, s));
                AFEM_CUDA_TRY(cudaStreamSynchronize(s));
                count_active();
            }
            if ((rc = residual())) return rc;
        }
    } else {
        std::vector<LevelVec<float>>& v = v32;
        v[0].b = r32;
        if ((rc = clear_levels<float>(g, k, v, s))) return rc;
        while (active > 0 && it < max_it) {
            // correction: `inner` float32 CG iterations on A_II e = r from e = 0
            AFEM_LAUNCH((pmg_f64_to_f32_kernel), gk, 256, 0, s, r, r32, int64_t(Ni) * k);
            AFEM_CUDA_TRY(cudaMemsetAsync(e32, 0, NK * sizeof(float), s));
            for (int j = 0; j < inner && it < max_it; ++j, ++it) {
                if ((rc = vcycle<float>(g, v, 0, k, s))) return rc;
                AFEM_CUDA_TRY(cudaMemcpyAsync(rz_old, rz, k * sizeof(double), cudaMemcpyDeviceToDevice, s));
                AFEM_CUDA_TRY(cudaMemsetAsync(rz, 0, k * sizeof(double), s));
                coldot<float>(r32, v[0].x, Ni, k, rz, s);
                pupdate<float>(p32, v[0].x, rz, rz_old, Ni, k, j == 0 ? 1 : 0, s);
                if ((rc = launch_stiffness32(m, p32, q32, k, 1, s, nullptr))) return rc;
                AFEM_CUDA_TRY(cudaMemsetAsync(pq, 0, k * sizeof(double), s));
                coldot<float>(p32, q32, Ni, k, pq, s);
                xr_update<float>(e32, r32, p32, q32, rz, pq, Ni, k, s);
            }
            AFEM_CUDA_TRY(cudaGetLastError());
            // W += e (float64), then the float64 residual decides
            AFEM_LAUNCH((pmg_add_f32_kernel), gk, 256, 0, s, W, e32, int64_t(Ni) * k);
            ++outer;
            if ((rc = residual())) return rc;
        }
    }
    if (iters_out) *iters_out = it;
    if (outer_out) *outer_out = outer;
    bool finite = true;
    for (int c = 0; c < k; ++c) {
        const double rel = hb[c] > 0.0 ? std::sqrt(hr[c] / hb[c]) : 0.0;
        if (!std::isfinite(rel)) finite = false;
        if (relres_out) relres_out[c] = rel;
    }
    if (!finite) return set_error(AFEM_ENAN, "afem_poisson_batch: non-finite residual");
    if (active > 0) return set_error(AFEM_ECG_MAXIT, "afem_poisson_batch: CG reached max_it before rtol");
    return AFEM_OK;
}

}  // namespace afem

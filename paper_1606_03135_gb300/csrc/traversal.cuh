// traversal.cuh -- device code of the traversal and of the own-stencil solves, instantiated in
// assemble.cu (saddle-point factorizations) and nullspace.cu (null-space solves): local systems,
// factorizations, refinement, and the persistent kernels that run them.  assemble.cu describes
// the traversal, nullspace.cuh the null-space solve.
#pragma once
#include <cuda_runtime.h>

#include "fp64_int.cuh"
#include "nullspace.cuh"
#include "rbffd_internal.cuh"

namespace rbffd {

constexpr int kNT = 128;     // default stencil team: one warp per SM sub-partition
constexpr int kMaxNT = 512;  // largest team (big systems, when few fit in shared memory)
constexpr int kMidNT = 256;  // fallback solves with two to four systems per SM
// Device code is compiled for a team size NT of 128 (small systems, many per SM) or 512
// (large systems, one or a few per SM); the LDL^T traversal also for 96, 64 and 32 (one warp
// per stencil), the fallback solves also for 256 (two to four systems per SM).  The host
// picks the instantiation per launch.

// CTAs per SM the register allocation must allow for a team size (the shared-memory limit of
// small systems): 40 registers for 96- and 128-thread teams, 64 for 32-, 64- and 256-thread
// teams.
__host__ __device__ constexpr int team_min_blocks(int nt) {
    return nt == 32 ? 32 : (nt == 64 ? 16 : (nt == 96 ? 16 : (nt == 128 ? 12 : (nt == 256 ? 4 : 1))));
}

// Layouts of a local system: the full matrix (LU), the packed lower triangle (LDL^T), the null
// space of the constraints (nullspace.cuh).
constexpr int kFull = kLayFull, kPacked = kLayPacked, kNull = kLayNull;

// As above for the null-space solves: their products keep 16 words of sums and 16 of operands in
// registers per thread.
__host__ __device__ constexpr int null_min_blocks(int nt) {
    return nt == 32 ? 16 : (nt == 64 ? 12 : (nt == 96 ? 10 : (nt == 128 ? 8 : (nt == 256 ? 4 : 1))));
}
__host__ __device__ constexpr int min_blocks(int lay, int nt) {
    return lay == kNull ? null_min_blocks(nt) : team_min_blocks(nt);
}

// Per-CTA shared-memory views of one local system.  Two layouts of the saddle-point system:
//   full   (LU):     A is K x S row-major holding [A_hat | B_hat]; X = A + K, xs = S
//   packed (LDL^T):  T holds the lower triangle of A_hat by rows (row i starts at i(i+1)/2);
//                    X is the K x q right-hand-side block with row stride xs (odd)
struct StencilSmem {
    double* A;
    double* T;
    double* X;
    int xs;
    double* xi;     // n x D scaled stencil coordinates
    double* rdiag;  // K reciprocal pivots (LDL^T: 1x1 reciprocal; for a 2x2 block at rows p,
                    //   p+1 the inverse's entry 00 at p and entry 11 at p+1)
    double* dinv1;  // K  LDL^T 2x2 inverse entry 01 (at the block's first row)
    double* wv;     // K  unscaled pivot column(s) of the current LDL^T step
    double* wv2;    // K
    int* perm;      // K  original unknown held by each row (symmetric pivoting)
    int* rowof;     // K  row holding each original unknown
    unsigned char* pk;  // K  1: 1x1 pivot, 2: first row of a 2x2 pivot, 0: its second row
    double* lam;    // qmax Lebesgue values of the solved columns (all chunks)
    int* cols;      // qmax ball position of each solved column
    int* colof;     // n column of each ball position, or -1
    unsigned char* keep;  // qmax kept-for-coverage flags
};

// Squared distance of two scaled stencil nodes inside a local system, with FMA:
// fma(t_D, t_D, ... fma(t_1, t_1, t_0 t_0)), t_c = a_c - b_c (6 FP64 operations in 3D instead
// of 8).  Symmetric in a and b (b - a = -(a - b) exactly).  Only the local systems of plans
// that refine nothing use it (a.fma_r2): ill-conditioned systems amplify its different
// rounding, so plans that refine keep sqdist_rn (no FMA, as the oracle forms it), and so do
// the stencils, balls and every structural comparison.
template <int D>
__device__ __forceinline__ double sqdist_local(const double* a, const double* b) {
    double t = __dsub_rn(a[0], b[0]);
    double s = __dmul_rn(t, t);
#pragma unroll
    for (int c = 1; c < D; ++c) {
        t = __dsub_rn(a[c], b[c]);
        s = __fma_rn(t, t, s);
    }
    return s;
}

// Monomial basis tables in shared memory (built on the host in graded order):
//   psi_l = psi_parent[l] * xi_var[l]            (l >= 1; psi_0 = 1)
//   Laplacian psi_l = sum_a lap_coef[l][a] * psi_lap_child[l][a]
struct Basis {
    const short* parent;
    const short* var;
    const short* lap_child;
    const short* lap_coef;
};

// The parameters of one stencil: size n, monomials M, system size K = n + M, PHS exponent m,
// right-hand-side factor m (m + D - 2) and the basis tables of its degree.
struct Shape {
    int n, M, K, m, ell;
    double coef;
    Basis bs;
};

template <int D>
__device__ __forceinline__ Shape shape_of(const SolveArgs& a, const short* sbasis, int j) {
    const int ell = a.node_ell ? (int)a.node_ell[j] : a.ell;
    Shape s;
    s.ell = ell;
    s.n = a.node_n ? a.node_n[j] : a.n;
    s.M = a.Mof[ell];
    s.K = s.n + s.M;
    s.m = a.node_m ? (int)a.node_m[j] : a.m;
    s.coef = exact_double(s.m * (s.m + D - 2));
    const short* b = sbasis + a.boff[ell];
    s.bs.parent = b;
    s.bs.var = b + s.M;
    s.bs.lap_child = b + 2 * s.M;
    s.bs.lap_coef = b + 2 * s.M + s.M * D;
    return s;
}

template <int D, bool PACKED>
__device__ __forceinline__ void carve(char* p, int n, int K, int qmax, int S, StencilSmem& sm) {
    if (PACKED) {
        sm.A = nullptr;
        sm.T = reinterpret_cast<double*>(p);
        p += ((size_t)tri(K) + 1) / 2 * 2 * 8;
        sm.X = reinterpret_cast<double*>(p);
        sm.xs = S;
        p += (size_t)K * S * 8;
    } else {
        sm.A = reinterpret_cast<double*>(p);
        sm.T = nullptr;
        sm.X = sm.A + K;
        sm.xs = S;
        p += (size_t)K * S * 8;
    }
    sm.xi = reinterpret_cast<double*>(p);
    p += (size_t)n * D * 8;
    sm.rdiag = reinterpret_cast<double*>(p);
    p += (size_t)K * 8;
    sm.dinv1 = reinterpret_cast<double*>(p);
    p += (size_t)K * 8;
    sm.wv = reinterpret_cast<double*>(p);
    p += (size_t)K * 8;
    sm.wv2 = reinterpret_cast<double*>(p);
    p += (size_t)K * 8;
    sm.lam = reinterpret_cast<double*>(p);
    p += (size_t)qmax * 8;
    sm.cols = reinterpret_cast<int*>(p);
    p += (size_t)qmax * 4;
    sm.colof = reinterpret_cast<int*>(p);
    p += (size_t)n * 4;
    sm.perm = reinterpret_cast<int*>(p);
    p += (size_t)K * 4;
    sm.rowof = reinterpret_cast<int*>(p);
    p += (size_t)K * 4;
    sm.pk = reinterpret_cast<unsigned char*>(p);
    p += (size_t)K;
    sm.keep = reinterpret_cast<unsigned char*>(p);
}

__device__ __forceinline__ const short* load_basis(char* smem, const short* g, int count) {
    short* s = reinterpret_cast<short*>(smem);
    for (int e = threadIdx.x; e < count; e += blockDim.x) s[e] = g[e];
    return s;
}

// Assemble the local system of stencil j (§4.1) and its q right-hand sides (the columns in
// sm.cols) in shared memory, with the whole CTA.  Full layout: both triangles of A_hat and
// B_hat beside it.  Packed layout: the lower triangle of A_hat and B_hat apart.
template <int D, bool PACKED, int NT>
__device__ void assemble_local(const SolveArgs& a, const Shape& sh, int j, int q,
                               const StencilSmem& sm) {
    const int tid = threadIdx.x;
    const int n = sh.n, M = sh.M, K = sh.K, m = sh.m;
    const Basis& bs = sh.bs;
    double* X = sm.X;
    const int xs = sm.xs;
    const double* xc = a.X + (size_t)j * D;
    // Scaled coordinates (x - x_c) / rho_j, correctly rounded: the weights of ill-conditioned
    // stencils are as sensitive to the node positions as to the solve, so these match the
    // oracle's exactly.  Only the threads that hold a node compute rho_j.
    if (tid < n) {
        double r2c = a.rho2[j];
        if (__double_as_longlong(r2c) <= 0) r2c = 1.0;
        const double rho = sqrt(r2c);
        for (int t = tid; t < n; t += NT) {
            const int id = a.nbr[(size_t)j * a.n + t];
            for (int c = 0; c < D; ++c)
                sm.xi[t * D + c] = __ddiv_rn(__dsub_rn(a.X[(size_t)id * D + c], xc[c]), rho);
        }
    }
    if (PACKED) {
        for (int e = tid; e < tri(K); e += NT) sm.T[e] = 0.0;
        for (int e = tid; e < K * q; e += NT) {
            const int r = e / q, c = e - r * q;
            X[r * xs + c] = 0.0;
        }
    } else {
        const int Wd = K + q, S = xs;
        for (int e = tid; e < K * Wd; e += NT) {
            const int r = e / Wd, c = e - r * Wd;
            sm.A[r * S + c] = 0.0;
        }
    }
    __syncthreads();
    // A_ab = r^m and, for solved ball members, the phi-part of the right-hand side
    // m (m + D - 2) r^(m-2) (Laplacian of r^m in D dimensions), pair by pair
    // (pairs a < b; row a of the strict upper triangle has n-1-a entries, and rows a and
    // n-2-a together have n, so the flattened index steps in O(1))
    if (n > 1) {
        const int rows = n - 1, L2 = n;
        const int total = ((rows + 1) >> 1) * L2;
        int pr = tid / L2, off = tid - (tid / L2) * L2;
        const int di = NT / L2, dj = NT - di * L2;
        for (int e = tid; e < total; e += NT) {
            const int len0 = rows - pr;
            const bool first = off < len0;
            const int ra = first ? pr : rows - 1 - pr;
            const int t = first ? off : off - len0;
            if (first || ra != pr) {
                const int rb = ra + 1 + t;
                const double r2 = a.fma_r2 ? sqdist_local<D>(sm.xi + ra * D, sm.xi + rb * D)
                                           : sqdist_rn<D>(sm.xi + ra * D, sm.xi + rb * D);
                const double r = sqrt_fast(r2);
                double pm2 = r;
                for (int s = 0; s < (m - 3) / 2; ++s) pm2 = __dmul_rn(pm2, r2);
                const double pm = __dmul_rn(pm2, r2);
                if (PACKED) {
                    sm.T[tri(rb) + ra] = pm;
                } else {
                    sm.A[ra * xs + rb] = pm;
                    sm.A[rb * xs + ra] = pm;
                }
                const int ca = sm.colof[ra], cb = sm.colof[rb];
                if (cb >= 0 && cb < q) X[ra * xs + cb] = __dmul_rn(sh.coef, pm2);
                if (ca >= 0 && ca < q) X[rb * xs + ca] = __dmul_rn(sh.coef, pm2);
            }
            pr += di;
            off += dj;
            if (off >= L2) { off -= L2; ++pr; }
        }
    }
    // P: one stencil point per thread, each monomial = an earlier one times one coordinate
    for (int r = tid; r < n; r += NT) {
        if (PACKED) {
            sm.T[tri(n) + r] = 1.0;
            for (int l = 1; l < M; ++l)
                sm.T[tri(n + l) + r] = sm.T[tri(n + bs.parent[l]) + r] * sm.xi[r * D + bs.var[l]];
        } else {
            double* row = sm.A + r * xs + n;
            row[0] = 1.0;
            sm.A[n * xs + r] = 1.0;
            for (int l = 1; l < M; ++l) {
                const double v = row[bs.parent[l]] * sm.xi[r * D + bs.var[l]];
                row[l] = v;
                sm.A[(n + l) * xs + r] = v;
            }
        }
    }
    __syncthreads();
    // psi-part of the right-hand sides: Laplacian of each monomial at each solved member,
    // from the monomial values already computed for that member
    for (int e = tid; e < M * q; e += NT) {
        const int l = e / q, c = e - l * q;
        const int t = sm.cols[c];
        double s = 0.0;
        for (int d = 0; d < D; ++d) {
            const int ch = bs.lap_child[l * D + d];
            if (ch >= 0) {
                const double pv = PACKED ? sm.T[tri(n + ch) + t] : sm.A[t * xs + n + ch];
                s = fma(exact_double(bs.lap_coef[l * D + d]), pv, s);
            }
        }
        X[(n + l) * xs + c] = s;
    }
    __syncthreads();
}

// LU with partial pivoting of [A_hat | B_hat] in the full layout (the paper's decomposition,
// §4.3 cost model (2/3) K^3 + 2 K^2 q), then back substitution.  Returns false (uniformly)
// on an exactly zero pivot; on success row r of the right-hand-side block holds unknown r.
template <int NT>
__device__ bool factor_solve_lu(int K, int q, const StencilSmem& sm) {
    __shared__ int s_ok;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int S = sm.xs;
    const int Wd = K + q;
    for (int r = tid; r < K; r += NT) { sm.rowof[r] = r; sm.perm[r] = r; }  // unknowns stay in place
    // the pivot search, row swap, reciprocal and multipliers are done by warp 0 alone (FP64
    // work counts per warp instruction, so the other warps must not repeat it)
    for (int p = 0; p < K; ++p) {
        if (wid == 0) {
            unsigned long long bv = 0ull;
            int bi = 0x7fffffff;
            for (int i = p + lane; i < K; i += 32) {
                const unsigned long long v = abs_bits(sm.A[i * S + p]);
                if (v > bv || (v == bv && i < bi)) { bv = v; bi = i; }
            }
            for (int o = 16; o > 0; o >>= 1) {
                const unsigned long long ov = __shfl_xor_sync(0xffffffffu, bv, o);
                const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
                if (ov > bv || (ov == bv && oi < bi)) { bv = ov; bi = oi; }
            }
            if (bv == 0ull) {
                if (lane == 0) s_ok = 0;
            } else {
                if (bi != p) {
                    for (int c = p + lane; c < Wd; c += 32) {
                        const double t = sm.A[p * S + c];
                        sm.A[p * S + c] = sm.A[bi * S + c];
                        sm.A[bi * S + c] = t;
                    }
                    __syncwarp();
                }
                const double rcp = rcp_fixed(sm.A[p * S + p]);
                if (lane == 0) { sm.rdiag[p] = rcp; s_ok = 1; }
                for (int i = p + 1 + lane; i < K; i += 32) sm.A[i * S + p] *= rcp;
            }
        }
        __syncthreads();
        if (!s_ok) return false;
        const int wr = K - p - 1, wc = Wd - p - 1;
        const int total = wr * wc;
        if (tid < total) {
            int ii = tid / wc, jj = tid - (tid / wc) * wc;
            const int di = NT / wc, dj = NT - di * wc;
            const double* Ap = sm.A + p * S + p + 1;
            double* Ab = sm.A + (p + 1) * S;
#pragma unroll 4
            for (int e = tid; e < total; e += NT) {
                double* row = Ab + ii * S;
                row[p + 1 + jj] = fma(-row[p], Ap[jj], row[p + 1 + jj]);
                ii += di;
                jj += dj;
                if (jj >= wc) { jj -= wc; ++ii; }
            }
        }
        __syncthreads();
    }
    // back substitution, q columns at once
    for (int p = K - 1; p >= 0; --p) {
        for (int c = tid; c < q; c += NT) sm.A[p * S + K + c] *= sm.rdiag[p];
        __syncthreads();
        const int total = p * q;
        if (tid < total) {
            int ii = tid / q, jj = tid - (tid / q) * q;
            const int di = NT / q, dj = NT - di * q;
            const double* xp = sm.A + p * S + K;
#pragma unroll 4
            for (int e = tid; e < total; e += NT) {
                double* row = sm.A + ii * S;
                row[K + jj] = fma(-row[p], xp[jj], row[K + jj]);
                ii += di;
                jj += dj;
                if (jj >= q) { jj -= q; ++ii; }
            }
        }
        __syncthreads();
    }
    return true;
}

// Forward substitution with the unit lower factor of one column Xc (row stride xs) by one
// warp, 32 rows at a time (2x2 pivots update a row with both columns in one expression, as in
// the factorization; a block never splits a 2x2 pivot): inside a block the lanes keep x in
// registers and take each pivot's value by a shuffle; below the block every lane applies the
// block's updates to its rows in pivot order.  Each entry receives the same FMAs in the same
// order as in forward_subst, with one warp synchronisation per block instead of per pivot.
__device__ __forceinline__ void forward_subst_warp(int K, const StencilSmem& sm, double* Xc, int xs) {
    const int lane = threadIdx.x & 31;
    for (int b0 = 0; b0 < K;) {
        int b1 = min(b0 + 32, K);
        if (b1 < K && sm.pk[b1 - 1] == 2) --b1;
        const int i = b0 + lane;
        double x = i < b1 ? Xc[i * xs] : 0.0;
        for (int p = b0; p < b1;) {
            const int k = sm.pk[p];
            const double xp = __shfl_sync(0xffffffffu, x, p - b0);
            const double xq = __shfl_sync(0xffffffffu, x, min(p + 1 - b0, 31));
            if (i > p + k - 1 && i < b1) {
                const double* Ti = sm.T + tri(i);
                x = k == 1 ? fma(-Ti[p], xp, x) : fma(-Ti[p + 1], xq, fma(-Ti[p], xp, x));
            }
            p += k;
        }
        if (i < b1) Xc[i * xs] = x;
        __syncwarp();
        for (int r = b1 + lane; r < K; r += 32) {
            const double* Tr = sm.T + tri(r);
            double xr = Xc[r * xs];
            for (int p = b0; p < b1;) {
                const int k = sm.pk[p];
                xr = k == 1 ? fma(-Tr[p], Xc[p * xs], xr)
                            : fma(-Tr[p + 1], Xc[(p + 1) * xs], fma(-Tr[p], Xc[p * xs], xr));
                p += k;
            }
            Xc[r * xs] = xr;
        }
        __syncwarp();
        b0 = b1;
    }
}

// Blocked triangular solves of the columns 0 .. q-1 of sm.X with the whole team, 32 unknowns
// at a time, for teams that hold one to four systems per SM (256 and 512 threads): a warp
// solves a column's diagonal block (lanes keep x in registers, each pivot's value by a
// shuffle), then every thread updates the column's remaining rows with that block in pivot
// order.  On GB300 a warp issues FP64 instructions to one quarter of the SM's FP64 units
// only, so a triangular solve by a single warp runs at a quarter of the SM's rate when few
// systems share the SM; here the rows' updates spread over all four.  (With ten or more
// systems per SM the step-by-step forms keep the pipe busier.)  Each entry receives the same
// FMAs in the same order as in the step-by-step forms (forward_subst; the back substitution
// of ldlt_solve_tail), so results are bit-identical.

// Forward substitution with the unit lower factor (a block never splits a 2x2 pivot).
template <int NT>
__device__ void forward_subst_blocked(int K, int q, const StencilSmem& sm) {
    constexpr int NW = NT / 32;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int xs = sm.xs;
    for (int b0 = 0; b0 < K;) {
        int b1 = min(b0 + 32, K);
        if (b1 < K && sm.pk[b1 - 1] == 2) --b1;
        for (int c = wid; c < q; c += NW) {
            double* Xc = sm.X + c;
            const int i = b0 + lane;
            double x = i < b1 ? Xc[i * xs] : 0.0;
            for (int p = b0; p < b1;) {
                const int k = sm.pk[p];
                const double xp = __shfl_sync(0xffffffffu, x, p - b0);
                const double xq = __shfl_sync(0xffffffffu, x, min(p + 1 - b0, 31));
                if (i > p + k - 1 && i < b1) {
                    const double* Ti = sm.T + tri(i);
                    x = k == 1 ? fma(-Ti[p], xp, x) : fma(-Ti[p + 1], xq, fma(-Ti[p], xp, x));
                }
                p += k;
            }
            if (i < b1) Xc[i * xs] = x;
        }
        __syncthreads();
        for (int e = tid; e < (K - b1) * q; e += NT) {
            const int r = b1 + e / q, c = e - (e / q) * q;
            const double* Tr = sm.T + tri(r);
            const double* Xc = sm.X + c;
            double xr = Xc[r * xs];
            for (int p = b0; p < b1;) {
                const int k = sm.pk[p];
                xr = k == 1 ? fma(-Tr[p], Xc[p * xs], xr)
                            : fma(-Tr[p + 1], Xc[(p + 1) * xs], fma(-Tr[p], Xc[p * xs], xr));
                p += k;
            }
            sm.X[r * xs + c] = xr;
        }
        __syncthreads();
        b0 = b1;
    }
}

// Back substitution with L^T (after the D solve): x_j -= L[i][j] x_i for j < i, i descending.
template <int NT>
__device__ void back_subst_blocked(int K, int q, const StencilSmem& sm) {
    constexpr int NW = NT / 32;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int xs = sm.xs;
    for (int b1 = K; b1 > 0;) {
        const int b0 = max(b1 - 32, 0);
        for (int c = wid; c < q; c += NW) {
            double* Xc = sm.X + c;
            const int j = b0 + lane;
            double x = j < b1 ? Xc[j * xs] : 0.0;
            for (int i = b1 - 1; i > b0; --i) {
                const double xi = __shfl_sync(0xffffffffu, x, i - b0);
                if (j < i) x = fma(-sm.T[tri(i) + j], xi, x);
            }
            if (j < b1) Xc[j * xs] = x;
        }
        __syncthreads();
        for (int e = tid; e < b0 * q; e += NT) {
            const int r = e / q, c = e - (e / q) * q;
            const double* Xc = sm.X + c;
            double xr = Xc[r * xs];
            for (int i = b1 - 1; i >= b0; --i) xr = fma(-sm.T[tri(i) + r], Xc[i * xs], xr);
            sm.X[r * xs + c] = xr;
        }
        __syncthreads();
        b1 = b0;
    }
}

// D solve and back substitution of the right-hand-side columns 0 .. q-1 held in sm.X, after
// the forward substitution (carried through the factorization, or forward_subst).
template <int NT>
__device__ __forceinline__ void ldlt_solve_tail(int K, int q, const StencilSmem& sm) {
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int xs = sm.xs;
    double* T = sm.T;
    double* X = sm.X;
    // D solve: 1x1 rows scale by the reciprocal pivot, 2x2 blocks multiply by their inverse;
    // then back substitution with L^T: once x_i is final, x_j -= L[i][j] x_i for j < i.
    // With at most one column per warp (q <= NW), warp w owns column w and its K sequential
    // steps need only warp synchronisation; otherwise all threads share every step (the
    // flattened (row, column) pairs keep the lanes busy) with a barrier per step.  Both do
    // the same operations on every element.
    constexpr int NW = NT / 32;
    if (q <= NW && NT < 256) {
        if (wid < q) {
            double* Xc = X + wid;
            for (int i = lane; i < K; i += 32) {
                const int k = sm.pk[i];
                double* Bi = Xc + i * xs;
                if (k == 1) {
                    *Bi *= sm.rdiag[i];
                } else if (k == 2) {  // rows i, i + 1 form a 2x2 block
                    double* Bn = Bi + xs;
                    const double y0 = *Bi, y1 = *Bn;
                    *Bi = fma(sm.rdiag[i], y0, sm.dinv1[i] * y1);
                    *Bn = fma(sm.dinv1[i], y0, sm.rdiag[i + 1] * y1);
                }
            }
            __syncwarp();
            for (int i = K - 1; i > 0; --i) {
                const double* Li = T + tri(i);
                const double xv = Xc[i * xs];
                for (int jj = lane; jj < i; jj += 32) Xc[jj * xs] = fma(-Li[jj], xv, Xc[jj * xs]);
                __syncwarp();
            }
        }
        return;
    }
    for (int e = tid; e < K * q; e += NT) {
        const int i = e / q, c = e - (e / q) * q;
        const int k = sm.pk[i];
        double* Bi = X + i * xs + c;
        if (k == 1) {
            *Bi *= sm.rdiag[i];
        } else if (k == 2) {
            double* Bn = Bi + xs;
            const double y0 = *Bi, y1 = *Bn;
            *Bi = fma(sm.rdiag[i], y0, sm.dinv1[i] * y1);
            *Bn = fma(sm.dinv1[i], y0, sm.rdiag[i + 1] * y1);
        }
    }
    __syncthreads();
    if constexpr (NT >= 256) {
        back_subst_blocked<NT>(K, q, sm);
        return;
    }
    for (int i = K - 1; i > 0; --i) {
        const int total = i * q;
        if (tid < total) {
            int jj = tid / q, cc = tid - (tid / q) * q;
            const int dj = NT / q, dc = NT - dj * q;
            const double* Li = T + tri(i);
            const double* xi = X + i * xs;
#pragma unroll 4
            for (int e = tid; e < total; e += NT) {
                double* xj = X + jj * xs;
                xj[cc] = fma(-Li[jj], xi[cc], xj[cc]);
                jj += dj;
                cc += dc;
                if (cc >= q) { cc -= q; ++jj; }
            }
        }
        __syncthreads();
    }
}

// Symmetric indefinite LDL^T factorization with Bunch-Kaufman partial pivoting (J. R. Bunch
// and L. Kaufman, "Some stable methods for calculating inertia and solving symmetric linear
// systems", Math. Comp. 31 (1977)) of the symmetric saddle-point matrix [A P; P^T 0] in the
// packed layout, with the right-hand sides carried along; (1/3) K^3 + 2 K^2 q flops.  1x1
// and 2x2 pivots with alpha = (1 + sqrt(17)) / 8; symmetric swaps are tracked in sm.perm.
// Returns false (uniformly) on an exactly singular pivot column.  On success sm.rowof[u] is
// the row of the right-hand-side block that holds unknown u.
// Pivot ratio of the factorization, written by factor_solve_ldlt<NT, true>: floor(log2) of
// max |D block entry| times floor(log2) of max |D^-1 block entry|, i.e. an estimate (within a
// factor 4) of log2 of max |d| / min |d| over the pivots, a lower bound of the system's
// condition number.  Read after a barrier.
__shared__ int s_pivot_log2_ratio;
constexpr int kRefinePivotLog2 = 16;  // refine systems whose pivots span at least 2^16

// Biased IEEE exponent of |v| (an integer-pipe floor(log2 |v|) + 1023).
__device__ __forceinline__ int exp_bits(double v) { return (int)((abs_bits(v) >> 52) & 0x7ff); }

// One pivot step at p of the factorization below, by warp 0: the Bunch-Kaufman choice (1x1,
// possibly after a symmetric swap, or 2x2), the reciprocal pivot or the 2x2 inverse, and the
// scaled column(s) of L in place; the unscaled pivot column is kept in wb (a 1x1 step) or in
// sm.wv and sm.wv2 (a 2x2 step) for the trailing update.  Lane 0 publishes s_ok and s_kind.
__shared__ int s_ok, s_kind;

template <bool TRACK>
__device__ __forceinline__ void pivot_step(int K, int q, int p, const StencilSmem& sm, double* wb,
                                           int& e_d, int& e_r) {
    const int lane = threadIdx.x & 31;
    const int xs = sm.xs;
    double* T = sm.T;
    double* X = sm.X;
    // The lane's first two entries of the pivot column and the reciprocal of the
    // diagonal, in one straight-line block so the reciprocal's integer chain overlaps
    // the loads and the search; the usual 1x1 step without a swap then scales these
    // registers directly.
    const double dpp = T[tri(p) + p];
    const int i0 = p + 1 + lane, i1 = i0 + 32;
    const double w0 = i0 < K ? T[tri(i0) + p] : 0.0;
    const double w1 = i1 < K ? T[tri(i1) + p] : 0.0;
    bool slow;
    const double rcp_p = rcp_core(dpp, &slow);
    // lambda = max |A[i][p]|, i > p, on magnitude keys (the top 32 bits of |A[i][p]|,
    // an order-preserving truncation), lowest index among equal keys; two warp
    // reductions instead of a shuffle tree
    unsigned lk = 0u;
    int r = 0x7fffffff;
    {
        const unsigned k0 = i0 < K ? mag_key(w0) : 0u;
        const unsigned k1 = i1 < K ? mag_key(w1) : 0u;
        if (k0 > lk) { lk = k0; r = i0; }
        if (k1 > lk) { lk = k1; r = i1; }
    }
    for (int i = i1 + 32; i < K; i += 32) {  // columns longer than 64
        const unsigned v = mag_key(T[tri(i) + p]);
        if (v > lk) { lk = v; r = i; }
    }
    const unsigned lmax = __reduce_max_sync(0xffffffffu, lk);
    r = (int)__reduce_min_sync(0xffffffffu,
                               (lk == lmax && lmax != 0u) ? (unsigned)r : 0x7fffffffu);
    const unsigned long long lv = (unsigned long long)lmax << 32;
    // the pivot choice only has to be a valid Bunch-Kaufman choice, so the tests run in
    // FP32 on values rebuilt from the FP64 bit patterns (no FP64 instructions)
    const unsigned long long pv = abs_bits(dpp);
    const float lam = approx_f32(lv), app = approx_f32(pv);
    const float af = 0.6403882f;
    int kind = 1, swap_a = p, swap_b = p;
    bool ok = true;
    if (lv == 0ull) {
        ok = pv != 0ull;  // column already eliminated: 1x1 pivot if nonzero
    } else if (!(app >= af * lam)) {
        // sigma = max |A_rj| over the active part of row/column r, j != r
        unsigned sk = 0u;
        for (int jj = p + lane; jj < K; jj += 32) {
            if (jj == r) continue;
            const unsigned b = mag_key(jj < r ? T[tri(r) + jj] : T[tri(jj) + r]);
            sk = b > sk ? b : sk;
        }
        sk = __reduce_max_sync(0xffffffffu, sk);
        const float sig = approx_f32((unsigned long long)sk << 32),
                    arr = approx_f32(abs_bits(T[tri(r) + r]));
        if (app * sig >= af * lam * lam) {
            kind = 1;
        } else if (arr >= af * sig) {
            kind = 1; swap_a = p; swap_b = r;
        } else {
            kind = 2; swap_a = p + 1; swap_b = r;
        }
    }
    if (ok && swap_a != swap_b) {
        // symmetric swap of unknowns ua < ub in the packed lower triangle, one uniform
        // loop per segment (row parts left of ua, the part between, the columns below
        // ub, the right-hand-side rows, the diagonal pair)
        const int ua = swap_a, ub = swap_b;
        auto exch = [](double* x, double* y) { const double t = *x; *x = *y; *y = t; };
        for (int e = lane; e < ua; e += 32) exch(T + tri(ua) + e, T + tri(ub) + e);
        for (int i = ua + 1 + lane; i < ub; i += 32) exch(T + tri(i) + ua, T + tri(ub) + i);
        for (int i = ub + 1 + lane; i < K; i += 32) exch(T + tri(i) + ua, T + tri(i) + ub);
        for (int c = lane; c < q; c += 32) exch(X + ua * xs + c, X + ub * xs + c);
        if (lane == 0) {
            exch(T + tri(ua) + ua, T + tri(ub) + ub);
            const int t = sm.perm[ua]; sm.perm[ua] = sm.perm[ub]; sm.perm[ub] = t;
        }
        __syncwarp();
    }
    if (ok) {
        if (kind == 1 && swap_a == swap_b && !slow) {  // the usual step: all in registers
            if (lane == 0) { sm.rdiag[p] = rcp_p; sm.pk[p] = 1; }
            if (TRACK && lane == 0) {
                e_d = max(e_d, exp_bits(dpp));
                e_r = max(e_r, exp_bits(rcp_p));
            }
            const double s0 = w0 * rcp_p, s1 = w1 * rcp_p;
            if (i0 < K) { wb[i0] = w0; T[tri(i0) + p] = s0; }
            if (i1 < K) { wb[i1] = w1; T[tri(i1) + p] = s1; }
            for (int i = i1 + 32; i < K; i += 32) {
                const double w = T[tri(i) + p];
                wb[i] = w;
                T[tri(i) + p] = w * rcp_p;
            }
        } else if (kind == 1) {  // after a swap (or an extreme pivot): reload
            const double rcp = rcp_fixed(T[tri(p) + p]);
            if (lane == 0) { sm.rdiag[p] = rcp; sm.pk[p] = 1; }
            if (TRACK && lane == 0) {
                e_d = max(e_d, exp_bits(T[tri(p) + p]));
                e_r = max(e_r, exp_bits(rcp));
            }
            for (int i = p + 1 + lane; i < K; i += 32) {
                const double w = T[tri(i) + p];
                wb[i] = w;
                T[tri(i) + p] = w * rcp;
            }
        } else {
            const double d0 = T[tri(p) + p], d1 = T[tri(p + 1) + p], d2 = T[tri(p + 1) + p + 1];
            const double rdet = rcp_fixed(fma(d0, d2, -d1 * d1));
            const double i00 = d2 * rdet, i01 = -d1 * rdet, i11 = d0 * rdet;
            if (lane == 0) {
                sm.rdiag[p] = i00; sm.dinv1[p] = i01; sm.rdiag[p + 1] = i11;
                sm.pk[p] = 2; sm.pk[p + 1] = 0;
                T[tri(p + 1) + p] = 0.0;  // L has no entry inside a 2x2 pivot block
                if (TRACK) {
                    e_d = max(e_d, max(exp_bits(d0), max(exp_bits(d1), exp_bits(d2))));
                    e_r = max(e_r, max(exp_bits(i00), max(exp_bits(i01), exp_bits(i11))));
                }
            }
            for (int i = p + 2 + lane; i < K; i += 32) {
                const double w1 = T[tri(i) + p], w2 = T[tri(i) + p + 1];
                sm.wv[i] = w1;
                sm.wv2[i] = w2;
                T[tri(i) + p] = fma(w1, i00, w2 * i01);
                T[tri(i) + p + 1] = fma(w1, i01, w2 * i11);
            }
        }
    }
    if (lane == 0) { s_ok = ok ? 1 : 0; s_kind = kind; }
}

// Trailing update after the pivot step at p (kind 1 or 2) by the threads U0 .. NT-1; wb holds a
// 1x1 step's unscaled pivot column (sm.wv for a 2x2 step, with sm.wv2).
template <int NT, int U0>
__device__ __forceinline__ void trailing_update(int K, int q, int p, int kind, const StencilSmem& sm,
                                                const double* wb, bool skip_next) {
    constexpr int UT = NT - U0;
    const int ut = (int)threadIdx.x - U0;
    const int xs = sm.xs;
    double* T = sm.T;
    double* X = sm.X;
    // Trailing update of the lower triangle and of the right-hand sides: row i (> p0)
    // has (i - p0) triangle entries followed by q right-hand-side entries.  Rows r and
    // rows-1-r are paired into one virtual row of constant length rows + 1 + 2q, so the
    // flattened index steps in O(1).  The FP64 work is branch-free: source operands are
    // selected with integer arithmetic so every lane issues the same FMA (a divergent
    // FP64 instruction costs the whole warp on the FP64 pipe).
    const int p0 = p + kind - 1;
    const int rows = K - p0 - 1;
    if (rows > 0) {
        const int L2 = rows + 1 + 2 * q;
        const int total = ((rows + 1) >> 1) * L2;
        if (ut < total) {
            int pr = ut / L2, off = ut - (ut / L2) * L2;
            const int di = UT / L2, dj = UT - di * L2;
            for (int e = ut; e < total; e += UT) {
                const int len0 = pr + 1 + q;
                const bool first = off < len0;
                const int r = first ? pr : rows - 1 - pr;
                const int t = first ? off : off - len0;
                // an odd middle row pairs with itself: once only; with skip_next column p0 + 1 is
                // left to warp 0
                if ((first || r != pr) && (t != 0 || !skip_next)) {
                    const int i = p0 + 1 + r;
                    double* Ti = T + tri(i);
                    const bool trin = t <= r;
                    const int jj = p0 + 1 + t;      // triangle column
                    const int c = t - (r + 1);      // right-hand-side column
                    double* dst = trin ? Ti + jj : X + i * xs + c;
                    const double* s1 = trin ? wb + jj : X + p * xs + c;
                    if (kind == 1) {
                        *dst = fma(-Ti[p], *s1, *dst);
                    } else {
                        const double* s2 = trin ? sm.wv2 + jj : X + (p + 1) * xs + c;
                        *dst = fma(-Ti[p + 1], *s2, fma(-Ti[p], *s1, *dst));
                    }
                }
                pr += di;
                off += dj;
                if (off >= L2) { off -= L2; ++pr; }
            }
        }
    }
}

// Look-ahead of the next pivot for 512-thread teams (one system per SM, where nothing hides
// the serial pivot step): while the other warps apply the 1x1 step at p, warp 0 applies it
// to column pn = p + 1 (the FMA every entry of the trailing update gets) and tries the usual
// next step there, a 1x1 pivot without a swap, which the column alone decides.  If it holds
// (and the pivot is not extreme), the step is stored exactly as pivot_step would store it,
// its unscaled column in wn (the other buffer: the update running now reads wc); otherwise
// the updated column stays unscaled for pivot_step.  Results are bit-identical either way.
template <bool TRACK>
__device__ __forceinline__ bool lookahead_pivot(int K, int p, const StencilSmem& sm, const double* wc,
                                                double* wn, int& e_d, int& e_r) {
    const int lane = threadIdx.x & 31;
    double* T = sm.T;
    const int pn = p + 1;
    const double f = wc[pn];
    const double dpp = fma(-T[tri(pn) + p], f, T[tri(pn) + pn]);
    const int i0 = pn + 1 + lane, i1 = i0 + 32;
    const double w0 = i0 < K ? fma(-T[tri(i0) + p], f, T[tri(i0) + pn]) : 0.0;
    const double w1 = i1 < K ? fma(-T[tri(i1) + p], f, T[tri(i1) + pn]) : 0.0;
    bool slow;
    const double rcp_p = rcp_core(dpp, &slow);
    unsigned lk = 0u;
    {
        const unsigned k0 = i0 < K ? mag_key(w0) : 0u;
        const unsigned k1 = i1 < K ? mag_key(w1) : 0u;
        lk = k0 > k1 ? k0 : k1;
    }
    for (int i = i1 + 32; i < K; i += 32) {
        const double w = fma(-T[tri(i) + p], f, T[tri(i) + pn]);
        T[tri(i) + pn] = w;
        const unsigned v = mag_key(w);
        lk = v > lk ? v : lk;
    }
    const unsigned long long lv = (unsigned long long)__reduce_max_sync(0xffffffffu, lk) << 32;
    const unsigned long long pv = abs_bits(dpp);
    const float lam = approx_f32(lv), app = approx_f32(pv);
    const float af = 0.6403882f;
    const bool take = lv != 0ull && app >= af * lam && !slow;
    if (lane == 0) T[tri(pn) + pn] = dpp;
    if (take) {
        if (lane == 0) { sm.rdiag[pn] = rcp_p; sm.pk[pn] = 1; }
        if (TRACK && lane == 0) {
            e_d = max(e_d, exp_bits(dpp));
            e_r = max(e_r, exp_bits(rcp_p));
        }
        if (i0 < K) { wn[i0] = w0; T[tri(i0) + pn] = w0 * rcp_p; }
        if (i1 < K) { wn[i1] = w1; T[tri(i1) + pn] = w1 * rcp_p; }
        for (int i = i1 + 32; i < K; i += 32) {
            const double w = T[tri(i) + pn];
            wn[i] = w;
            T[tri(i) + pn] = w * rcp_p;
        }
    } else {
        if (i0 < K) T[tri(i0) + pn] = w0;
        if (i1 < K) T[tri(i1) + pn] = w1;
    }
    return take;
}

template <int NT, bool TRACK = false>
__device__ bool factor_solve_ldlt(int K, int q, const StencilSmem& sm) {
    const int tid = threadIdx.x, wid = tid >> 5;
    int e_d = 0, e_r = 0;  // (thread 0, TRACK) largest exponents of |D| and |D^-1| entries
    for (int r = tid; r < K; r += NT) sm.perm[r] = r;
    __syncthreads();
    int p = 0;
    if constexpr (NT == 512) {
        // Warp 0 looks one pivot ahead (lookahead_pivot) while warps 1-15 update; the 1x1
        // steps alternate their unscaled column between sm.wv and sm.wv + K (= sm.wv2, which
        // only 2x2 steps use otherwise), and the look-ahead's outcome alternates between two
        // flags, so no flag or column is rewritten while another warp may still read it.
        __shared__ int s_took[2];
        int cur = 0, it = 0;
        bool have_pivot = false;
        while (p < K) {
            if (!have_pivot) {
                if (wid == 0) pivot_step<TRACK>(K, q, p, sm, sm.wv + cur * K, e_d, e_r);
                __syncthreads();
                if (!s_ok) return false;
            }
            const int kind = have_pivot ? 1 : s_kind;
            const double* wb = kind == 2 ? sm.wv : sm.wv + cur * K;
            const bool look = kind == 1 && p + 1 < K;
            if (wid == 0) {
                if (look) {
                    const bool took = lookahead_pivot<TRACK>(K, p, sm, wb, sm.wv + (cur ^ 1) * K, e_d, e_r);
                    if ((tid & 31) == 0) s_took[it & 1] = took ? 1 : 0;
                }
            } else {
                trailing_update<NT, 32>(K, q, p, kind, sm, wb, look);
            }
            __syncthreads();
            have_pivot = look && s_took[it & 1] != 0;
            if (have_pivot) cur ^= 1;
            ++it;
            p += kind;
        }
    } else {
        while (p < K) {
            if (wid == 0) pivot_step<TRACK>(K, q, p, sm, sm.wv, e_d, e_r);
            __syncthreads();
            if (!s_ok) return false;
            const int kind = s_kind;
            trailing_update<NT, 0>(K, q, p, kind, sm, sm.wv, false);
            __syncthreads();
            p += kind;
        }
    }
    // The inverse permutation (read after the caller's next barrier).
    for (int r = tid; r < K; r += NT) sm.rowof[sm.perm[r]] = r;
    if (TRACK && tid == 0) s_pivot_log2_ratio = e_d + e_r - 2 * 1023;
    ldlt_solve_tail<NT>(K, q, sm);
    return true;
}

// ------------------------------------------------------------------ right-hand sides in chunks
// The factorization carries at most a.qcap right-hand sides (shared memory is sized for that
// many); a center with more solves the rest afterwards, a.qcap at a time, with the stored
// factors.  Every column gets the same operations, in the same order, as it would have had
// in the first chunk, so the weights do not depend on the chunk a column falls in.

// psi_l(x) by the parent recurrence, multiplied in the order the monomial block is built.
template <int D>
__device__ __forceinline__ double mono_value(const Basis& bs, int l, const double* x) {
    unsigned code = 0;  // the variables from l up to the constant, 2 bits each
    int depth = 0;
    while (l > 0) {
        code = (code << 2) | (unsigned)bs.var[l];
        ++depth;
        l = bs.parent[l];
    }
    double v = 1.0;
    for (int i = 0; i < depth; ++i) {
        v = v * x[code & 3u];
        code >>= 2;
    }
    return v;
}

// Right-hand-side entry of unknown u for the column of stencil position t: m (m + D - 2)
// r^(m-2) (as in the pair loop) for a stencil node, the Laplacian of psi_(u-n) at node t for a
// monomial.
template <int D>
__device__ __forceinline__ double rhs_entry(const Shape& sh, int u, int t, const double* xi,
                                            bool fma_r2) {
    const int n = sh.n;
    double v = 0.0;
    if (u < n) {
        if (u != t) {
            const double r2 = fma_r2 ? sqdist_local<D>(xi + u * D, xi + t * D)
                                     : sqdist_rn<D>(xi + u * D, xi + t * D);
            double pm2 = sqrt_fast(r2);
            for (int k = 0; k < (sh.m - 3) / 2; ++k) pm2 = __dmul_rn(pm2, r2);
            v = __dmul_rn(sh.coef, pm2);
        }
    } else {
        const int l = u - n;
        for (int d = 0; d < D; ++d) {
            const int ch = sh.bs.lap_child[l * D + d];
            if (ch >= 0)
                v = fma(exact_double(sh.bs.lap_coef[l * D + d]), mono_value<D>(sh.bs, ch, xi + t * D), v);
        }
    }
    return v;
}

// Right-hand sides of columns c0 .. c0+qk-1 into sm.X, rows in the factorization's permuted
// order (row r holds unknown perm[r]).
template <int D, int NT>
__device__ void chunk_rhs(const Shape& sh, int c0, int qk, const StencilSmem& sm, bool fma_r2) {
    const int K = sh.K;
    for (int e = threadIdx.x; e < K * qk; e += NT) {
        const int r = e / qk, c = e - (e / qk) * qk;
        sm.X[r * sm.xs + c] = rhs_entry<D>(sh, sm.perm[r], sm.cols[c0 + c], sm.xi, fma_r2);
    }
}

// Forward substitution with the unit lower factor, step by step as the factorization applied
// it to the carried columns (a 2x2 pivot's two columns update a row in one expression).
template <int NT>
__device__ void forward_subst(int K, int q, const StencilSmem& sm) {
    const int xs = sm.xs;
    for (int p = 0; p < K;) {
        const int k = sm.pk[p];
        const int p0 = p + k - 1;
        const int total = (K - p0 - 1) * q;
        for (int e = threadIdx.x; e < total; e += NT) {
            const int r = e / q, c = e - (e / q) * q;
            const int i = p0 + 1 + r;
            const double* Ti = sm.T + tri(i);
            double* dst = sm.X + i * xs + c;
            if (k == 1) *dst = fma(-Ti[p], sm.X[p * xs + c], *dst);
            else *dst = fma(-Ti[p + 1], sm.X[(p + 1) * xs + c], fma(-Ti[p], sm.X[p * xs + c], *dst));
        }
        __syncthreads();
        p += k;
    }
}

template <int NT>
__device__ __forceinline__ void lebesgue_values(int n, int K, int q, const StencilSmem& sm,
                                                int off = 0);

// Right-hand side of the normal derivative at the stencil center (the origin of the scaled
// coordinates) for unknown u of node i's own stencil (§5, a Neumann row): d/dn ||y - xi_u||^m
// at y = 0 is -m ||xi_u||^(m-2) (xi_u . n), and of the monomials only the linear ones have a
// nonzero gradient there (d/dn xi_a = n_a).
template <int D>
__device__ __forceinline__ double neumann_at(const Shape& sh, const double* nv, int u, const double* xj) {
    if (u < sh.n) {
        const double mm = exact_double(sh.m);
        double r2 = xj[0] * xj[0], dot = xj[0] * nv[0];
        for (int c = 1; c < D; ++c) {
            r2 = fma(xj[c], xj[c], r2);
            dot = fma(xj[c], nv[c], dot);
        }
        double pm2 = sqrt_fast(r2);  // r^(m-2), m odd
        for (int t = 0; t < (sh.m - 3) / 2; ++t) pm2 *= r2;
        return -mm * pm2 * dot;
    }
    const int l = u - sh.n;
    return (l > 0 && sh.bs.parent[l] == 0) ? nv[sh.bs.var[l]] : 0.0;
}
template <int D>
__device__ __forceinline__ double neumann_value(const Shape& sh, const double* nv, int u, const double* xi) {
    return neumann_at<D>(sh, nv, u, xi + (u < sh.n ? u * D : 0));
}

// Normals of any length: the null-space solves hold right-hand sides in units fixed by the exponent,
// so they take the normal times 2^-e, its largest component in (1/2, 1] (unit vectors, in 2D and 3D:
// e = 0), and the row is scaled back at the end.  Returns e (0 for a zero normal).
template <int D>
__device__ __forceinline__ int scaled_normal(const SolveArgs& a, int i, double* nv) {
    double top = 0.0;
    for (int c = 0; c < D; ++c) {
        nv[c] = a.nrm[(size_t)i * D + c];
        top = fmax(top, fabs(nv[c]));
    }
    int e = 0;
    const double m = frexp(top, &e);  // in [1/2, 1)
    if (m == 0.5) --e;
    if (top == 0.0) e = 0;
    for (int c = 0; c < D; ++c) nv[c] = scalbn(nv[c], -e);
    return e;
}

// Normal-derivative right-hand side of node i's own stencil, replacing column 0 of the
// right-hand-side block (unknowns in index order, before the factorization).
template <int D, int NT>
__device__ void neumann_rhs(const Shape& sh, const double* nv, const StencilSmem& sm) {
    for (int j = threadIdx.x; j < sh.n + sh.M; j += NT) sm.X[j * sm.xs] = neumann_value<D>(sh, nv, j, sm.xi);
}

// Team sizes whose traversal kernels carry the refinement step: the 96- and 128-thread teams
// run with 40 registers for small systems (many per SM), and the planner gives plans that
// refine (largest system K >= 100, at most a few per SM) 256- or 512-thread teams, or 32 or
// 64 when forced.  The fallback kernel carries it at every team size (ALL_TEAMS).
__host__ __device__ constexpr bool team_refines(int nt) { return nt != 96 && nt != 128; }

// Per-CTA scratch of the refinement step of this launch, or nullptr when the plan refines
// nothing.  (Whether a system is refined is decided after its factorization.)
template <int NT, bool ALL_TEAMS = false>
__device__ __forceinline__ double* refine_scratch(const SolveArgs& a) {
    if constexpr (!ALL_TEAMS && !team_refines(NT)) {
        return nullptr;
    } else {
        return a.rs != nullptr ? a.rs + (size_t)blockIdx.x * a.rs_stride : nullptr;
    }
}

// The residual's dot products sum_v A_uv x0_v are split into kRefineSegs fixed ranges of v
// (the same for every team size), summed in order within a range and then combined in a
// fixed order, so every thread of a team has short independent chains and the bits do not
// depend on the team.
constexpr int kRefineSegs = 4;

// Partial sum over v in segment g of A_uv x0_v: gA is the full assembled matrix (row v at
// v K, so the threads of a warp, holding consecutive u, read one contiguous row), gX0 holds
// x0 by unknown (unknown v of column c at v qk + c: one address for the whole warp).
__device__ __forceinline__ double residual_part(int u, int c, int g, int K, int qk,
                                                const double* __restrict__ gA,
                                                const double* __restrict__ gX0) {
    const int len = (K + kRefineSegs - 1) / kRefineSegs;
    const int v0 = g * len, v1 = min(K, v0 + len);
    double s = 0.0;
#pragma unroll 8
    for (int v = v0; v < v1; ++v) s = fma(__ldcg(gA + (size_t)v * K + u), __ldcg(gX0 + v * qk + c), s);
    return s;
}

// One step of iterative refinement (J. H. Wilkinson, "Rounding Errors in Algebraic Processes",
// 1963) of the columns c0 .. c0+qk-1 held in sm.X after their LDL^T solve:
// x1 = x0 + (L D L^T)^-1 (b - A x0), the residual formed in FP64 with the assembled matrix A
// (gA, copied in full before the factorization overwrote it) and the right-hand sides rebuilt
// bit for bit.  On the ill-conditioned systems of large stencils (condition
// numbers up to ~1e10) the first solution's forward error is dominated by the symmetric-
// pivoting factorization; one step brings it down to that of the assembled system itself.
// Only systems whose pivot ratio (s_pivot_log2_ratio) reaches 2^kRefinePivotLog2 are refined,
// unless a.refine_all: the well-conditioned majority keeps its first solution.  kind: 0 the
// Laplacian right-hand sides of the columns in sm.cols, 2 the normal derivative at the center
// of node i (one column).  gX0 holds x0 (K x qk).  With at most one column per warp each warp
// forward-substitutes its own column; the arithmetic of an entry is the same either way, so
// every team size gives the same bits.
template <int D, int NT>
__device__ void refine_columns(const SolveArgs& a, const Shape& sh, int c0, int qk,
                               const StencilSmem& sm, const double* __restrict__ gA,
                               double* __restrict__ gX0, int kind, int i) {
    constexpr int NW = NT / 32;
    const int K = sh.K, xs = sm.xs, tid = threadIdx.x, wid = tid >> 5;
    double* gP = gX0 + (size_t)K * qk;  // kRefineSegs partial sums per entry
    __syncthreads();  // (the last solve steps may have been warp-synchronous)
    // adaptive: only systems whose pivots span at least 2^16 (unless every system is refined)
    if (a.refine_all == 0 && s_pivot_log2_ratio < kRefinePivotLog2) return;
    for (int e = tid; e < K * qk; e += NT) {  // x0 by unknown
        const int r = e / qk, c = e - r * qk;
        gX0[sm.perm[r] * qk + c] = sm.X[r * xs + c];
    }
    if (kind == 2) {
        for (int r = tid; r < K; r += NT) sm.X[r * xs] = neumann_value<D>(sh, a.nrm + (size_t)i * D, sm.perm[r], sm.xi);
    } else {
        chunk_rhs<D, NT>(sh, c0, qk, sm, a.fma_r2 != 0);
    }
    __syncthreads();
    for (int e = tid; e < K * qk * kRefineSegs; e += NT) {  // (unknown, column, segment) items
        const int g = e / (K * qk), uc = e - g * (K * qk);
        const int u = uc / qk, c = uc - u * qk;
        gP[e] = residual_part(u, c, g, K, qk, gA, gX0);
    }
    __syncthreads();
    for (int e = tid; e < K * qk; e += NT) {  // r = b - ((p0 + p1) + (p2 + p3)), rows permuted
        const int r = e / qk, c = e - r * qk;
        const int uc = sm.perm[r] * qk + c;
        const double* P = gP + uc;
        const size_t st = (size_t)K * qk;
        sm.X[r * xs + c] = sm.X[r * xs + c] - ((__ldcg(P) + __ldcg(P + st)) + (__ldcg(P + 2 * st) + __ldcg(P + 3 * st)));
    }
    __syncthreads();
    if (NT >= 256) {  // forward substitution
        forward_subst_blocked<NT>(K, qk, sm);
    } else if (qk <= NW) {  // a warp per column with warp synchronisation only
        if (wid < qk) forward_subst_warp(K, sm, sm.X + wid, xs);
    } else {
        forward_subst<NT>(K, qk, sm);
    }
    ldlt_solve_tail<NT>(K, qk, sm);
    __syncthreads();
    for (int e = tid; e < K * qk; e += NT) {
        const int r = e / qk, c = e - r * qk;
        sm.X[r * xs + c] += __ldcg(gX0 + sm.perm[r] * qk + c);
    }
    if (tid == 0) atomicAdd(&a.ctr->sum_k2r, (unsigned long long)K * K * qk);
    __syncthreads();
}

// The refinement step for the columns that can be kept (refine_columns on a subset).  With a
// Lebesgue test (SEQ, FALLBACK) a column whose first solution's Lebesgue value exceeds the
// test's reference value by more than 2^-10 of it fails the test whatever the refinement does
// (a step changes the values by far less on the systems it is for: about the condition number
// times the rounding, below 1e-5), and its weights are discarded; only the center, the
// reference column and the other columns are refined.  They are moved to the front of the
// right-hand-side block (and sm.cols with them), refined there and moved back; each column's
// arithmetic does not depend on the others, so a kept column gets the same bits as when every
// column is refined.  cref is the reference column (0, or 1 with the centroid option); the
// chunk's unrefined Lebesgue values are left in sm.lam for the caller to recompute.  The
// scratch slot holds the moved block after the refinement's own arrays (6 K q_cap + q_cap).
template <int D, int NT>
__device__ void refine_kept_columns(const SolveArgs& a, const Shape& sh, int c0, int qk,
                                    const StencilSmem& sm, double* __restrict__ gA, int cref,
                                    int j) {
    __syncthreads();
    if (a.refine_all == 0 && s_pivot_log2_ratio < kRefinePivotLog2) return;
    double* gX0 = gA + a.rs_x0;
    if (a.mode == RBFFD_STAB_OFF || qk == 1) {
        refine_columns<D, NT>(a, sh, c0, qk, sm, gA, gX0, 0, j);
        return;
    }
    const int K = sh.K, xs = sm.xs, tid = threadIdx.x;
    lebesgue_values<NT>(sh.n, K, qk, sm, c0);
    __syncthreads();
    // the selection, in column order, by warp 0: kept columns first (map[c'] = column of
    // position c'); sm.keep[c0 ..] serves as the map (the test writes it afterwards)
    __shared__ int s_qr;
    unsigned char* map = sm.keep + c0;
    if (tid < 32) {
        const double lref = sm.lam[cref];
        const double lim = lref * (1.0 + 0x1p-10);
        int nsel = 0;
        for (int b = 0; b < qk; b += 32) {  // selected columns, in order
            const int c = b + tid;
            const bool sel = c < qk && (c0 + c == 0 || c0 + c == cref || sm.lam[c0 + c] <= lim);
            const unsigned bal = __ballot_sync(0xffffffffu, sel);
            if (sel) map[nsel + __popc(bal & ((1u << tid) - 1u))] = (unsigned char)c;
            nsel += __popc(bal);
        }
        int nrest = nsel;
        for (int b = 0; b < qk; b += 32) {  // then the others, in order
            const int c = b + tid;
            const bool sel = c < qk && (c0 + c == 0 || c0 + c == cref || sm.lam[c0 + c] <= lim);
            const bool other = c < qk && !sel;
            const unsigned bal = __ballot_sync(0xffffffffu, other);
            if (other) map[nrest + __popc(bal & ((1u << tid) - 1u))] = (unsigned char)c;
            nrest += __popc(bal);
        }
        if (tid == 0) s_qr = nsel;
    }
    __syncthreads();
    const int qr = s_qr;
    if (qr == qk) {
        refine_columns<D, NT>(a, sh, c0, qk, sm, gA, gX0, 0, j);
        return;
    }
    double* gT = gX0 + (size_t)5 * K * qk;   // the block in the new column order
    int* gC = reinterpret_cast<int*>(gT + (size_t)K * qk);  // sm.cols of the chunk, saved
    for (int e = tid; e < K * qk; e += NT) {
        const int c = e / K, r = e - c * K;
        gT[e] = sm.X[r * xs + map[c]];
    }
    for (int c = tid; c < qk; c += NT) gC[c] = sm.cols[c0 + c];
    __syncthreads();
    for (int e = tid; e < K * qr; e += NT) {
        const int c = e / K, r = e - c * K;
        sm.X[r * xs + c] = __ldcg(gT + e);
    }
    for (int c = tid; c < qk; c += NT) sm.cols[c0 + c] = __ldcg(gC + map[c]);
    __syncthreads();
    refine_columns<D, NT>(a, sh, c0, qr, sm, gA, gX0, 0, j);  // (ends with a barrier)
    for (int e = tid; e < K * qr; e += NT) {  // the refined columns over their first solutions
        const int c = e / K, r = e - c * K;
        gT[e] = sm.X[r * xs + c];
    }
    __syncthreads();
    for (int e = tid; e < K * qk; e += NT) {  // back to the original order
        const int c = e / K, r = e - c * K;
        sm.X[r * xs + map[c]] = __ldcg(gT + e);
    }
    for (int c = tid; c < qk; c += NT) sm.cols[c0 + c] = __ldcg(gC + c);
    __syncthreads();
}

// The assembled symmetric matrix (packed lower triangle in shared memory) to gA in full,
// row-major K x K, before the factorization overwrites it.
template <int NT>
__device__ __forceinline__ void copy_full_matrix(int K, const StencilSmem& sm, double* __restrict__ gA) {
    for (int e = threadIdx.x; e < K * K; e += NT) {
        const int r = e / K, c = e - r * K;
        gA[e] = r >= c ? sm.T[tri(r) + c] : sm.T[tri(c) + r];
    }
}

// Columns c0 .. c0+qk-1 with the stored LDL^T factors: right-hand sides, forward substitution,
// D solve, back substitution (refined like the first chunk) and Lebesgue values (a chunk after
// the first of a center).
template <int D, int NT>
__device__ __forceinline__ void solve_chunk(const SolveArgs& a, const Shape& sh, int c0, int qk,
                                            const StencilSmem& sm, int j, int cref) {
    chunk_rhs<D, NT>(sh, c0, qk, sm, a.fma_r2 != 0);
    __syncthreads();
    if constexpr (NT >= 256) forward_subst_blocked<NT>(sh.K, qk, sm);
    else forward_subst<NT>(sh.K, qk, sm);
    ldlt_solve_tail<NT>(sh.K, qk, sm);
    if constexpr (team_refines(NT)) {
        if (double* gA = refine_scratch<NT>(a))
            refine_kept_columns<D, NT>(a, sh, c0, qk, sm, gA, cref, j);
    }
    __syncthreads();
    lebesgue_values<NT>(sh.n, sh.K, qk, sm, c0);
}

// Assemble, factor and solve the first q columns of stencil j (refined when its shape asks).
template <int D, bool PACKED, int NT>
__device__ bool solve_local(const SolveArgs& a, const Shape& sh, int j, int q,
                            const StencilSmem& sm, int cref) {
    assemble_local<D, PACKED, NT>(a, sh, j, q, sm);
    if constexpr (!PACKED) {
        return factor_solve_lu<NT>(sh.K, q, sm);
    } else {
        double* gA = refine_scratch<NT>(a);
        if (gA) copy_full_matrix<NT>(sh.K, sm, gA);
        if (!factor_solve_ldlt<NT, team_refines(NT)>(sh.K, q, sm)) return false;
        if constexpr (team_refines(NT)) {
            if (gA) refine_kept_columns<D, NT>(a, sh, 0, q, sm, gA, cref, j);
        }
        return true;
    }
}

// Local L-Lebesgue value sum_r |w_r| of every solved column: warp w sums the columns w, w + NW,
// ... (the columns it back-substituted), over the unknowns u whose original index perm[u] is
// a stencil node (not a polynomial coefficient).
template <int NT>
__device__ __forceinline__ void lebesgue_values(int n, int K, int q, const StencilSmem& sm,
                                                int off) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int c = wid; c < q; c += (NT / 32)) {
        double s = 0.0;
        for (int u = lane; u < K; u += 32) {
            const double v = sm.X[u * sm.xs + c];
            s += sm.perm[u] < n ? fabs(v) : 0.0;
        }
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) sm.lam[off + c] = s;
    }
}

// ------------------------------------------------------------------ null-space solves
// Stencil coordinates (x - x_c) / rho_j, rounded to FP64 as everywhere (the quotient by a reciprocal
// and one residual).
struct Radius { double rho, rcp; };
__device__ __forceinline__ Radius ns_radius(const SolveArgs& a, int j) {
    double r2c = a.rho2[j];
    if (__double_as_longlong(r2c) <= 0) r2c = 1.0;
    const double rho = sqrt_fast(r2c);
    return {rho, rcp_fixed(rho)};
}
template <int D>
__device__ __forceinline__ double ns_coordinate(const SolveArgs& a, int j, int t, int c, const Radius& r) {
    const int id = a.nbr[(size_t)j * a.n + t];
    const double dx = __dsub_rn(a.X[(size_t)id * D + c], a.X[(size_t)j * D + c]);
    const double x = dx * r.rcp;
    return fma(fma(-x, r.rho, dx), r.rcp, x);
}

// All of them in units of 2^-kCoordBits (which holds every bit of a coordinate of 2^-8 and more), and
// the identity order.
constexpr int kCoordBits = 61;
template <int D, int NT>
__device__ void ns_coordinates(const SolveArgs& a, const Shape& sh, int j, const NullSmem& sm) {
    const Radius r = ns_radius(a, j);
#pragma unroll 1
    for (int e = threadIdx.x; e < sh.n * D; e += NT) {
        const int t = e / D, c = e - t * D;
        sm.xi[e] = to_fixed(ns_coordinate<D>(a, j, t, c, r), -kCoordBits);
        if (c == 0) sm.order[t] = t;
    }
}

// Unit of the g rows in the elimination: 2^gs times the nodes' rows', so that ghat may reach
// 8 2^gs: 64 at degree 2, 512, 1024 and 2048 at 3, 4 and 5, two to three times the largest
// entries met in quasi-uniform, boundary and clustered stencils (24, 184, 439, 1023).  For a normal
// derivative (kind 2, |g| <= 1) 8 to 128 is as wide; in the units of the Laplacians' its weights were
// four times further from a double-double solve.
__device__ __forceinline__ int ns_g_shift(int ell, int kind) {
    if (kind == 2) return ell < 2 ? 0 : ell - 1;
    return ell < 2 ? 1 : (ell == 2 ? 3 : ell + 3);
}

// The tableau of the constraints in fixed point (rows: nodes, then the q columns' right-hand sides
// g).  kind 2: the normal derivative at the center of node j's own stencil (one column), else
// Laplacians at the nodes in sm.cols.
template <int D, int NT>
__device__ void ns_constraints_fixed(const SolveArgs& a, const Shape& sh, int j, int q, int gs,
                                     const NullSmem& sm, int kind) {
    const int tid = threadIdx.x;
    const int n = sh.n, M = sh.M, ldm = sm.ldm;
    const Basis& bs = sh.bs;
    long long* T = fixed(sm.T);
#pragma unroll 1
    for (int t = tid; t < n; t += NT) {  // each monomial = an earlier one times one coordinate
        int2 x[D];
#pragma unroll
        for (int c = 0; c < D; ++c) x[c] = split_limbs(shift_right(sm.xi[t * D + c], kCoordBits - kTabBits));
        long long* row = T + t * ldm;
        row[0] = 1ll << kTabBits;
#pragma unroll 1
        for (int l = 1; l < M; ++l) {
            const int v = bs.var[l];
            int2 xv = x[0];
            if (v == 1) xv = x[1];
            if (D == 3 && v == 2) xv = x[D - 1];
            row[l] = mul_limbs(split_limbs(row[bs.parent[l]]), xv);
        }
    }
    __syncthreads();
#pragma unroll 1
    for (int e = tid; e < M * q; e += NT) {
        const int c = small_div(e, M), l = e - c * M;
        long long v = 0;
        if (kind == 2) {
            double nv[D];
            const double x0[D] = {};
            scaled_normal<D>(a, j, nv);
            v = to_fixed(neumann_at<D>(sh, nv, n + l, x0), gs - kTabBits);
        } else {
            const long long* row = T + sm.cols[c] * ldm;
            for (int d = 0; d < D; ++d) {
                const int ch = bs.lap_child[l * D + d];
                if (ch >= 0) v += row[ch] * bs.lap_coef[l * D + d];
            }
            v = shift_fixed(v, -gs);
        }
        T[(n + c) * ldm + l] = v;
    }
    __syncthreads();
}

// The same in FP64, for the stencils whose elimination leaves the fixed-point ranges.
template <int D, int NT>
__device__ void ns_constraints(const SolveArgs& a, const Shape& sh, int j, int q, const NullSmem& sm,
                               int kind) {
    const int tid = threadIdx.x;
    const int n = sh.n, M = sh.M, ldm = sm.ldm;
    const Basis& bs = sh.bs;
    const Radius r = ns_radius(a, j);
#pragma unroll 1
    for (int t = tid; t < n; t += NT) {
        double x[D];
        for (int c = 0; c < D; ++c) x[c] = ns_coordinate<D>(a, j, t, c, r);
        double* row = sm.T + t * ldm;
        row[0] = 1.0;
#pragma unroll 1
        for (int l = 1; l < M; ++l) {
            const int v = bs.var[l];
            row[l] = row[bs.parent[l]] * (v == 0 ? x[0] : (v == 1 ? x[1] : x[D - 1]));
        }
        sm.order[t] = t;
    }
    __syncthreads();
#pragma unroll 1
    for (int e = tid; e < M * q; e += NT) {
        const int c = e / M, l = e - c * M;
        double v = 0.0;
        if (kind == 2) {
            double nv[D];
            const double x0[D] = {};
            scaled_normal<D>(a, j, nv);
            v = neumann_at<D>(sh, nv, n + l, x0);
        } else {
            const double* row = sm.T + sm.cols[c] * ldm;
            for (int d = 0; d < D; ++d) {
                const int ch = bs.lap_child[l * D + d];
                if (ch >= 0) v = fma(exact_double(bs.lap_coef[l * D + d]), row[ch], v);
            }
        }
        sm.T[(n + c) * ldm + l] = v;
    }
    __syncthreads();
}

template <int D, int NT>
__device__ __noinline__ bool ns_eliminate_fp64(const SolveArgs& a, const Shape& sh, int j, int q,
                                               int eg_min, const NullSmem& sm, int kind) {
    if (threadIdx.x == 0) s_ns_eb = 0;  // (rows that left the fixed-point range may have raised it)
    ns_constraints<D, NT>(a, sh, j, q, sm, kind);
    if (!ns_eliminate<NT>(sh.n, sh.M, q, sm)) return false;
    ns_scales<NT>(sh.n, sh.M, q, eg_min, sm);
    __syncthreads();
    ns_rows_to_limbs<NT>(sh.n, sh.M, q, sm);
    __syncthreads();
    return true;
}

// The kernel.  A polynomial p of degree m - 1 in r changes A by P Y^T + Y P^T and so neither S nor the
// weights (2 ell + 1 >= m), as long as the same p is taken off f.  The solves use
//   phi(r) = r^m - p(r^2) = 2^m z^((m-1)/2) (u - beta),   u = r / 2, z = u^2 (r <= 2: the radius is 1)
// with the beta that makes |phi| small: 9, 16 and 23 times below 2^m for m = 3, 5, 7.  S is formed of
// entries of that size, and the grids of A, C and its sums are as much finer.  With r^m itself their
// rounding was as large as the squared distances' in 2D.  Median errors over 120 rows against an
// 80-bit solve (r^7, this / r^m itself / the saddle-point layout): disk, degree 3, n = 21, 2.3e-13 /
// 3.1e-13 / 2.3e-13; degree 4, n = 31, 1.6e-12 / 2.4e-12 / 1.8e-12; lattice, degree 4, 3.9e-13 /
// 1.5e-12 / 4.0e-13; ball, degree 4, n = 71, 2.2e-12 / 2.4e-12 / 2.5e-12; degree 5, n = 113, 1.2e-11 /
// 1.5e-11 / 1.3e-11.  It costs about 30 instructions a pair and saves the products of lower limbs that
// the sums needed before (552 plans: the same time, geometric mean of the ratios 1.00).
struct KernelUnits {
    int beta;    // of 256
    int eA, eF;  // |phi| < 2^eA, |f| < 2^eF
    int fs;      // eF = m - 2 + fs
    int c1, c3;  // f = 2^(m-2) (c1 u z^k - beta c3 z^k), k = (m - 3) / 2: the Laplacian's factors, or
                 // (kind 2) those of the derivative against -(x . n)
};

template <int D>
__device__ __forceinline__ KernelUnits ns_units(int m, int kind) {
    KernelUnits k;
    k.beta = m == 3 ? 229 : (m == 5 ? 242 : 245);
    k.eA = m == 3 ? 0 : m - 4;
    k.fs = kind == 2 ? 1 : (m == 3 ? 3 : 4);
    k.eF = m - 2 + k.fs;
    k.c1 = kind == 2 ? m : m * (m + D - 2);
    k.c3 = kind == 2 ? m - 1 : (m - 1) * (m + D - 3);
    return k;
}

// What phi and f of a pair are made of: phi in 2^-62 of 2^m, pk = z^k (u - beta) in 2^-62, z in 2^-63,
// and delta, below.
struct PairPowers {
    long long phi, pk, z;
    int delta;
};

// a z 2^-64 for z >= 0 (__mul64hi would look at the sign of z too).
__device__ __forceinline__ long long mul_by(long long a, long long z) {
    return (long long)__umul64hi((unsigned long long)a, (unsigned long long)z) - ((a >> 63) & z);
}

// The squared distance in u is formed in FP64 without FMA, rounded as the oracle's: the weights are as
// far from an exact solve as that rounding puts every FP64 solver's, and so near to theirs.  In p it
// has to be exact, or p would be no polynomial: z and the exact square differ by delta in 2^-63, a
// dozen bits, found from the low words of the coordinates' integer differences.  The root and the
// powers are fixed point.
template <int D>
__device__ __noinline__ PairPowers ns_powers(const long long* xa, const long long* xb, int m, int beta) {
    double r2 = 0.0;
    unsigned H = 0u;
    long long mid = 0;
    unsigned long long low = 0;
#pragma unroll
    for (int c = 0; c < D; ++c) {
        const long long d = xa[c] - xb[c];  // (the sum of d^2 is 2^(2 kCoordBits) r^2 = 2^124 z)
        const double t = __ll2double_rn(d);
        r2 = c == 0 ? __dmul_rn(t, t) : __dadd_rn(r2, __dmul_rn(t, t));
        const int hi = (int)((d + (1ll << 31)) >> 32), lo = (int)d;
        H += (unsigned)(hi * hi);
        mid += (long long)hi * lo;
        low += (unsigned long long)((long long)lo * lo);
    }
    const unsigned exact = (H << 3) + (unsigned)(mid >> 28) + (unsigned)(low >> 61);  // 2^63 z, low word
    const unsigned long long b = (unsigned long long)__double_as_longlong(r2);
    const int e = (int)(b >> 52) - 1023 - 2 * kCoordBits, odd = e & 1;  // r^2 = w 4^h, w in [1, 4)
    const unsigned long long N = ((b & 0xFFFFFFFFFFFFFull) | (1ull << 52)) << (10 + odd);  // w 2^62
    const unsigned long long zr = N >> min(2 + odd - e, 63) << 1;
    PairPowers o;
    o.delta = (int)((unsigned)zr - exact);
    o.z = (long long)min(zr, 0x7fffffffffffffffull);
    const unsigned long long u =
        ((unsigned long long)sqrt_core(N) << 2) >> min(1 - ((e - odd) >> 1), 63);
    long long p = (long long)u - ((long long)beta << (kPowerBits - 8));
    const int k = (m - 3) / 2;
    if (k > 0) p = mul_by(p << 1, o.z);
    if (k > 1) p = mul_by(p << 1, o.z);
    o.pk = p;
    // beta (z^(k+1) - its exact value) = beta (k + 1) z^k delta, z^k with 12 bits
    const int zt = (int)(o.z >> 51), zk = k == 0 ? 4096 : (k == 1 ? zt : zt * zt >> 12);
    o.phi = mul_by(p << 1, o.z) + ((long long)o.delta * (beta * (k + 1) * zk) >> 21);
    return o;
}

// v c 2^-s, 0 <= c < 2^20, s <= 32.
__device__ __forceinline__ long long scale_by(long long v, int c, int s) {
    return (((v >> 32) * c) << (32 - s)) + (((v & 0xffffffffll) * c) >> s);
}

// f of a pair, in 2^(eF - kPowerBits): c1 u z^k - beta c3 z^k = c1 pk + beta (c1 - c3) z^k, and as above
// for the exact z^k of p.
__device__ __forceinline__ long long ns_rhs_fixed(const PairPowers& o, int m, const KernelUnits& ku) {
    const long long zk = m == 3 ? 1ll << kPowerBits : (m == 5 ? o.z >> 1 : (long long)__umul64hi(o.z, o.z));
    const int zt = (int)(o.z >> 51), dz = m == 3 ? 0 : (m == 5 ? 4096 : 2 * zt);  // k z^(k-1)
    const long long fix = (long long)o.delta * (ku.beta * ku.c3) * dz >> 21;
    return scale_by(o.pk, ku.c1, ku.fs) + scale_by(zk, (ku.c1 - ku.c3) * ku.beta, ku.fs + 8) + (fix >> ku.fs);
}

// From f's unit to that of f1 in a column of scale 2^eg.
__device__ __forceinline__ int ns_f1_shift(const KernelUnits& ku, int eg) {
    return ku.eF - kPowerBits - (ku.eA + eg + kSumUnit - 1);
}

// A11 (limbs, over the eliminated rows of the tableau), A21 (in C) and what the columns' f share
// with them: the pairs of tableau rows with at least one basic node, (i, j) with j < M and i > j,
// flattened by columns; f's entries at the other nodes of a column whose node is not basic either
// start from zero (ns_finish adds them with A22).  A21 and f1 count 2^(eA + scale of the row - 61) (the
// unit of ns_product_c), f2 2^(eF - 62).  In integers but for the squared distance: about 230 issue
// slots per warp and pair, where the FP64 form has 14 FP64 instructions of 64 cycles each.
template <int D, int NT>
__device__ void ns_pairs(const Shape& sh, int q, const KernelUnits& ku, const NullSmem& sm) {
    const int tid = threadIdx.x;
    const int n = sh.n, M = sh.M, m = sh.m, ldm = sm.ldm, s = n - M, eB = s_ns_eb;
    const int rect = s * M, total = rect + (M >> 1) * M;
#pragma unroll 1
    for (int e = tid; e < total; e += NT) {
        int i, j;  // tableau rows i > j, j < M
        if (e < rect) {
            i = M + small_div(e, M);
            j = e - (i - M) * M;
        } else {  // rows p + 1 and M - 1 - p of the triangle have M pairs (a middle row is its own)
            const int p = small_div(e - rect, M), o = e - rect - p * M;
            const bool low = o <= p;
            if (!low && M - 1 - p == p + 1) continue;
            i = low ? p + 1 : M - 1 - p;
            j = low ? o : o - p - 1;
        }
        const int ra = sm.order[i], rb = sm.order[j];
        const PairPowers o = ns_powers<D>(sm.xi + ra * D, sm.xi + rb * D, m, ku.beta);
        if (i < M) {
            const int2 v = split_limbs(shift_fixed(o.phi, m - ku.eA - (kPowerBits - kFixBits)));
            *limbs(sm.T + i * ldm + j) = v;
            *limbs(sm.T + j * ldm + i) = v;
        } else {
            fixed(sm.C)[(i - M) * ldm + j] = shift_fixed(o.phi, m - kPowerBits - (ku.eA + eB + kSumUnit - 1));
        }
        const int ca = sm.colof[ra], cb = sm.colof[rb];
        if ((ca >= 0 && ca < q) || (cb >= 0 && cb < q)) {
            const long long f = ns_rhs_fixed(o, m, ku);
#pragma unroll 1
            for (int k = 0; k < 2; ++k) {  // f of column c at row r
                const int c = k ? cb : ca, r = k ? i : j;
                if (c < 0 || c >= q) continue;
                fixed(sm.X)[c * sm.ldx + (r < M ? r : sm.x2 + r - M)] = r < M ? shift_fixed(f, ns_f1_shift(ku, sm.eg[c])) : f;
            }
        }
    }
#pragma unroll 1
    for (int t = tid; t < n; t += NT) {  // r = 0: phi = 0, and f = 0 but at r^3
        const int p = sm.pos[t], c = sm.colof[t];
        if (p < M) sm.T[p * ldm + p] = 0.0;
        if (c >= 0 && c < q) {
            long long* X = fixed(sm.X) + c * sm.ldx;
            const long long f = ns_rhs_fixed(ns_powers<D>(sm.xi + t * D, sm.xi + t * D, m, ku.beta), m, ku);
            if (p < M) {
                X[p] = shift_fixed(f, ns_f1_shift(ku, sm.eg[c]));
            } else {
#pragma unroll 1
                for (int i = 0; i < s; ++i) X[sm.x2 + i] = i == p - M ? f : 0;
            }
        }
    }
}

// A22 joins S and f's remaining entries the columns of the first chunk, pair by pair (a <= b of the
// nodes that are not basic; columns a and s - 1 - a of the triangle together have s + 1 entries), and
// S becomes doubles.
template <int D, int NT>
__device__ void ns_finish(const Shape& sh, int qk, const KernelUnits& ku, int kind, const NullSmem& sm) {
    const int n = sh.n, M = sh.M, s = n - M, m = sh.m, eB = s_ns_eb, eC = s_ns_ec;
    const int unit = eB + eC + kSumUnit, half = (s + 1) >> 1;
#pragma unroll 1
    for (int e = threadIdx.x; e < half * (s + 1); e += NT) {
        const int p = small_div(e, s + 1), o = e - p * (s + 1);
        const bool first = o < s - p;
        const int j = first ? p : s - 1 - p, i = first ? p + o : o - 1;
        if (!first && j == p) continue;  // an odd middle column pairs with itself
        double* d = sm.S + col_start(j, s) + i;
        long long a22 = 0;
        if (i != j) {
            const int ra = sm.order[M + i], rb = sm.order[M + j];
            const PairPowers o = ns_powers<D>(sm.xi + ra * D, sm.xi + rb * D, m, ku.beta);
            a22 = shift_fixed(o.phi, m - kPowerBits - unit);
            const int ca = sm.colof[ra], cb = sm.colof[rb];
            if (kind != 2 && ((ca >= 0 && ca < qk) || (cb >= 0 && cb < qk))) {
                const long long f = ns_rhs_fixed(o, m, ku);
                const int u = ku.eF - kPowerBits - kSumUnit - eC;  // of f, against 2^eg units
                if (ca >= 0 && ca < qk) fixed(sm.X)[ca * sm.ldx + sm.x2 + j] += shift_fixed(f, u - sm.eg[ca]);
                if (cb >= 0 && cb < qk) fixed(sm.X)[cb * sm.ldx + sm.x2 + i] += shift_fixed(f, u - sm.eg[cb]);
            }
        }
        *d = from_fixed(a22 + *fixed(d), unit);
    }
}

// The columns' right-hand sides to doubles.
template <int NT>
__device__ __forceinline__ void ns_rhs_to_fp64(int s, int c0, int qk, const NullSmem& sm) {
    const int eC = s_ns_ec;
#pragma unroll 1
    for (int e = threadIdx.x; e < s * qk; e += NT) {
        const int c = small_div(e, s);
        double* d = sm.X + c * sm.ldx + sm.x2 + e - c * s;
        *d = from_fixed(*fixed(d), sm.eg[c0 + c] + eC + kSumUnit);
    }
}

// One step of iterative refinement (Wilkinson) of the chunk's columns: the residual
// rho = f - A w in FP64 with the entries of A and f formed as the saddle-point systems form them
// (correctly rounded coordinates, no FMA in the squared distances), then S dv = rho_other -
// B rho_basic with the stored factors and w_basic -= B^T dv.  (The constraints hold by construction
// and are left alone.)  In plans that refine (K >= 100) systems whose pivots span at least 2^10 are
// refined (7% of the ball's, three quarters of the clustered cube's), or every system with
// a.refine_all.  Below that the unrefined weights are as good (ball, degree 5, n = 113, means over 190
// rows against an 80-bit solve, all refined from 2^10 on / none / the saddle-point layout: 1.84e-11 /
// 1.82e-11 / 1.97e-11); clustered sets need it (cube, degree 5, n = 90: 2.1e-10 / 8.7e-10 / 1.8e-10).
// gw: scratch of 2 n words per column and n D words.
constexpr int kNullRefineLog2 = 10;

template <int D, int NT>
__device__ __noinline__ void ns_refine(const SolveArgs& a, const Shape& sh, int j, int c0, int qk,
                                       const NullSmem& sm, int kind, double* gw) {
    const int tid = threadIdx.x, lane = tid & 31, n = sh.n, M = sh.M, s = n - M, m = sh.m;
    const int eB = s_ns_eb;
    double *gW = gw, *gR = gw + (size_t)n * qk, *gX = gw + (size_t)2 * n * qk;
    double r2c = a.rho2[j];
    if (__double_as_longlong(r2c) <= 0) r2c = 1.0;
    const double rho = sqrt(r2c);
#pragma unroll 1
    for (int e = tid; e < n * D; e += NT) {  // coordinates in tableau order
        const int p = e / D, c = e - p * D;
        const int id = a.nbr[(size_t)j * a.n + sm.order[p]];
        gX[e] = __ddiv_rn(__dsub_rn(a.X[(size_t)id * D + c], a.X[(size_t)j * D + c]), rho);
    }
#pragma unroll 1
    for (int e = tid; e < n * qk; e += NT) {
        const int c = small_div(e, n), p = e - c * n;
        gW[e] = p < M ? sm.T[(n + c0 + c) * sm.ldm + p] : sm.X[c * sm.ldx + sm.x2 + p - M];
    }
    __syncthreads();
    // rho: four columns share the entries of A, four lanes a row (a quarter of its terms each, summed
    // in one order whatever the team; with a lane per row 113 of a team's 256 threads walked 113
    // dependent terms: 3D degree 5, N = 4,000, delta = 1 6.93 ms of traversal, now 6.67)
    const int groups = (qk + 3) >> 2, part = (n + 3) >> 2, l4 = lane & 3;
#pragma unroll 1
    for (int e = tid; e < ((4 * n * groups + 31) & ~31); e += NT) {  // (whole warps)
        const int item = min(e >> 2, n * groups - 1);
        const int g = small_div(item, n), p = item - g * n, nc = min(4, qk - 4 * g);
        double x[D], r[4] = {};
        for (int d = 0; d < D; ++d) x[d] = gX[p * D + d];
        const double* w = gW + (size_t)4 * g * n;
        const int v1 = min((l4 + 1) * part, n);
#pragma unroll 2
        for (int v = l4 * part; v < v1; ++v) {
            double y[D];
            for (int d = 0; d < D; ++d) y[d] = gX[v * D + d];
            const double r2 = v == p ? 1.0 : sqdist_rn<D>(x, y);
            double pm = sqrt_fast(r2);
#pragma unroll 1
            for (int k = 0; k < (m - 1) / 2; ++k) pm = __dmul_rn(pm, r2);
            if (v == p) pm = 0.0;
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (c < nc) r[c] = fma(-pm, w[c * n + v], r[c]);
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            r[c] += __shfl_xor_sync(0xffffffffu, r[c], 1);
            r[c] += __shfl_xor_sync(0xffffffffu, r[c], 2);
        }
        if (l4 >= nc || e >= 4 * n * groups) continue;
        const int c = 4 * g + l4;  // lane l4 adds f of the group's column l4
        double f = l4 == 0 ? r[0] : (l4 == 1 ? r[1] : (l4 == 2 ? r[2] : r[3]));
        if (kind == 2) {
            double nv[D];
            scaled_normal<D>(a, j, nv);
            f += neumann_at<D>(sh, nv, 0, x);
        } else if (sm.order[p] != sm.cols[c0 + c]) {
            double y[D];
            const int t = sm.pos[sm.cols[c0 + c]];
            for (int d = 0; d < D; ++d) y[d] = gX[t * D + d];
            const double r2 = sqdist_rn<D>(x, y);
            double pm2 = sqrt_fast(r2);
#pragma unroll 1
            for (int k = 0; k < (m - 3) / 2; ++k) pm2 = __dmul_rn(pm2, r2);
            f += __dmul_rn(sh.coef, pm2);
        }
        gR[c * n + p] = f;
    }
    __syncthreads();
#pragma unroll 1
    for (int c = tid >> 5; c < qk; c += NT / 32) {  // rho_basic to limbs, in the words of f1
        int e = -200;
#pragma unroll 1
        for (int p = lane; p < M; p += 32) e = max(e, scale_exp(gR[c * n + p]));
        e = __reduce_max_sync(0xffffffffu, e);
#pragma unroll 1
        for (int p = lane; p < M; p += 32) limbs(sm.X + c * sm.ldx)[p] = to_limbs(gR[c * n + p], e);
        if (lane == 0) sm.ev[c] = (short)e;
    }
    __syncthreads();
#pragma unroll 1
    for (int e = tid; e < s * qk; e += NT) {
        const int c = small_div(e, s), i = e - c * s;
        LimbSum t;
#pragma unroll 1
        for (int k = 0; k < M; ++k) {
            t.mac(limbs(sm.T + (M + i) * sm.ldm)[k], limbs(sm.X + c * sm.ldx)[k]);
            if ((k & 15) == 15) t.fold();
        }
        sm.X[c * sm.ldx + sm.x2 + i] =
            gR[c * n + M + i] - from_fixed(t.total(), eB + sm.ev[c] + kSumUnit);
    }
    __syncthreads();
    ns_forward<NT>(s, qk, sm);
    ns_back<NT>(s, qk, sm);
    __syncthreads();
    ns_basic_correction<NT>(n, M, c0, qk, sm);
#pragma unroll 1
    for (int e = tid; e < s * qk; e += NT) {
        const int c = small_div(e, s), i = e - c * s;
        sm.X[c * sm.ldx + sm.x2 + i] += gW[c * n + M + i];
    }
    if (tid == 0) atomicAdd(&a.ctr->sum_k2r, (unsigned long long)sh.K * sh.K * qk);
    __syncthreads();
}

// Acquire-release fence at device scope: orders this thread's earlier memory operations, and
// those of its CTA that a barrier made visible to it, before its later ones, as seen by every
// thread of the device.  Only threads that publish (or consume) traversal state execute it.
__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

// The columns c0 .. c0+qk-1 of a stencil that the null space cannot solve, from its saddle-point
// system like the plans of the other layouts (unrefined): constraints that depend on each other, as
// on lattices, or a pivot of S at the level of its rounding (nodes within about 1e-8 of their
// distance to the others).  The system lies in one of the plan's blocks in global memory, taken for
// the time of the solve (whoever holds one waits for nobody); the columns go through it kSaddleCols
// at a time, and their weights to the places that ns_weight reads.  False on an exactly zero pivot.
__shared__ int s_ns_saddle;  // this stencil's columns come from here

template <int D, int NT>
__device__ __noinline__ bool saddle_columns(const SolveArgs& a, const Shape& sh, int j, int c0, int qk,
                                            const NullSmem& sm, int kind) {
    __shared__ int s_block;
    const int tid = threadIdx.x, n = sh.n, M = sh.M, K = sh.K;
    if (tid == 0) {
        const unsigned long long t0 = globaltimer_ns();
        int b = (int)(blockIdx.x % (unsigned)a.sd_slots);
        while (atomicCAS(&a.sd_lock[b], 0, 1) != 0) {
            b = b + 1 == a.sd_slots ? 0 : b + 1;
            if (globaltimer_ns() - t0 > a.timeout_ns) {
                set_error(a.ctr, RBFFD_ETIMEOUT);
                b = -1;
                break;
            }
            __nanosleep(64);
        }
        fence_gpu();  // (its last holder is done with it)
        s_block = b;
        s_ns_saddle = 1;
    }
    __syncthreads();
    const int block = s_block;
    if (block < 0) return false;
    StencilSmem st;
    carve<D, true>(a.sd + (size_t)block * a.sd_stride, a.n, a.K, kSaddleCols, kSaddleCols | 1, st);
    bool ok = true;
#pragma unroll 1
    for (int b = 0; b < qk && ok; b += kSaddleCols) {
        const int q = min(kSaddleCols, qk - b), first = c0 + b;
#pragma unroll 1
        for (int t = tid; t < n; t += NT) {
            const int c = sm.colof[t] - first;
            st.colof[t] = c >= 0 && c < q ? c : -1;
        }
        if (tid < q) st.cols[tid] = sm.cols[first + tid];
        __syncthreads();
        if (b == 0) {
            assemble_local<D, true, NT>(a, sh, j, q, st);
            if (kind == 2) {
                double nv[D];
                scaled_normal<D>(a, j, nv);
                neumann_rhs<D, NT>(sh, nv, st);
                __syncthreads();
            }
            ok = factor_solve_ldlt<NT>(K, q, st);
        } else {
            chunk_rhs<D, NT>(sh, 0, q, st, a.fma_r2 != 0);
            __syncthreads();
            forward_subst<NT>(K, q, st);
            ldlt_solve_tail<NT>(K, q, st);
        }
        __syncthreads();
#pragma unroll 1
        for (int e = tid; ok && e < q * n; e += NT) {
            const int c = small_div(e, n), r = e - c * n;
            const double w = st.X[st.rowof[r] * st.xs + c];
            if (r < M) sm.T[(n + first + c) * sm.ldm + r] = w;
            else sm.X[(b + c) * sm.ldx + sm.x2 + r - M] = w;
        }
        __syncthreads();
    }
#pragma unroll 1
    for (int t = tid; t < n; t += NT) sm.pos[t] = t;
    if (tid == 0) {
        fence_gpu();
        atomicExch(&a.sd_lock[block], 0);
    }
    __syncthreads();
    return ok;
}

// The columns c0 .. c0+qk-1 from their f rows on (the triangle's products and factorization with
// the first chunk).  f counts 2^(eF - kPowerBits).
template <int D, int NT, bool ALL_TEAMS>
__device__ bool ns_columns(const SolveArgs& a, const Shape& sh, int j, int c0, int qk, const KernelUnits& ku,
                           const NullSmem& sm, int kind) {
    const int n = sh.n, M = sh.M, s = n - M, eA = ku.eA, eF = ku.eF;
    const bool first = c0 == 0;
    ns_product_c<NT>(n, M, first ? 0 : s, c0, qk, eA, sm);
    __syncthreads();
    if (first) {
        ns_c_to_limbs<NT>(s, M, eA, sm);
    }
    ns_columns_to_limbs<NT>(n, M, c0, qk, eA, eF, sm);
    __syncthreads();
    ns_product_s<NT>(n, M, first, c0, qk, sm);
    __syncthreads();
    if (first) {
        ns_finish<D, NT>(sh, qk, ku, kind, sm);
        __syncthreads();
    }
    ns_rhs_to_fp64<NT>(s, c0, qk, sm);
    __syncthreads();
    if (first) {
        if (!ns_factor<NT>(s, qk, sm)) return false;
    } else {
        ns_forward<NT>(s, qk, sm);
    }
    ns_back<NT>(s, qk, sm);
    __syncthreads();
    ns_basic_weights<NT>(n, M, c0, qk, sm);
    __syncthreads();
    if (double* gw = refine_scratch<NT, ALL_TEAMS>(a)) {
        if (a.refine_all != 0 || s_ns_ratio >= kNullRefineLog2)
            ns_refine<D, NT>(a, sh, j, c0, qk, sm, kind, gw);
    }
    return true;
}

// The first q1 of the q columns of stencil j (see ns_constraints_fixed for kind).
template <int D, int NT, bool ALL_TEAMS = false>
__device__ bool ns_solve(const SolveArgs& a, const Shape& sh, int j, int q, int q1,
                         const NullSmem& sm, int kind) {
    const int tid = threadIdx.x, n = sh.n, M = sh.M;
    const KernelUnits ku = ns_units<D>(sh.m, kind);
    const int gs = ns_g_shift(sh.ell, kind);
    const int eg_min = ku.eF - ku.eA - 1;  // f1 fits the unit of its products (ns_product_c)
    if (tid == 0) {
        s_ns_eb = 0;
        s_ns_ec = ku.eA - 2;  // A22 (scale 2^eA) fits the unit of the sums
        s_ns_saddle = 0;
    }
    ns_coordinates<D, NT>(a, sh, j, sm);
    __syncthreads();
    ns_constraints_fixed<D, NT>(a, sh, j, q, gs, sm, kind);
    if (!ns_eliminate_fixed<NT>(n, M, q, gs, eg_min, sm) &&
        !ns_eliminate_fp64<D, NT>(a, sh, j, q, eg_min, sm, kind))
        return saddle_columns<D, NT>(a, sh, j, 0, q1, sm, kind);
#pragma unroll 1
    for (int t = tid; t < n; t += NT) sm.pos[sm.order[t]] = t;
    __syncthreads();
    ns_pairs<D, NT>(sh, q1, ku, sm);
    __syncthreads();
    if (kind == 2) {
        double nv[D];
        scaled_normal<D>(a, j, nv);
#pragma unroll 1
        for (int u = tid; u < n; u += NT) {  // (the center is the origin: node 0)
            const int p = sm.pos[u];
            double dot = 0.0;
            for (int c = 0; c < D; ++c)
                dot = fma(__ll2double_rn(sm.xi[u * D + c]) * (1.0 / (1ll << kCoordBits)), nv[c], dot);
            const long long f = ns_rhs_fixed(ns_powers<D>(sm.xi + u * D, sm.xi, sh.m, ku.beta), sh.m, ku);
            fixed(sm.X)[p < M ? p : sm.x2 + p - M] =
                to_fixed(-dot * from_fixed(f, ku.eF - kPowerBits),
                         p < M ? ku.eA + sm.eg[0] + kSumUnit - 1 : ku.eF - kPowerBits);
        }
        __syncthreads();
    }
    return ns_columns<D, NT, ALL_TEAMS>(a, sh, j, 0, q1, ku, sm, kind) ||
           saddle_columns<D, NT>(a, sh, j, 0, q1, sm, kind);
}

// Lebesgue values of the columns of a chunk: eight lanes per column, each over every eighth node of
// the stencil in order.
template <int NT>
__device__ __forceinline__ void ns_lebesgue(const Shape& sh, int c0, int qk, const NullSmem& sm) {
    const int part = threadIdx.x & 7;
#pragma unroll 1
    for (int cb = 0; cb < qk; cb += NT / 8) {  // (whole warps reach the shuffles)
        const int c = min(cb + (int)(threadIdx.x >> 3), qk - 1);
        double s = 0.0;
#pragma unroll 1
        for (int r = part; r < sh.n; r += 8) s += fabs(ns_weight(sh.n, sh.M, r, c0, c, sm));
        for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (part == 0) sm.lam[c0 + c] = s;
    }
}

// A later chunk of columns with the stored factors.
template <int D, int NT>
__device__ __forceinline__ bool ns_solve_chunk(const SolveArgs& a, const Shape& sh, int j, int c0,
                                               int qk, const NullSmem& sm) {
    if (s_ns_saddle) {
        const bool ok = saddle_columns<D, NT>(a, sh, j, c0, qk, sm, 0);
        if (ok) ns_lebesgue<NT>(sh, c0, qk, sm);
        return ok;
    }
    const int n = sh.n, M = sh.M;
    const KernelUnits ku = ns_units<D>(sh.m, 0);
#pragma unroll 1
    for (int e = threadIdx.x; e < n * qk; e += NT) {
        const int c = small_div(e, n), u = e - c * n, p = sm.pos[u], t = sm.cols[c0 + c];
        const long long f = ns_rhs_fixed(ns_powers<D>(sm.xi + u * D, sm.xi + t * D, sh.m, ku.beta), sh.m, ku);
        fixed(sm.X)[c * sm.ldx + (p < M ? p : sm.x2 + p - M)] =
            p < M ? shift_fixed(f, ns_f1_shift(ku, sm.eg[c0 + c])) : f;
    }
    __syncthreads();
    ns_columns<D, NT, false>(a, sh, j, c0, qk, ku, sm, 0);
    ns_lebesgue<NT>(sh, c0, qk, sm);
    return true;
}

// Weight of stencil position r in column c0 + c, column c of the chunk held in shared memory.
__device__ __forceinline__ double weight(const Shape&, int r, int, int c, const StencilSmem& sm) {
    return sm.X[sm.rowof[r] * sm.xs + c];
}
__device__ __forceinline__ double weight(const Shape& sh, int r, int c0, int c, const NullSmem& sm) {
    return ns_weight(sh.n, sh.M, r, c0, c, sm);
}

template <int LAY> struct SmemType { using T = StencilSmem; };
template <> struct SmemType<kNull> { using T = NullSmem; };
template <int LAY> using SmemOf = typename SmemType<LAY>::T;

// ------------------------------------------------------------------ traversal state machine
__device__ __forceinline__ void push_center(const SolveArgs& a, int k) {
    fence_gpu();
    const int slot = atomicAdd(&a.ctr->q_tail, 1);
    atomicExch(&a.queue[slot], k);
}

__device__ __forceinline__ void release(const SolveArgs& a, int k) {
    const int old = atomicSub(&a.pending[k], 1);
    if (old == 1) {
        fence_gpu();
        if (atomicCAS(&a.state[k], kUndecided, kCenter) == kUndecided) {
            atomicMin(&a.owner[k], k);
            push_center(a, k);
        }
    }
}

// node i has just become covered: its own ball releases its later members
__device__ inline void on_covered(const SolveArgs& a, int i) {
    atomicAdd(&a.ctr->done, 1);
    const int L = a.ball_len[i];
    const int* nb = a.nbr + (size_t)i * a.n;
#pragma unroll 1
    for (int t = 1; t < L; ++t) {
        const int k = nb[t];
        if (k > i) release(a, k);
    }
}

// Speculation.  At delta < 1 a center can wait on earlier centers (a chain of dependency
// levels), so CTAs can find the queue empty.  Such a CTA solves ahead the lowest-index node
// that is still undecided: its center column and every later ball member not owned by an
// earlier center at that moment, all written to the node's own weight slots.  Ownership only
// moves to earlier centers, so the columns the node needs if it does become a center are a
// subset of these, and their arithmetic is the same as in a regular solve (the columns of a
// factorization are independent); the center then only runs the test and publishes.  A node
// that ends up covered wastes its speculative solve, done while the CTA would have been idle.
__device__ inline int pick_spec(const SolveArgs& a) {
    const int k = atomicAdd(&a.ctr->spec_next, 1);  // one candidate per idle poll
    if (k >= a.N || *((volatile int*)&a.state[k]) != kUndecided) return -1;
    return atomicCAS(&a.spec[k], 0, 1) == 0 ? k : -1;
}

// One CTA per center.  Thread 0 claims the next queue slot and waits (bounded) for it to be
// filled; the CTA then solves the center, tests and writes its columns, and resolves the
// traversal state of its ball members.
// Registers are capped per team size (team_min_blocks) so that the CTAs that fit an SM's
// shared memory also fit its register file.  CHUNKED (LDL^T only) is the instantiation for
// plans whose largest ball has more columns than one factorization carries; the other one
// has no code for later chunks, so it keeps the registers of the one-chunk path.
template <int D, int LAY, int NT, bool CHUNKED>
__global__ void __launch_bounds__(NT, min_blocks(LAY, NT)) k_traversal(SolveArgs a, size_t per_cta, int basis_bytes) {
    extern __shared__ __align__(16) char smem[];
    __shared__ int s_j, s_q, s_rej, s_own, s_k, s_sp, s_ref, s_refonly;
    const short* sbasis = load_basis(smem, a.basis, a.basis_count);
    SmemOf<LAY> sm;
    if constexpr (LAY == kNull) carve_ns<D>(smem + basis_bytes, a.n, a.M, a.qcap, a.qmax, sm);
    else carve<D, LAY == kPacked>(smem + basis_bytes, a.n, a.K, a.qmax, a.stride, sm);
    __syncthreads();
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int ns = a.n, N = a.N;  // ns: row stride of nbr and of a weight slot
    const double nan = __longlong_as_double(0x7ff8000000000000LL);
    int slot = -1;  // thread 0: the claimed queue slot, kept while the CTA speculates

    for (;;) {
        if (tid == 0) {
            int j = -1, k = -1, sp = 0;
            bool leave = false;
            if (slot < 0 && a.elastic > 0) {
                // Elastic grid: holding no slot, this CTA may leave; the CTAs that hold the
                // unfilled slots (at least a.elastic of them) process every entry still to
                // come, and none of them leaves while it holds one.
                const int waiting = *((volatile int*)&a.ctr->q_head) - *((volatile int*)&a.ctr->q_tail);
                leave = waiting >= a.elastic;
            }
            if (slot < 0 && !leave) slot = atomicAdd(&a.ctr->q_head, 1);
            if (!leave && slot < N) {
                const unsigned long long t0 = globaltimer_ns();
                unsigned nsl = 32;
                for (;;) {
                    j = *((volatile int*)&a.queue[slot]);
                    if (j >= 0) break;
                    if (*((volatile int*)&a.ctr->done) >= N || *((volatile int*)&a.ctr->abort) != 0) {
                        j = -1;
                        break;
                    }
                    if (globaltimer_ns() - t0 > a.timeout_ns) {
                        set_error(a.ctr, RBFFD_ETIMEOUT);
                        atomicExch(&a.ctr->abort, 1);
                        j = -1;
                        break;
                    }
                    if (a.spec && (k = pick_spec(a)) >= 0) break;  // idle: solve ahead
                    __nanosleep(nsl);
                    if (nsl < 2048) nsl <<= 1;
                }
            }
            if (j >= 0) {
                slot = -1;
                if (a.spec) sp = *((volatile int*)&a.spec[j]);
                fence_gpu();  // acquire what the centers that released j (or its solve) published
            }
            s_j = j;
            s_k = k;
            s_sp = sp;
            s_rej = 0;
            s_own = 0;
        }
        __syncthreads();
        const int jc = s_j, ks = s_k;
        if (jc < 0 && ks < 0) break;
        const bool ahead = jc < 0;           // a speculative solve of node ks
        const bool made = !ahead && s_sp == 2;  // center jc whose solve was made ahead
        const int j = ahead ? ks : jc;
        const Shape sh = shape_of<D>(a, sbasis, j);
        const int n = sh.n;

        // columns: the center and every later ball member not already kept by an earlier center.
        // With the centroid reference of the Lebesgue test, the reference node's column goes to
        // position 1 (after the center), and is solved as one more column when it is not such
        // a member (reference only: never kept).
        const int L = a.ball_len[j];
        if (wid == 0) {
            int q = 0;
#pragma unroll 1
            for (int t0 = 0; t0 < n; t0 += 32) {
                const int t = t0 + lane;
                bool inc = false;
                if (t < L) {
                    if (t == 0) inc = true;
                    else {
                        const int i = a.nbr[(size_t)j * ns + t];
                        inc = (i > j) && (__ldcg(&a.owner[i]) >= j) && !(a.bc && a.bc[i]);
                    }
                }
                const unsigned bal = __ballot_sync(0xffffffffu, inc);
                const int pos = q + __popc(bal & ((1u << lane) - 1u));
                if (inc) sm.cols[pos] = t;
                if (t < n) sm.colof[t] = inc ? pos : -1;
                q += __popc(bal);
            }
            __syncwarp();
            if (lane == 0) {
                int ref = 0, only = 0;
                if (a.ref_pos) {
                    const int tref = a.ref_pos[j];
                    if (tref > 0) {  // the reference column to position 1
                        int p = sm.colof[tref];
                        if (p < 0) { p = q++; sm.cols[p] = tref; only = 1; }
                        const int t1 = sm.cols[1];
                        sm.cols[1] = tref; sm.colof[tref] = 1;
                        sm.cols[p] = t1; sm.colof[t1] = p;
                        ref = 1;
                    }
                }
                s_q = q;
                s_ref = ref;
                s_refonly = only;
            }
        }
        __syncthreads();
        const int q = s_q;
        const long long base = a.slot_off[j];
        double r2c = a.rho2[j];
        if (__double_as_longlong(r2c) <= 0) r2c = 1.0;
        const double inv_r2 = rcp_fixed(r2c);
        bool ok = true;
        // The columns pass through the right-hand-side block a.qcap at a time: the first chunk
        // is carried through the factorization, later ones use the stored factors (LDL^T only;
        // with LU a.qcap covers every ball).  A center whose solve was made ahead only reads
        // its Lebesgue values.  A ball always holds its center, so q >= 1.
        if (made) {
#pragma unroll 1
            for (int c = tid; c < q; c += NT) sm.lam[c] = __ldcg(&a.slot_lam[base + sm.cols[c]]);
        } else {
            const int q1 = CHUNKED ? min(q, a.qcap) : q;
            if constexpr (LAY == kNull) {
                ok = ns_solve<D, NT>(a, sh, j, q, q1, sm, 0);
                if (ok) ns_lebesgue<NT>(sh, 0, q1, sm);
            } else {
                ok = solve_local<D, LAY == kPacked, NT>(a, sh, j, q1, sm, s_ref);
                if (ok) lebesgue_values<NT>(n, sh.K, q1, sm);
            }
        }
        __syncthreads();
        const int qc = (CHUNKED && !made) ? min(q, a.qcap) : q;
        // the solved columns c0 .. c0+qk-1 (held in sm.X as 0 .. qk-1) to the weight slots
        auto emit = [&](int c0, int qk) {
            const int cref = s_ref;                       // the test's reference column
            const int conly = s_refonly ? cref : -1;      // a reference-only column
            if (ahead) {  // every column goes to the node's own slots
                if (!ok) return;
#pragma unroll 1
                for (int e = tid; e < qk * n; e += NT) {
                    const int c = e / n, r = e - c * n;
                    if (c0 + c == conly) continue;
                    a.slot_w[(base + sm.cols[c0 + c]) * ns + r] = weight(sh, r, c0, c, sm) * inv_r2;
                }
#pragma unroll 1
                for (int c = tid; c < qk; c += NT)
                    if (c0 + c != conly) a.slot_lam[base + sm.cols[c0 + c]] = sm.lam[c0 + c];
                return;
            }
            // Lebesgue test (§4.2.1) per column; the center keeps its own row
            int failed = 0, own = 0;
#pragma unroll 1
            for (int c = c0 + tid; c < c0 + qk; c += NT) {
                if (c == conly) { sm.keep[c] = 0; continue; }
                const double lam = ok ? sm.lam[c] : nan;
                const bool test_ok =
                    ok && (c == 0 || __double_as_longlong(lam) <= __double_as_longlong(sm.lam[cref]));
                bool keep;
                if (!ok) keep = (c == 0);
                else if (a.mode != RBFFD_STAB_SEQ) keep = true;
                else keep = test_ok;
                sm.keep[c] = keep ? 1 : 0;
                a.slot_lam[base + sm.cols[c]] = lam;
                a.slot_pass[base + sm.cols[c]] = (c == 0 || test_ok) ? 1 : 0;
                failed += c > 0 && !test_ok;
                own += keep && (a.mode != RBFFD_STAB_FALLBACK || c == 0 || test_ok);
            }
            if (failed) atomicAdd_block(&s_rej, failed);
            if (own) atomicAdd_block(&s_own, own);
            __syncthreads();
#pragma unroll 1
            for (int e = tid; !made && e < qk * n; e += NT) {  // (made ahead: already in the slots)
                const int c = e / n, r = e - c * n;
                if (!sm.keep[c0 + c]) continue;
                a.slot_w[(base + sm.cols[c0 + c]) * ns + r] =
                    ok ? weight(sh, r, c0, c, sm) * inv_r2 : nan;
            }
        };
        emit(0, qc);
        if constexpr (CHUNKED) {
#pragma unroll 1
            for (int c0 = qc; c0 < q; c0 += qc) {  // later chunks (more columns than a.qcap)
                const int qk = min(qc, q - c0);
                __syncthreads();  // sm.X is read until here
                // (the shape is read again rather than kept in registers)
                if (ok) {
                    if constexpr (LAY == kNull) ok = ns_solve_chunk<D, NT>(a, shape_of<D>(a, sbasis, j), j, c0, qk, sm);
                    else solve_chunk<D, NT>(a, shape_of<D>(a, sbasis, j), c0, qk, sm, j, s_ref);
                }
                __syncthreads();
                emit(c0, qk);
            }
        }
        if (ahead) {  // publish every column, then the node's flag
            __syncthreads();
            if (tid == 0) {
                fence_gpu();
                atomicExch(&a.spec[j], ok ? 2 : 3);
                atomicAdd(&a.ctr->n_spec, 1ull);
            }
            continue;
        }
        // ownership: the earliest center keeping a row owns it
#pragma unroll 1
        for (int c = tid; c < q; c += NT) {
            if (c > 0 && sm.keep[c]) atomicMin(&a.owner[a.nbr[(size_t)j * ns + sm.cols[c]]], j);
        }
        __syncthreads();
        // resolve: kept members become covered; every later ball member loses a dependency.
        // Each publishing thread fences first, so the CTA's ownership updates (ordered before
        // it by the barrier) are visible wherever its state changes are.
#pragma unroll 1
        for (int t = 1 + tid; t < L; t += NT) {
            const int i = a.nbr[(size_t)j * ns + t];
            if (i <= j) continue;
            const int c = sm.colof[t];
            const bool kept = c >= 0 && sm.keep[c];
            fence_gpu();
            if (kept && atomicCAS(&a.state[i], kUndecided, kCovered) == kUndecided) on_covered(a, i);
            release(a, i);
        }
        if (tid == 0) {
            if (!ok) {
                atomicAdd(&a.ctr->n_singular, 1);
                set_error(a.ctr, RBFFD_ESINGULAR);
            }
            const unsigned long long K = (unsigned long long)sh.K;
            atomicAdd(&a.ctr->sum_k3, K * K * K);
            atomicAdd(&a.ctr->sum_k2q, K * K * (unsigned long long)s_own);
            atomicAdd(&a.ctr->sum_k2c, K * K * (unsigned long long)q);
            atomicAdd(&a.ctr->n_centers, 1ull);
            atomicAdd(&a.ctr->sum_cols, (unsigned long long)q);
            atomicAdd(&a.ctr->n_rejected, (unsigned long long)s_rej);
            if (made) atomicAdd(&a.ctr->n_spec_used, 1ull);
            atomicAdd(&a.ctr->done, 1);
        }
        __syncthreads();
    }
}

// FALLBACK re-solves (one right-hand side each), one launch per stencil class: `cls` is the
// degree this launch handles (-1: all), n_cls/K_cls the largest stencil/system of the class,
// so shared memory is sized for the class and a single column.
template <int D, int LAY, int NT>
__global__ void __launch_bounds__(NT, min_blocks(LAY, NT)) k_fallback_solve(SolveArgs a, int cls, int n_cls,
                                                           int K_cls, int xs_cls,
                                                           int basis_bytes) {
    extern __shared__ __align__(16) char smem[];
    const short* sbasis = load_basis(smem, a.basis, a.basis_count);
    SmemOf<LAY> sm;
    if constexpr (LAY == kNull) carve_ns<D>(smem + basis_bytes, n_cls, K_cls - n_cls, 1, 1, sm);
    else carve<D, LAY == kPacked>(smem + basis_bytes, n_cls, K_cls, 1, xs_cls, sm);
    __syncthreads();
    const int tid = threadIdx.x;
    const int count = *((volatile int*)&a.ctr->fb_count);
    const double nan = __longlong_as_double(0x7ff8000000000000LL);
    for (int w = blockIdx.x; w < count; w += gridDim.x) {
        const int i = a.fb_list[w];
        if (cls >= 0 && (int)a.node_ell[i] != cls) continue;  // another class's launch
        const int kind = a.bc ? (int)a.bc[i] : 0;  // boundary rows (§5) share this launch
        const Shape sh = shape_of<D>(a, sbasis, i);
        const long long slot = a.slot_off[i];
        if (kind == 1) {  // Dirichlet: the identity row, exactly
            for (int r = tid; r < sh.n; r += NT) a.slot_w[slot * a.n + r] = (r == 0) ? 1.0 : 0.0;
            if (tid == 0) a.slot_lam[slot] = 1.0;
            continue;
        }
        for (int t = tid; t < sh.n; t += NT) sm.colof[t] = (t == 0) ? 0 : -1;
        if (tid == 0) sm.cols[0] = 0;
        __syncthreads();
        bool ok;
        if constexpr (LAY != kNull) {
            assemble_local<D, LAY == kPacked, NT>(a, sh, i, 1, sm);
            if (kind == 2) {
                neumann_rhs<D, NT>(sh, a.nrm + (size_t)i * D, sm);
                __syncthreads();
            }
        }
        if constexpr (LAY == kNull) {
            ok = ns_solve<D, NT, true>(a, sh, i, 1, 1, sm, kind);
            if (ok) ns_lebesgue<NT>(sh, 0, 1, sm);
        } else if constexpr (LAY == kPacked) {
            double* gA = refine_scratch<NT, true>(a);
            if (gA) copy_full_matrix<NT>(sh.K, sm, gA);
            ok = factor_solve_ldlt<NT, true>(sh.K, 1, sm);
            if (ok && gA) refine_columns<D, NT>(a, sh, 0, 1, sm, gA, gA + a.rs_x0, kind, i);
        } else {
            ok = factor_solve_lu<NT>(sh.K, 1, sm);
        }
        if constexpr (LAY != kNull) {
            if (ok) lebesgue_values<NT>(sh.n, sh.K, 1, sm);
        }
        __syncthreads();
        double r2c = a.rho2[i];
        if (__double_as_longlong(r2c) <= 0) r2c = 1.0;
        // weights of the scaled problem times rho^-2 (Laplacian) or rho^-1 (normal derivative)
        const double scale = kind == 2 ? rcp_fixed(sqrt(r2c)) : rcp_fixed(r2c);
        int en = 0;
        if constexpr (LAY == kNull) {
            double nv[D];
            if (kind == 2) en = scaled_normal<D>(a, i, nv);
        }
        for (int r = tid; r < sh.n; r += NT)
            a.slot_w[slot * a.n + r] = ok ? scalbn(weight(sh, r, 0, 0, sm), en) * scale : nan;
        if (tid == 0) {
            a.slot_lam[slot] = ok ? scalbn(sm.lam[0], en) : nan;
            if (!ok) {
                atomicAdd(&a.ctr->n_singular, 1);
                set_error(a.ctr, RBFFD_ESINGULAR);
            }
            const unsigned long long K = (unsigned long long)sh.K;
            atomicAdd(&a.ctr->sum_k3, K * K * K);
            atomicAdd(&a.ctr->sum_k2q, K * K);
            atomicAdd(&a.ctr->sum_k2c, K * K);
            if (kind == 0) atomicAdd(&a.ctr->n_fallback, 1ull);
            atomicAdd(&a.ctr->sum_cols, 1ull);
        }
        __syncthreads();
    }
}

}  // namespace rbffd

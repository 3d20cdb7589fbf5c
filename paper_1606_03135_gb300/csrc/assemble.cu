// assemble.cu -- the overlapped RBF-FD traversal (§4.1) with local L-Lebesgue stabilization
// (§4.2.1), the local FP64 solves, the CSR scatter and y = L u.
//
// Traversal as a dataflow.  The sequential rule "visit k = 0..N-1; an uncovered k becomes a
// center and keeps the members of its retention ball that pass the Lebesgue test" has a
// unique outcome: k is a center iff no earlier center keeps it, and a row belongs to the
// earliest center keeping it.  Whether center j keeps node i depends only on stencil j and
// x_i, so node k's fate is final as soon as every earlier node whose ball contains k (its
// in-neighbours, counted in `indeg`) is final.  A persistent kernel runs this: a node whose
// in-neighbours are all final and none kept it is pushed to a work queue as a center; a CTA
// pops it, factors its local system once, solves the right-hand sides of its still-open
// ball members, and then (i) marks the members it keeps as covered and (ii) releases one
// dependency of each later ball member.  Every device-side wait is bounded by a timeout and
// ends the kernel with RBFFD_ETIMEOUT.
//
// Local solve (one team of 32 to 512 threads per stencil).  The (n+M) x (n+M) saddle-point
// matrix [A P; P^T 0] of §4.1 and the q right-hand sides of the overlapped system (one per
// solved ball member) are formed in shared memory.  Most plans of one stencil shape with r^7 or
// below solve in the null space of P^T (nullspace.cuh: most of the work in fixed point on the
// integer pipe; the plan's rule stands in api.cu).  For the others the
// lower triangle is stored packed and factored as L D L^T with Bunch-Kaufman pivoting, the
// right-hand sides carried along ((1/3) K^3 + 2 K^2 q flops); the paper's
// partial-pivot LU of the full [A_hat | B_hat] array ((2/3) K^3 + 2 K^2 q) is the
// RBFFD_FACTOR_LU option.  Every FP64 warp instruction occupies all 32 lanes of the narrow
// FP64 pipe whatever its active mask, so the updates are flattened over (row, column) pairs
// to keep lanes busy, and scalar work (pivot tests, reciprocals, square roots) is moved to
// the integer and FP32 pipes where it can be.
//
// Own-stencil rows (one right-hand side): FALLBACK re-solves of rows that failed the test,
// and the boundary rows of §5 (Dirichlet identity, Neumann normal derivative).
#include <cuda_runtime.h>

#include <mutex>

#include "rbffd_internal.cuh"
#include "traversal.cuh"

namespace rbffd {

// Bytes of one CTA's local system; *stride_out is S (full) or xs (packed).
size_t solve_smem_per_cta(int n, int K, int qcap, int qmax, int D, int lay, int* stride_out) {
    if (lay == kLayNull) {
        if (stride_out) *stride_out = 0;
        return ns_smem_bytes(n, K - n, qcap, qmax, D);
    }
    const bool packed = lay == kLayPacked;
    int stride = packed ? qcap : K + qcap;
    if ((stride & 1) == 0) ++stride;  // odd row stride: column walks hit distinct banks
    if (stride_out) *stride_out = stride;
    const size_t mat = packed ? ((size_t)tri(K) + 1) / 2 * 2 + (size_t)K * stride
                              : (size_t)K * stride;
    size_t b = mat * 8 + (size_t)n * D * 8 + (size_t)K * 4 * 8 + (size_t)qmax * 8 +
               (size_t)(qmax + n) * 4 + (size_t)K * 2 * 4 + (size_t)K + (size_t)qmax;
    return (b + 15) & ~size_t(15);
}

size_t basis_smem_bytes(int count) { return ((size_t)count * sizeof(short) + 15) & ~size_t(15); }

__global__ void k_traversal_init(int N, const int* __restrict__ indeg,
                                 const unsigned char* __restrict__ bc, int* state, int* pending,
                                 int* owner, int* queue, unsigned char* fb_flag, int* spec,
                                 int* sd_lock, int sd_slots) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
        state[i] = (bc && bc[i]) ? kBoundary : kUndecided;
        if (spec) spec[i] = 0;
        pending[i] = indeg[i];
        owner[i] = kNoOwner;
        queue[i] = -1;
        fb_flag[i] = 0;
        if (i < sd_slots) sd_lock[i] = 0;  // (sd_slots <= N)
    }
}

// Boundary nodes (§5) take no part in the overlapped traversal: each releases the later
// members of its ball (which counted it as a possible center), is done at once, and is queued
// for its own-stencil row with the fallback rows.
__global__ void k_boundary_release(SolveArgs a) {
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < a.N; q += gridDim.x * blockDim.x) {
        if (!a.bc[q]) continue;
        const int* nb = a.nbr + (size_t)q * a.n;
        for (int t = 1; t < a.ball_len[q]; ++t)
            if (nb[t] > q) atomicSub(&a.pending[nb[t]], 1);
        a.owner[q] = q;
        a.fb_flag[q] = 1;
        a.fb_list[atomicAdd(&a.ctr->fb_count, 1)] = q;
        atomicAdd(&a.ctr->done, 1);
    }
}

__global__ void k_traversal_seed(SolveArgs a) {
    if (a.no_seed) return;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < a.N; i += gridDim.x * blockDim.x) {
        if (a.pending[i] == 0 && a.state[i] == kUndecided) {
            a.state[i] = kCenter;
            a.owner[i] = i;
            push_center(a, i);
        }
    }
}

// Reference point of the Lebesgue test in its centroid reading (§4.2.1): for every node j,
// the position in its stencil (n_j nodes) of the node nearest the stencil's centroid; one warp
// per node.  The centroid is the mean of the stencil's nodes: lane 0 sums each coordinate in
// kNN order from 0.0 and divides by n_j (at most 128 additions per coordinate, once per plan),
// then broadcasts it; ties in the distance go to the lower position.  It depends on the
// stencil only, so it runs once per plan, before the traversal.
template <int D>
__global__ void k_centroid_ref(const double* X, const int* nbr, const int* node_n, int N, int ns,
                               unsigned char* ref_pos) {
    const int lane = threadIdx.x & 31;
    const int j = (int)((blockIdx.x * (size_t)blockDim.x + threadIdx.x) >> 5);
    if (j >= N) return;  // (warp-uniform)
    const int n = node_n ? node_n[j] : ns;
    const int* nb = nbr + (size_t)j * ns;
    double c[D];
#pragma unroll
    for (int d = 0; d < D; ++d) {
        double s = 0.0;
        if (lane == 0) {
            for (int t = 0; t < n; ++t) s = __dadd_rn(s, __ldg(&X[(size_t)nb[t] * D + d]));
            s = __ddiv_rn(s, exact_double(n));
        }
        c[d] = __shfl_sync(0xffffffffu, s, 0);
    }
    unsigned long long best = ~0ull;  // this lane's smallest squared distance (bits; r2 >= 0)
    int tb = 0x7fffffff;              // and its lowest position
    for (int t = lane; t < n; t += 32) {
        const unsigned long long k =
            (unsigned long long)__double_as_longlong(sqdist_rn<D>(X + (size_t)nb[t] * D, c));
        if (k < best) { best = k; tb = t; }
    }
    unsigned long long m = best;
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long v = __shfl_xor_sync(0xffffffffu, m, o);
        m = v < m ? v : m;
    }
    const unsigned t = __reduce_min_sync(0xffffffffu, best == m ? (unsigned)tb : 0x7fffffffu);
    if (lane == 0) ref_pos[j] = (unsigned char)t;
}

// FALLBACK mode: rows whose owner column failed the test get their own delta = 1 stencil.
__global__ void k_fallback_collect(SolveArgs a) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < a.N; i += gridDim.x * blockDim.x) {
        const int s = a.owner[i];
        if (s == i || s == kNoOwner) continue;
        const int* nb = a.nbr + (size_t)s * a.n;
        const int L = a.ball_len[s];
        int t = -1;
        for (int u = 1; u < L; ++u)
            if (nb[u] == i) { t = u; break; }
        if (t < 0) { set_error(a.ctr, RBFFD_ECUDA); continue; }
        if (!a.slot_pass[a.slot_off[s] + t]) {
            a.fb_flag[i] = 1;
            a.fb_list[atomicAdd(&a.ctr->fb_count, 1)] = i;
        }
    }
}

// Per-node stencils only: the length of every row (the size of the stencil that produced
// it), into `len`, for the row-pointer scan.
__global__ void k_row_len(SolveArgs a, int* __restrict__ len) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < a.N; i += gridDim.x * blockDim.x) {
        const int s = a.fb_flag[i] ? i : a.owner[i];
        len[i] = (s == kNoOwner) ? 0 : a.node_n[s];
    }
}

// CSR: row i takes the weights of the column computed for it by its owner stencil (or its
// own fallback stencil), with the columns sorted ascending.  Uniform stencils: row i starts
// at i n; per-node stencils: row_ptr was scanned from the row lengths.
__global__ void __launch_bounds__(256) k_finalize(SolveArgs a, long long* __restrict__ row_ptr,
                                                  int* __restrict__ col, double* __restrict__ val,
                                                  double* __restrict__ lam_row,
                                                  unsigned char* __restrict__ is_center) {
    extern __shared__ int fin_smem[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, wpb = blockDim.x >> 5;
    const int ns = a.n;
    const bool uniform = a.node_n == nullptr;
    int* cs = fin_smem + wib * ns;
    for (int i = blockIdx.x * wpb + wib; i < a.N; i += gridDim.x * wpb) {
        const bool fb = a.fb_flag[i] != 0;
        const int s = fb ? i : a.owner[i];
        if (s == kNoOwner) {
            if (lane == 0) set_error(a.ctr, RBFFD_ECUDA);
            continue;
        }
        const int n = uniform ? ns : a.node_n[s];
        int t = 0;
        if (s != i) {
            const int L = a.ball_len[s];
            int found = -1;
            for (int u0 = 1; u0 < L; u0 += 32) {
                const int u = u0 + lane;
                const bool hit = u < L && a.nbr[(size_t)s * ns + u] == i;
                const unsigned b = __ballot_sync(0xffffffffu, hit);
                if (b && found < 0) found = u0 + __ffs(b) - 1;
            }
            t = found;
            if (t < 0) {
                if (lane == 0) set_error(a.ctr, RBFFD_ECUDA);
                continue;
            }
        }
        const long long slot = a.slot_off[s] + t;
        const long long rp = uniform ? (long long)i * ns : row_ptr[i];
        for (int r = lane; r < n; r += 32) cs[r] = a.nbr[(size_t)s * ns + r];
        __syncwarp();
        for (int r = lane; r < n; r += 32) {
            const int c = cs[r];
            int rank = 0;
            for (int u = 0; u < n; ++u) rank += cs[u] < c;
            col[rp + rank] = c;
            val[rp + rank] = a.slot_w[slot * ns + r];
        }
        if (lane == 0) {
            if (fb) a.owner[i] = i;  // a fallback row names its own stencil
            if (uniform) {
                row_ptr[i] = rp;
                if (i == a.N - 1) row_ptr[a.N] = (long long)a.N * ns;
            }
            lam_row[i] = a.slot_lam[slot];
            is_center[i] = fb ? ((a.bc && a.bc[i]) ? 3 : 2) : (s == i ? 1 : 0);
        }
        __syncwarp();
    }
}

// y = L u, kSpmvLanes lanes per row.  An FP64 warp instruction takes 16 cycles of the SM's FP64
// units however many lanes it uses, so a whole warp per row was bound by its reduction: two FMAs
// and five shuffle-adds per row of 45 entries, 36 us of FP64 issue for N = 100,000 (53 us in all,
// against 8 us for the matrix's bytes).  Four lanes per row take 12 FMAs and two adds for eight
// rows, 9 us.  Each lane keeps four entries in flight (values, columns, then the gathers of u):
// 20.6 us, the latency of the gathers and the loads of the matrix.
constexpr int kSpmvLanes = 4;
__global__ void __launch_bounds__(256) k_spmv(int N, const long long* __restrict__ row_ptr,
                                              const int* __restrict__ col,
                                              const double* __restrict__ val,
                                              const double* __restrict__ u, double* __restrict__ y) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int l = (int)(t & (kSpmvLanes - 1));
    const int i = (int)min(t / kSpmvLanes, (long long)N - 1);  // (whole warps reach the shuffles)
    const long long b = row_ptr[i], e = row_ptr[i + 1];
    double s = 0.0;
    for (long long k = b + l; k < e; k += 4 * kSpmvLanes) {
        double v[4], x[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const long long kk = k + j * kSpmvLanes;
            const bool in = kk < e;
            v[j] = in ? __ldg(&val[kk]) : 0.0;
            x[j] = in ? __ldg(&u[__ldg(&col[kk])]) : 0.0;
        }
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (k + j * kSpmvLanes < e) s = fma(v[j], x[j], s);
    }
    for (int o = kSpmvLanes / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (l == 0 && t / kSpmvLanes < N) y[i] = s;
}

// Values of the time-stepping matrix of §5 on L's pattern, one warp per row: interior rows
// e_i - c L_i, boundary rows unchanged.  Rounded as 1 - c v and -(c v).
__global__ void __launch_bounds__(256) k_timestep(int N, const long long* __restrict__ row_ptr,
                                                  const int* __restrict__ col,
                                                  const double* __restrict__ val,
                                                  const unsigned char* __restrict__ bc, double c,
                                                  double* __restrict__ out) {
    const int lane = threadIdx.x & 31;
    const int wpb = blockDim.x >> 5;
    for (int i = blockIdx.x * wpb + (threadIdx.x >> 5); i < N; i += gridDim.x * wpb) {
        const bool boundary = bc && bc[i];
        for (long long k = row_ptr[i] + lane; k < row_ptr[i + 1]; k += 32) {
            const double v = val[k];
            const double cv = __dmul_rn(c, v);
            out[k] = boundary ? v : (col[k] == i ? __dsub_rn(1.0, cv) : -cv);
        }
    }
}

// ------------------------------------------------------------------ launchers
static int sm_count() {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    return v > 0 ? v : 1;
}

// The dynamic shared-memory limit is a per-kernel setting shared by every host thread, so it
// is always raised to the device maximum (never lowered to one plan's need): plans assembled
// concurrently on other streams cannot undercut each other's launches.  Raised once per
// (device, kernel); occupancy answers are cached per (device, kernel, block, shared memory),
// so planning does not repeat these driver queries while the GPU waits.
namespace {
struct SmemRaised { int dev; const void* k; };
struct OccEntry { int dev; const void* k; int nt; size_t smem; int per_sm; };
std::mutex g_attr_mu;
SmemRaised g_raised[128];
int g_n_raised = 0;
OccEntry g_occ[512];
int g_n_occ = 0;
}  // namespace

static cudaError_t allow_max_smem(const void* kern) {
    int dev = 0, mx = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lk(g_attr_mu);
    for (int i = 0; i < g_n_raised; ++i)
        if (g_raised[i].dev == dev && g_raised[i].k == kern) return cudaSuccess;
    cudaDeviceGetAttribute(&mx, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, kern);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             mx - (int)fa.sharedSizeBytes);
    if (e == cudaSuccess && g_n_raised < 128) g_raised[g_n_raised++] = {dev, kern};
    return e;
}

static cudaError_t occupancy(int* per_sm, const void* kern, int nt, size_t smem) {
    int dev = 0;
    cudaGetDevice(&dev);
    {
        std::lock_guard<std::mutex> lk(g_attr_mu);
        for (int i = 0; i < g_n_occ; ++i)
            if (g_occ[i].dev == dev && g_occ[i].k == kern && g_occ[i].nt == nt &&
                g_occ[i].smem == smem) {
                *per_sm = g_occ[i].per_sm;
                return cudaSuccess;
            }
    }
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, kern, nt, smem);
    if (e == cudaSuccess) {
        std::lock_guard<std::mutex> lk(g_attr_mu);
        if (g_n_occ < 512) g_occ[g_n_occ++] = {dev, kern, nt, smem, *per_sm};
    }
    return e;
}

// The traversal kernel for a layout and team size, or nullptr (LU has 128- and 512-thread teams
// and no chunked right-hand sides).
template <int D, bool CH>
static const void* packed_traversal_kernel(int nt) {
    switch (nt) {
        case 32: return (const void*)k_traversal<D, kPacked, 32, CH>;
        case 64: return (const void*)k_traversal<D, kPacked, 64, CH>;
        case 96: return (const void*)k_traversal<D, kPacked, 96, CH>;
        case kNT: return (const void*)k_traversal<D, kPacked, kNT, CH>;
        case kMidNT: return (const void*)k_traversal<D, kPacked, kMidNT, CH>;
        case kMaxNT: return (const void*)k_traversal<D, kPacked, kMaxNT, CH>;
        default: return nullptr;
    }
}

template <int D>
static const void* traversal_kernel(int lay, int nt, bool chunked) {
    if (lay == kNull) return null_traversal_kernel(D, nt, chunked);
    if (lay == kPacked)
        return chunked ? packed_traversal_kernel<D, true>(nt) : packed_traversal_kernel<D, false>(nt);
    if (chunked) return nullptr;
    return nt == kNT ? (const void*)k_traversal<D, kFull, kNT, false>
                     : (nt == kMaxNT ? (const void*)k_traversal<D, kFull, kMaxNT, false> : nullptr);
}

// The own-stencil kernel: 128-, 256- (not LU) and 512-thread teams.
template <int D>
static const void* fallback_kernel(int lay, int nt) {
    if (lay == kNull) return null_fallback_kernel(D, nt);
    if (lay == kPacked)
        return nt == kMaxNT   ? (const void*)k_fallback_solve<D, kPacked, kMaxNT>
               : nt == kMidNT ? (const void*)k_fallback_solve<D, kPacked, kMidNT>
                              : (const void*)k_fallback_solve<D, kPacked, kNT>;
    return nt == kMaxNT ? (const void*)k_fallback_solve<D, kFull, kMaxNT>
                        : (const void*)k_fallback_solve<D, kFull, kNT>;
}

// Resident CTAs per SM of a kernel (RBFFD_EINVAL: none, or no such kernel).
static int resident(const void* k, int nt, size_t smem, int* per_sm) {
    *per_sm = 0;
    if (!k) return RBFFD_EINVAL;
    if (RB_CUDA(allow_max_smem(k)) || RB_CUDA(occupancy(per_sm, k, nt, smem)) || *per_sm < 1)
        return RBFFD_EINVAL;
    return RBFFD_OK;
}

// Team size for a launch when none is forced: 128 threads when more than four stencils fit an
// SM's shared memory, 256 when two to four fit (LDL^T), else 512 so that the one resident
// stencil still keeps enough warps busy.  The LDL^T traversal takes 96 threads instead of 128
// unless that keeps fewer stencils resident: more stencils in flight hide more of each one's
// serial pivot steps (2D, K = 46,
// 13 columns: 13 stencils of 96 threads beat 12 of 128 by 7%), and at equal residency the
// smaller team wastes fewer lanes in its short steps (2D, 21 columns: 1.11 against 1.17 ms;
// 3D, K = 65, one column: 15.5 against 15.7 ms).  A
// forced size (32, 64, 96 and 256 exist for LDL^T only) is taken as given.
template <int D, bool TRAVERSAL>
static int pick_team(int lay, size_t smem, int force, int* nt_out, int* per_sm_out,
                     bool chunked = false, bool refined = false) {
    auto occ = [&](int nt, int* ps) {
        return resident(TRAVERSAL ? traversal_kernel<D>(lay, nt, chunked) : fallback_kernel<D>(lay, nt),
                        nt, smem, ps);
    };
    int nt = force, rc;
    if (refined && nt != 0 && !team_refines(nt)) return RBFFD_EINVAL;  // no refinement step there
    if (nt == 0 && lay == kNull) {
        // Null-space solves: a warp per system while at least 12 of them share an SM (enough warps
        // to hide each other's latency, no barriers), 128 threads down to five, 256 for two to
        // four, 512 for one.  Traversal ms (32 / 128 threads): 3D ball N = 100k delta 1.0 (16 systems
        // per SM) 9.1 / 10.8, 0.4 (8) 7.0 / 6.1, 0.2 (6) 9.0 / 6.5; 2D square N = 40k delta 1.0 (16)
        // 1.68 / 2.40, 0.3 (12) 0.86 / 0.85.  Plans that refine (not in 128-thread teams): 64 from
        // six systems on, else 256: 3D degree 4 N = 12k delta 1.0 (6; 64 / 256) 3.8 / 4.1, 0.4 (3)
        // 2.5 / 1.8.
        int per_sm = 0;
        if ((rc = occ(32, &per_sm))) return rc;
        const bool many = refined ? per_sm >= 6 : per_sm >= 5;
        nt = per_sm >= 12 ? 32 : (many ? (refined ? 64 : kNT) : (per_sm >= 2 ? kMidNT : kMaxNT));
    }
    if (nt == 0) {
        int per_sm = 0;
        if ((rc = occ(kNT, &per_sm))) return rc;
        // The fallback's one-column systems hide each other's serial pivot steps when two or
        // more share an SM (512-thread teams run one per SM: their registers fill it); two to
        // four per SM take 256-thread teams (mixed cube, K = 106, four per SM: 315 -> 302 ms
        // of fallback solves against 128-thread teams).
        // 256-thread teams exist for LDL^T only; their 64 registers let four share an SM,
        // where the 512-thread teams' registers allow one.
        const int mid = lay != kFull ? kMidNT : kMaxNT;
        nt = TRAVERSAL ? (per_sm <= 1 ? kMaxNT : ((per_sm <= 4 || refined) ? mid : kNT))
                       : (per_sm <= 1 ? kMaxNT : (per_sm <= 4 ? mid : kNT));
        if (TRAVERSAL && lay != kFull && nt == kNT) {
            int p96 = 0;
            if ((rc = occ(96, &p96))) return rc;
            if (p96 >= per_sm) nt = 96;
        }
    }
    if ((rc = occ(nt, per_sm_out))) return rc;
    *nt_out = nt;
    return RBFFD_OK;
}

// Host-side preparation, done once per plan (not per assembly, so that rbffd_assemble only
// enqueues stream work and can be captured in a CUDA graph): raise the kernels' shared-memory
// limit, choose team sizes and size the persistent grid from the occupancy.  fb[c] holds the
// fallback launch of stencil class c.
template <int D>
static int prepare(int lay, int n, int K, int qcap, int qmax, int basis_count, LaunchPlan* lp) {
    int stride = 0;
    const size_t bb = basis_smem_bytes(basis_count);
    const size_t smem = bb + solve_smem_per_cta(n, K, qcap, qmax, D, lay, &stride);
    int per_sm = 0, rc;
    lp->chunked = lay != kFull && qcap < qmax;
    if ((rc = pick_team<D, true>(lay, smem, lp->force_nt, &lp->nt, &per_sm, lp->chunked,
                                 lay != kFull && K >= lp->refine_min_K)))
        return rc;
    lp->grid = per_sm * sm_count();
    lp->smem = smem;
    for (int c = 0; c < lp->n_fb; ++c) {
        FallbackClass& f = lp->fb[c];
        const size_t fs = bb + solve_smem_per_cta(f.n, f.K, 1, 1, D, lay, &f.xs);
        if ((rc = pick_team<D, false>(lay, fs, 0, &f.nt, &per_sm))) return rc;
        f.grid = per_sm * sm_count();
        f.smem = fs;
    }
    return RBFFD_OK;
}

int prepare_solve_kernels(int D, int lay, int n, int K, int qcap, int qmax, int basis_count,
                          LaunchPlan* lp) {
    return D == 2 ? prepare<2>(lay, n, K, qcap, qmax, basis_count, lp)
                  : prepare<3>(lay, n, K, qcap, qmax, basis_count, lp);
}

template <int D>
static int traversal(const SolveArgs& a, const LaunchPlan& lp, const int* indeg, cudaStream_t s,
                     int* launches, cudaEvent_t ev0, cudaEvent_t ev1) {
    const int basis_bytes = (int)basis_smem_bytes(a.basis_count);
    const int tb = 256, nb = (a.N + tb - 1) / tb;
    k_traversal_init<<<nb, tb, 0, s>>>(a.N, indeg, a.bc, a.state, a.pending, a.owner, a.queue,
                                       a.fb_flag, a.spec, a.sd_lock, a.sd_slots);
    if (a.bc) {
        k_boundary_release<<<nb, tb, 0, s>>>(a);
        ++*launches;
    }
    k_traversal_seed<<<nb, tb, 0, s>>>(a);
    *launches += 2;
    int grid = min(lp.grid, a.N);
    if (a.max_ctas > 0) grid = min(grid, a.max_ctas);
    // A plain launch suffices: a worker only waits for queue entries that workers already
    // running will push (the smallest unresolved node is always ready once every center
    // that holds a claimed entry is solved), so progress needs no co-residency, and plans
    // on other streams can run beside this grid.
    if (ev0) cudaEventRecord(ev0, s);
    size_t per_cta = lp.smem - basis_bytes;
    int bb = basis_bytes;
    SolveArgs args = a;
    const void* k = traversal_kernel<D>(a.lay, lp.nt, lp.chunked);
    if (!k) return RBFFD_EINVAL;
    void* params[] = {&args, &per_cta, &bb};
    const cudaError_t e = cudaLaunchKernel(k, dim3(grid), dim3(lp.nt), params, lp.smem, s);
    if (ev1) cudaEventRecord(ev1, s);
    ++*launches;
    if (e != cudaSuccess) return RB_CUDA(e);
    return RB_LAUNCHED(__func__);
}

int launch_centroid_ref(int D, const double* X, const int* nbr, const int* node_n, int N, int ns,
                        unsigned char* ref_pos, cudaStream_t s, int* launches) {
    const int tb = 256, nb = (int)(((size_t)N * 32 + tb - 1) / tb);
    if (D == 2) k_centroid_ref<2><<<nb, tb, 0, s>>>(X, nbr, node_n, N, ns, ref_pos);
    else k_centroid_ref<3><<<nb, tb, 0, s>>>(X, nbr, node_n, N, ns, ref_pos);
    ++*launches;
    return RB_LAUNCHED(__func__);
}

int launch_traversal(int D, const SolveArgs& a, const LaunchPlan& lp, const int* indeg,
                     cudaStream_t s, int* launches, cudaEvent_t ev0, cudaEvent_t ev1) {
    return D == 2 ? traversal<2>(a, lp, indeg, s, launches, ev0, ev1)
                  : traversal<3>(a, lp, indeg, s, launches, ev0, ev1);
}

int launch_fallback(int D, const SolveArgs& a, const LaunchPlan& lp, cudaStream_t s,
                    int* launches) {
    const int tb = 256, nb = (a.N + tb - 1) / tb;
    if (a.mode == RBFFD_STAB_FALLBACK) {  // rows that failed the test (boundary rows are queued)
        k_fallback_collect<<<nb, tb, 0, s>>>(a);
        ++*launches;
    }
    int basis_bytes = (int)basis_smem_bytes(a.basis_count);
    for (int c = 0; c < lp.n_fb; ++c) {
        FallbackClass f = lp.fb[c];
        SolveArgs af = a;  // refinement scratch laid out for this class's systems
        af.rs_stride = f.rs_stride;
        af.rs_x0 = f.rs_x0;
        const void* k = D == 2 ? fallback_kernel<2>(a.lay, f.nt) : fallback_kernel<3>(a.lay, f.nt);
        if (!k) return RBFFD_EINVAL;
        void* params[] = {&af, &f.cls, &f.n, &f.K, &f.xs, &basis_bytes};
        const int rc = RB_CUDA(cudaLaunchKernel(k, dim3(f.grid), dim3(f.nt), params, f.smem, s));
        if (rc) return rc;
        ++*launches;
    }
    return RB_LAUNCHED(__func__);
}

int launch_finalize(const SolveArgs& a, long long* row_ptr, int* col, double* val,
                    double* lam_row, unsigned char* is_center, cudaStream_t s, int* launches) {
    if (a.node_n) {  // rows of different lengths: scan their lengths into row_ptr first
        const int tb = 256, nb = (a.N + tb - 1) / tb;
        k_row_len<<<nb, tb, 0, s>>>(a, a.fb_list);
        ++*launches;
        int rc = launch_scan_i32_to_i64(a.fb_list, row_ptr, a.N, s, launches);
        if (rc) return rc;
    }
    const int wpb = 8;
    const int blocks = (a.N + wpb - 1) / wpb;
    k_finalize<<<blocks, wpb * 32, wpb * a.n * sizeof(int), s>>>(a, row_ptr, col, val, lam_row,
                                                                is_center);
    ++*launches;
    return RB_LAUNCHED(__func__);
}

int launch_timestep(int N, const long long* row_ptr, const int* col, const double* val,
                    const unsigned char* bc, double c, double* out, cudaStream_t s, int* launches) {
    const int wpb = 8;
    const int blocks = (N + wpb - 1) / wpb;
    k_timestep<<<blocks, wpb * 32, 0, s>>>(N, row_ptr, col, val, bc, c, out);
    ++*launches;
    return RB_LAUNCHED(__func__);
}

int launch_spmv(int N, int n, const long long* row_ptr, const int* col, const double* val,
                const double* u, double* y, cudaStream_t s, int* launches) {
    (void)n;
    const int tb = 256;
    const unsigned blocks = (unsigned)(((long long)N * kSpmvLanes + tb - 1) / tb);
    k_spmv<<<blocks, tb, 0, s>>>(N, row_ptr, col, val, u, y);
    ++*launches;
    return RB_LAUNCHED(__func__);
}

}  // namespace rbffd

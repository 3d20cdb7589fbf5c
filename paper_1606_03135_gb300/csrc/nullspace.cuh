// nullspace.cuh -- local solves in the null space of the polynomial constraints.
//
// The saddle-point system [A P; P^T 0] [w; .] = [f; g] of a stencil with n nodes and M monomials
// is reduced instead of factored whole.  M of the nodes (the basic ones, chosen by partial
// pivoting) carry the constraints: with P1 and P2 the rows of P at the basic and the s = n - M
// other nodes, B = P2 P1^-1 and ghat = P1^-T g,
//
//   w_basic = ghat - B^T v,   w_other = v,   S v = f2 - B f1 - (A21 - B A11) ghat,
//   S = Z^T A Z = A22 - B A12 - A21 B^T + B A11 B^T,   Z = [-B^T; I].
//
// With C = A21 - B A11 / 2 this is S = A22 - C B^T - B C^T, and a right-hand side is one more
// row of both factors: (ghat, f1 - A11 ghat / 2) in the places of (B, C).  r^m is conditionally
// definite of order (m + 1) / 2, so S is definite whenever ell >= (m - 1) / 2 (the host's rule for
// this layout) and is factored as L D L^T without pivoting.
//
// Why: GB300 issues 2 FP64 FMAs per clock and SM, against 64 32x32+64-bit integer multiply-adds
// (measured: 2.0 and 62.6).  In this form two thirds of the work are the two matrix products,
// which run on the integer pipe in fixed point: operands are 59-bit integers in two limbs
// (v = hi 2^28 + lo, |lo| <= 2^27) scaled by a power of two per matrix, a product is three
// multiply-adds (hi hi, hi lo + lo hi; lo lo is below 2^-62 of the scale) and the sums are exact.
// A is that of r^m less a polynomial (KernelUnits in traversal.cuh), which S does not see and which
// makes its entries, and with them the units, up to 23 times smaller.
#pragma once

#include "fp64_int.cuh"
#include "rbffd_internal.cuh"

namespace rbffd {

// ------------------------------------------------------------------ fixed point
constexpr int kFixBits = 58;   // |v| < 2^58 for an operand below its scale 2^e: v = x 2^(58 - e)
constexpr int kLimbBits = 28;
constexpr int kPowerBits = 62;  // of phi and of f, which are not operands of products

// The conversions and dot products below that are used in several places are functions of their
// own, loops are not unrolled beyond what hides their latency, and quotients of small integers take
// an FP32 reciprocal: the kernels run the phases of up to 16 systems side by side on an SM, and with
// everything inlined (218 KB of code) waiting for instructions took a third of the time (3D ball,
// N = 100,000, delta = 1: 16.7 ms, against 9.9 ms at 128 KB).

// a / b of integers 0 <= a < 2^20, 0 < b.
__device__ __forceinline__ int small_div(int a, int b) {
    return (int)__fdividef((float)a + 0.5f, (float)b);
}

// e with |x| < 2^e (zero: a very small one).
__device__ __forceinline__ int scale_exp(double x) {
    return max((int)((abs_bits(x) >> 52) & 0x7ff) - 1022, -200);
}

// round(x 2^-u) for |x| < 2^(62 + u).
static __device__ __noinline__ long long to_fixed(double x, int u) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int ex = (int)((b >> 52) & 0x7ff);
    const unsigned long long t = ex == 0 ? 0ull : ((b & 0xFFFFFFFFFFFFFull) | (1ull << 52)) << 10;
    const int r = min(max(1085 + u - ex, 1), 63);  // x 2^-u = t 2^-r
    const long long v = (long long)((t + (1ull << (r - 1))) >> r);
    return (b >> 63) ? -v : v;
}

// The two limbs of v: v = hi 2^28 + lo, -2^27 <= lo < 2^27.
__device__ __forceinline__ int2 split_limbs(long long v) {
    const int hi = (int)((v + (1ll << (kLimbBits - 1))) >> kLimbBits);
    return make_int2(hi, (int)((unsigned)v - ((unsigned)hi << kLimbBits)));
}

__device__ __forceinline__ int2 to_limbs(double x, int e) { return split_limbs(to_fixed(x, e - kFixBits)); }

__device__ __forceinline__ long long join_limbs(int2 l) {
    return ((long long)l.x << kLimbBits) + l.y;
}

// The double nearest T 2^u (rounded half up), built with integer instructions.
static __device__ __noinline__ double from_fixed(long long T, int u) {
    if (T == 0) return 0.0;
    const unsigned long long sign = T < 0 ? 1ull << 63 : 0ull;
    const unsigned long long a = T < 0 ? 0ull - (unsigned long long)T : (unsigned long long)T;
    const int lz = __clzll((long long)a);
    const unsigned long long nrm = a << lz;  // top bit at 63
    const unsigned long long m = (nrm >> 11) + ((nrm >> 10) & 1ull);  // 2^52 <= m <= 2^53
    const unsigned long long ex = (unsigned long long)(63 - lz + u + 1022);
    return __longlong_as_double((long long)(sign | ((ex << 52) + m)));  // (m's top bit adds one)
}

// v 2^-r, rounded half up, 1 <= r <= 63.
__device__ __forceinline__ long long shift_right(long long v, int r) {
    return (v + (1ll << (r - 1))) >> r;
}

// v 2^sh, rounded for sh < 0 (half up).
__device__ __forceinline__ long long shift_fixed(long long v, int sh) {
    const int r = min(-sh, 63);
    return sh >= 0 ? v << sh : (v + (1ll << (r - 1))) >> r;
}

// x y 2^-56 of two integers below 2^59 in magnitude, from their limbs (error below 2 units).
__device__ __forceinline__ long long mul_limbs(int2 x, int2 y) {
    const long long h = (long long)x.x * y.x;
    const long long m = (long long)x.x * y.y + (long long)x.y * y.x;
    return h + ((m + (1ll << (kLimbBits - 1))) >> kLimbBits);
}

// e with |v| < 2^e of an integer.
__device__ __forceinline__ int int_exp(long long v) { return 64 - __clzll(v < 0 ? -v : v); }

// Square roots in fixed point.  For N = R 2^sh with sh even and N in [2^62, 2^64), m = N 2^-62 in
// [1, 4): returns sqrt(m) 2^60 to within about 2 units.  r0 = m y0 from an FP32 seed y0 of
// 1 / sqrt(m), e = 1 - r0 y0 (below 2^-21), and the series sqrt(m) = r0 (1 + e / 2 + 3 e^2 / 8 +
// O(e^3)).
__device__ __forceinline__ long long sqrt_core(unsigned long long N) {
    const int odd = (int)(N >> 63);
    const float mf = __int_as_float(((127 + odd) << 23) | (int)((N >> (39 + odd)) & 0x7fffffu));
    float yf;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(yf) : "f"(mf));
    const unsigned yb = __float_as_uint(yf);
    const unsigned Y = (((yb & 0x7fffffu) | 0x800000u) << 1) >> (127 - (yb >> 23));  // y0 2^24
    const unsigned long long r0 = ((unsigned long long)(unsigned)(N >> 32) * Y << 6) +
                                  ((unsigned long long)(unsigned)N * Y >> 26);  // 2^60 r0
    const long long e = (1ll << 60) - (long long)(((r0 >> 32) * Y << 8) + ((r0 & 0xffffffffull) * Y >> 24));
    const int e32 = (int)(e >> 10);  // 2^50 e
    const long long c = (e >> 1) + (((long long)e32 * e32) >> 43) * 3;  // 2^60 (e / 2 + 3 e^2 / 8)
    const int ch = (int)(c >> 16), cl = (int)(c & 0xffff);
    const int rh = (int)(r0 >> 31), rl = (int)(r0 & 0x7fffffff);  // (r0 may reach just above 2)
    const long long d = ((long long)rh * ch + (((long long)rh * cl) >> 16) + (((long long)rl * ch) >> 31)) >> 13;
    return (long long)r0 + d;
}

// A sum of products of limbs: h counts 2^(2 kLimbBits), m counts 2^kLimbBits.
struct LimbSum {
    long long h = 0, m = 0;
    __device__ __forceinline__ void mac(int2 x, int2 y) {
        h += (long long)x.x * y.x;
        m += (long long)x.x * y.y;
        m += (long long)x.y * y.x;
    }
    __device__ __forceinline__ void fold() {
        h += m >> kLimbBits;
        m &= (1ll << kLimbBits) - 1;
    }
    // in units 2^(ex + ey - 60) for operands of scales 2^ex and 2^ey
    __device__ __forceinline__ long long total() const {
        return h + ((m + (1ll << (kLimbBits - 1))) >> kLimbBits);
    }
};

constexpr int kSumUnit = 2 * kLimbBits - 2 * kFixBits;  // -60

// ------------------------------------------------------------------ shared-memory layout
// Row stride of the tableau and of C in 8-byte words: an odd multiple of 16 bytes, so 16-byte
// loads of consecutive rows hit distinct banks.  Systems of one column run in teams of one warp,
// for which more of them per SM count for more than a two-way conflict, so there the pad is left
// out (3D, M = 20, n = 45, N = 100k, delta = 1: 16 systems per SM instead of 14, 9.1 ms instead of
// 10.0; with it left out at delta 0.4 and 0.2 too, 128-thread teams took 1% longer) unless rows would
// then share a quarter of the banks (2D, M = 15: 1.95 ms instead of 1.68).
__host__ __device__ __forceinline__ int ns_ldm(int M, int qmax) {
    const int e = (M + 1) / 2;
    return 2 * (qmax > 1 || (e & 3) == 0 ? e | 1 : e);
}
// A column's row of X: ns_x2 words (M of them and a pad for odd M, or s), then s more.
__host__ __device__ __forceinline__ int ns_x2(int n, int M) {
    const int s = n - M, Mp = (M + 1) & ~1;
    return Mp > s ? Mp : s;
}
// (an odd multiple of 16 bytes, like ns_ldm)
__host__ __device__ __forceinline__ int ns_ldx(int n, int M) {
    return 2 * (((ns_x2(n, M) + n - M + 1) / 2) | 1);
}

// Start of column j of a packed lower triangle of s rows: entry (i, j) at col_start(j, s) + i.
__host__ __device__ __forceinline__ int col_start(int j, int s) { return (j * (2 * s - j - 1)) >> 1; }

struct NullSmem {
    // 8-byte words, each a 64-bit integer, two limbs or a double at different times:
    double* T;    // (n + qmax) x ldm tableau: rows 0..M-1 A11 (limbs) once the basic nodes are
                  //   chosen, M..n-1 B, n.. ghat of every column (and at last its basic weights)
    double* C;    // s x ldm: A21, C, its limbs
    double* S;    // lower triangle by columns, s x s (col_start): the products' sums, then S
                  //   (doubles), then the unscaled factor columns; may lie over A11
    double* X;    // one row of ldx words per column of the chunk: f1 (then f1 - A11 ghat / 2, its
                  //   limbs, the limbs of v), and from word x2 on f2 (then v, doubles)
    long long* xi;  // n x D scaled stencil coordinates (ns_coordinates)
    double* rd;   // s reciprocal pivots
    double* wb;   // s unscaled pivot column
    short* eg;    // qmax scale exponents of the ghat rows
    short* ev;    // qcap scale exponents of v
    double* lam;  // qmax Lebesgue values of the solved columns (all chunks)
    // (stencil positions and columns are below 128)
    unsigned char* order;  // n: stencil position of each tableau row
    unsigned char* pos;    // n: tableau row of each stencil position
    signed char* colof;    // n column of each ball position, or -1
    unsigned char* cols;   // qmax ball position of each solved column
    unsigned char* keep;  // qmax kept-for-coverage flags
    int ldm, ldx, x2;
};

// S takes A11's place once C is formed, unless later chunks of columns need A11 (or it is larger).
__host__ __device__ __forceinline__ bool ns_s_over_a11(int n, int M, int qcap, int qmax) {
    const int s = n - M;
    return qcap >= qmax && s * (s + 1) / 2 <= M * ns_ldm(M, qmax);
}

// Bytes of one CTA's local system in this layout.
__host__ __device__ __forceinline__ size_t ns_smem_bytes(int n, int M, int qcap, int qmax, int D) {
    const size_t s = n - M, ldm = ns_ldm(M, qmax);
    const size_t tri_words = ns_s_over_a11(n, M, qcap, qmax) ? 0 : s * (s + 1) / 2;
    const size_t words = (n + qmax + s) * ldm + qcap * (size_t)ns_ldx(n, M) + tri_words + n * D +
                         (qcap < qmax ? 2 * s : 0) + qmax;
    const size_t b = words * 8 + ((size_t)qmax + qcap) * 2 + 3 * (size_t)n + 2 * qmax;
    return (b + 15) & ~size_t(15);
}

template <int D>
__device__ __forceinline__ void carve_ns(char* p, int n, int M, int qcap, int qmax, NullSmem& sm) {
    const int s = n - M;
    sm.ldm = ns_ldm(M, qmax);
    sm.ldx = ns_ldx(n, M);
    sm.x2 = ns_x2(n, M);
    double* w = reinterpret_cast<double*>(p);
    sm.T = w;
    w += (n + qmax) * sm.ldm;
    sm.C = w;
    w += s * sm.ldm;
    sm.X = w;
    w += qcap * sm.ldx;
    sm.S = sm.T;
    if (!ns_s_over_a11(n, M, qcap, qmax)) {
        sm.S = w;
        w += s * (s + 1) >> 1;
    }
    sm.xi = reinterpret_cast<long long*>(w);
    sm.rd = w;  // (the coordinates are done with when S is factored, unless later chunks need them)
    w += n * D;
    if (qcap < qmax) {
        sm.rd = w;
        w += 2 * s;
    }
    sm.wb = sm.rd + s;
    sm.lam = w;
    w += qmax;
    short* h = reinterpret_cast<short*>(w);
    sm.eg = h;
    h += qmax;
    sm.ev = h;
    h += qcap;
    unsigned char* c = reinterpret_cast<unsigned char*>(h);
    sm.order = c;
    c += n;
    sm.pos = c;
    c += n;
    sm.colof = reinterpret_cast<signed char*>(c);
    c += n;
    sm.cols = c;
    c += qmax;
    sm.keep = c;
}

__device__ __forceinline__ int2* limbs(double* p) { return reinterpret_cast<int2*>(p); }
__device__ __forceinline__ long long* fixed(double* p) { return reinterpret_cast<long long*>(p); }

// ------------------------------------------------------------------ the constraints
__shared__ int s_ns_ok, s_ns_eb, s_ns_ec;

// A team's barrier.
template <int NT>
__device__ __forceinline__ void team_sync() {
    if constexpr (NT == 32) __syncwarp();
    else __syncthreads();
}

// 2^121 / a for a in [2^63, 2^64) (relative error below 2^-58), from an FP32 seed and one cubic step.
__device__ __forceinline__ long long rcp_norm(unsigned long long a) {
    float rf;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rf) : "f"(__int_as_float(0x3F800000 | (int)((a >> 40) & 0x7fffffu))));
    const unsigned rb = __float_as_uint(rf);  // r0 = 1 / m to 23 bits for m = a 2^-63, in (1/2, 1]
    const unsigned r = (((rb & 0x7fffffu) | 0x800000u) << 1) >> (127 - (rb >> 23));  // r0 2^24
    // e = 1 - m r0 in 2^-60, below 2^-21
    const long long e = (1ll << 60) - (long long)(((unsigned long long)(unsigned)(a >> 32) * r << 5) +
                                                  ((unsigned long long)(unsigned)a * r >> 27));
    const int e32 = (int)(e >> 10);
    const long long c = e + (((long long)e32 * e32) >> 40);  // 2^60 (e + e^2)
    return ((long long)r << 34) + (((long long)r * c) >> 26);  // 2^58 r0 (1 + e + e^2) = 2^121 / a
}

// The sum over j = 0..len-1 of a row's limbs and a column's (stride ldm), in 2^-56 of the product of
// their units: two terms per 16-byte load of the row.
static __device__ __noinline__ long long row_dot_col(const double* row, const double* col, int ldm, int len) {
    const int4* r = reinterpret_cast<const int4*>(row);
    const int2* c = reinterpret_cast<const int2*>(col);
    LimbSum t, u;  // (two chains)
    int j = 0;
#pragma unroll 1
    for (; j + 3 < len; j += 4) {
        const int4 x = r[j >> 1], y = r[(j >> 1) + 1];
        const int2 c0 = c[j * ldm], c1 = c[(j + 1) * ldm], c2 = c[(j + 2) * ldm], c3 = c[(j + 3) * ldm];
        t.mac(make_int2(x.x, x.y), c0);
        u.mac(make_int2(x.z, x.w), c1);
        t.mac(make_int2(y.x, y.y), c2);
        u.mac(make_int2(y.z, y.w), c3);
        if ((j & 28) == 28) { t.fold(); u.fold(); }
    }
#pragma unroll 1
    for (; j < len; ++j) t.mac(reinterpret_cast<const int2*>(row)[j], c[j * ldm]);
    t.fold();
    u.fold();
    t.h += u.h;
    t.m += u.m;
    return t.total();
}

// The constraints in fixed point.  Crout's LU with partial pivoting of the tableau (rows 0..n-1 of
// P, then q rows g): in step k column k of the rows k.. and then row k right of the diagonal are
// brought up to date by dot products with the finished columns and rows, so every entry is one
// exact sum, rounded once; pivots are picked among the nodes' rows and swapped to row k.  Then
// B = L2 L1^-1 and ghat = L_g L1^-1, a row per thread, again by dot products (columns from the
// last to the first).  A term costs 4.5 instructions (3 of them 32 x 32 + 64 bit multiply-adds) where
// the rank-1 form of Gauss-Jordan elimination, one rounding per term, took about 30.
//
// Units: 2^-kTabBits for P, U, L and B, times 2^gs for the rows of g (gs from the degree); entries
// must stay below 2^59 units (8, and 8 2^gs), pivots at least 2^-kPivotBits: a column's entries are
// held to 2^-57, so a small pivot has few bits left, and one below the unit would look like an exact
// zero (flat stencils, whose monomials z^k are small: with pivots near 2^-18 the weights of degree 2
// would be 30 times further off than the coordinates' rounding puts them, from 2^-12 on they are
// not).  Quasi-uniform, boundary and clustered stencils of degree 2 to 5 have pivots of 2^-9 and
// more.  Stencils that leave these ranges are noticed and done again in FP64.  Returns false on a range (uniformly).  On return the rows of B and ghat
// are limbs at the scales s_ns_eb (once the team has met) and sm.eg (at least eg_min; a row's
// absolute sum stays below 4 times its scale, which bounds the products' sums).
constexpr int kTabBits = 56, kPivotBits = 12;

__device__ __forceinline__ bool limb_overflow(long long v) {
    const int hi = (int)(v >> 32);
    return (hi ^ (hi >> 31)) >= 0x07ffff00;  // |v| 2^-59 near 1
}

template <int NT>
__device__ bool ns_eliminate_fixed(int n, int M, int q, int gs, int eg_min, const NullSmem& sm) {
    __shared__ long long s_y;
    __shared__ int s_sh, s_piv;
    constexpr unsigned kLeast = 1u << (kTabBits - kPivotBits - 28);  // in the search's 2^28 units
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int ldm = sm.ldm, R = n + q;
    double* T = sm.T;
    bool bad = false;
#pragma unroll 1
    for (int k = 0; k < M; ++k) {
#pragma unroll 1
        for (int i = k + tid; i < R; i += NT) {  // column k
            const long long v = fixed(T)[i * ldm + k] - row_dot_col(T + i * ldm, T + k, ldm, k);
            fixed(T)[i * ldm + k] = v;
            bad |= limb_overflow(v);
        }
        team_sync<NT>();
        if (wid == 0) {
            unsigned best = 0u;
            int p = 0x7fffffff;
#pragma unroll 1
            for (int i = k + lane; i < n; i += 32) {
                const long long t = fixed(T)[i * ldm + k];
                const unsigned v = (unsigned)((t < 0 ? -t : t) >> 28);
                if (v > best) { best = v; p = i; }
            }
            const unsigned top = __reduce_max_sync(0xffffffffu, best);
            p = (int)__reduce_min_sync(0xffffffffu, best == top ? (unsigned)p : 0x7fffffffu);
            if (top < kLeast) p = -1;
            if (p > k) {
#pragma unroll 1
                for (int c = lane; c < M; c += 32) {
                    const double t = T[p * ldm + c];
                    T[p * ldm + c] = T[k * ldm + c];
                    T[k * ldm + c] = t;
                }
                if (lane == 0) { const int t = sm.order[k]; sm.order[k] = sm.order[p]; sm.order[p] = t; }
                __syncwarp();
            }
            const long long d = fixed(T)[k * ldm + k];
            const unsigned long long a = (unsigned long long)(d < 0 ? -d : d);
            const int lz = __clzll((long long)a);
            if constexpr (NT == 32) {
                if (p < 0) return false;
            }
            const long long y = rcp_norm(a << (lz & 63));
            if (lane == 0) { s_y = d < 0 ? -y : y; s_sh = lz; s_piv = p; }
        }
        team_sync<NT>();
        if (NT > 32 && s_piv < 0) return false;
        const int2 y = split_limbs(s_y);
        const int lz = s_sh;
        // 1 / d = y 2^(lz - 121): the multiplier v / d in 2^-56 is mul_limbs(v 2^e, y) 2^(lz - 9 - e)
        const int rows = R - k - 1, items = rows + M - k - 1;
#pragma unroll 1
        for (int e = tid; e < items; e += NT) {
            if (e < rows) {
                double* t = T + (k + 1 + e) * ldm + k;
                const long long v = *fixed(t);
                const int up = max(58 - int_exp(v), 0);  // (|v| 2^up < 2^58, or v is out of range)
                const long long w = mul_limbs(split_limbs(v << up), y);
                const int sh = lz - 9 - up;
                bad |= sh > 0 && int_exp(w) + sh > 59;
                const long long m = shift_fixed(w, sh);
                bad |= limb_overflow(m);
                *limbs(t) = split_limbs(m);
            } else {
                const int c = k + 1 + e - rows;
                const long long v = fixed(T)[k * ldm + c] - row_dot_col(T + k * ldm, T + c, ldm, k);
                bad |= limb_overflow(v);
                limbs(T)[k * ldm + c] = split_limbs(v);
            }
        }
        team_sync<NT>();
    }
#pragma unroll 1
    for (int i = M + tid; i < R; i += NT) {  // a row of B or ghat
        double* row = T + i * ldm;
        unsigned l1 = 0u;  // in 2^33 units, rounded up
#pragma unroll 1
        for (int k = M - 1; k >= 0; --k) {
            LimbSum t, u;
            int j = k + 1;
            if (j & 1) {
                if (j < M) t.mac(limbs(row)[j], limbs(T)[j * ldm + k]);
                ++j;
            }
#pragma unroll 1
            for (; j + 1 < M; j += 2) {
                const int4 x = reinterpret_cast<const int4*>(row)[j >> 1];
                t.mac(make_int2(x.x, x.y), limbs(T)[j * ldm + k]);
                u.mac(make_int2(x.z, x.w), limbs(T)[(j + 1) * ldm + k]);
                if ((j & 14) == 14) { t.fold(); u.fold(); }
            }
            if (j < M) t.mac(limbs(row)[j], limbs(T)[j * ldm + k]);
            t.fold();
            u.fold();
            t.h += u.h;
            t.m += u.m;
            const long long v = join_limbs(limbs(row)[k]) - t.total();
            bad |= limb_overflow(v);
            limbs(row)[k] = split_limbs(v);
            l1 += (unsigned)((unsigned long long)(v < 0 ? -v : v) >> 33) + 1u;
        }
        if (M & 1) limbs(row)[M] = make_int2(0, 0);
        const int e = 33 - kTabBits + 30 - __clz(l1);  // the row's absolute sum is below 4 2^e
        if (i < n) {
            atomicMax(&s_ns_eb, max(e, kFixBits - kTabBits));
        } else {
            const int e0 = gs + kFixBits - kTabBits, eg = max(max(e + gs, e0), eg_min);
            sm.eg[i - n] = eg;
            if (eg > e0)
#pragma unroll 1
                for (int k = 0; k < M; ++k) limbs(row)[k] = split_limbs(shift_fixed(join_limbs(limbs(row)[k]), e0 - eg));
        }
    }
    if (__syncthreads_or(bad)) return false;
    const int sh = kFixBits - kTabBits - s_ns_eb;
    if (sh < 0) {
#pragma unroll 1
        for (int i = M + tid; i < n; i += NT)
#pragma unroll 1
            for (int k = 0; k < M; ++k)
                limbs(T)[i * ldm + k] = split_limbs(shift_fixed(join_limbs(limbs(T)[i * ldm + k]), sh));
    }
    return true;
}

// The same three steps in FP64.  Returns false on a column that depends on the earlier ones: its
// largest entry left is below 2^-kRankBits of its largest one before (in sm.X).  Lattices have such
// columns, as polynomials that vanish at all of a stencil's nodes: rounding leaves up to 2^-49 of
// them, and 2^-34 with nodes 2^15 radii from the origin.  Thin stencils along an axis keep 2^-8,
// slabs of 1:1000 across the axes 2^-31.
constexpr int kRankBits = 34;

template <int NT>
__device__ bool ns_eliminate(int n, int M, int q, const NullSmem& sm) {
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int ldm = sm.ldm, R = n + q;
    double* T = sm.T;
#pragma unroll 1
    for (int c = tid; c < M; c += NT) {
        double top = 0.0;
#pragma unroll 1
        for (int i = 0; i < n; ++i) top = mag_key(T[i * ldm + c]) > mag_key(top) ? T[i * ldm + c] : top;
        sm.X[c] = top;
    }
    __syncthreads();
#pragma unroll 1
    for (int k = 0; k < M; ++k) {
        if (wid == 0) {
            unsigned best = 0u;
            int p = 0x7fffffff;
#pragma unroll 1
            for (int i = k + lane; i < n; i += 32) {
                const unsigned v = mag_key(T[i * ldm + k]);
                if (v > best) { best = v; p = i; }
            }
            const unsigned top = __reduce_max_sync(0xffffffffu, best);
            p = (int)__reduce_min_sync(0xffffffffu, best == top ? (unsigned)p : 0x7fffffffu);
            // (exponents of the two magnitudes; a zero column has none left)
            const bool left = top != 0u && (int)(mag_key(sm.X[k]) >> 20) - (int)(top >> 20) < kRankBits;
            if (left) {
                if (p != k) {
#pragma unroll 1
                    for (int c = lane; c < M; c += 32) {
                        const double t = T[k * ldm + c];
                        T[k * ldm + c] = T[p * ldm + c];
                        T[p * ldm + c] = t;
                    }
                    if (lane == 0) { const int t = sm.order[k]; sm.order[k] = sm.order[p]; sm.order[p] = t; }
                    __syncwarp();
                }
                const double rcp = rcp_fixed(T[k * ldm + k]);
#pragma unroll 1
                for (int i = k + 1 + lane; i < R; i += 32) T[i * ldm + k] *= rcp;
            }
            if (lane == 0) s_ns_ok = left;
        }
        __syncthreads();
        if (!s_ns_ok) return false;
        const int wc = M - 1, total = (R - k - 1) * wc;
        if (tid < total) {
            int r = tid / wc, c = tid - (tid / wc) * wc;
            const int dr = NT / wc, dc = NT - dr * wc;
            const double* Tk = T + k * ldm;
#pragma unroll 1
            for (int e = tid; e < total; e += NT) {
                const int cc = c + (c >= k);
                double* Ti = T + (k + 1 + r) * ldm;
                Ti[cc] = fma(-Ti[k], Tk[cc], Ti[cc]);
                r += dr;
                c += dc;
                if (c >= wc) { c -= wc; ++r; }
            }
        }
        __syncthreads();
    }
    return true;
}

template <int NT>
__device__ __forceinline__ void ns_scales(int n, int M, int q, int eg_min, const NullSmem& sm) {
    const int lane = threadIdx.x & 31;
#pragma unroll 1
    for (int r = M + (int)(threadIdx.x >> 5); r < n + q; r += NT / 32) {
        int e = -200;
        float l1 = 0.0f;
#pragma unroll 1
        for (int c = lane; c < M; c += 32) {
            const double v = sm.T[r * sm.ldm + c];
            e = max(e, scale_exp(v));
            l1 += approx_f32(abs_bits(v));
        }
        e = __reduce_max_sync(0xffffffffu, e);
        for (int o = 16; o > 0; o >>= 1) l1 += __shfl_xor_sync(0xffffffffu, l1, o);
        if (lane == 0) {
            const int el = (__float_as_int(l1) >> 23) - 126 - 2;  // l1 < 2^(el + 2)
            if (r < n) {
                atomicMax(&s_ns_eb, max(e, el));
            } else {
                sm.eg[r - n] = max(max(e, el), eg_min);
            }
        }
    }
}

template <int NT>
__device__ __forceinline__ void ns_rows_to_limbs(int n, int M, int q, const NullSmem& sm) {
    const int ldm = sm.ldm, Mp = (M + 1) & ~1;
    const int total = (n - M + q) * Mp;
#pragma unroll 1
    for (int e = threadIdx.x; e < total; e += NT) {
        const int r = e / Mp, c = e - r * Mp;
        double* t = sm.T + (M + r) * ldm + c;
        const int ex = r < n - M ? s_ns_eb : sm.eg[r - (n - M)];
        *limbs(t) = c < M ? to_limbs(*t, ex) : make_int2(0, 0);
    }
}

// ------------------------------------------------------------------ the two products
// C = A21 - B A11 / 2 for the rows i0.. of [B; ghat of columns c0..] (the row of a column is in X),
// in units 2^(eA + scale of the row - 61) as A21 and f1 come: 2 x 2 outputs per thread, two terms of
// the sum per pair of 16-byte loads.
template <int NT>
__device__ void ns_product_c(int n, int M, int i0, int c0, int qk, int eA, const NullSmem& sm) {
    const int s = n - M, ldm = sm.ldm, rows = s + qk;
    const int nr = (rows - i0 + 1) >> 1, nc = (M + 1) >> 1;
    long long top = 0;  // (of the rows of C) the bits of all |C|
#pragma unroll 1
    for (int e = threadIdx.x; e < nr * nc; e += NT) {
        const int tr = small_div(e, nc), j = 2 * (e - tr * nc);
        const int i = i0 + 2 * tr;
        const bool two_i = i + 1 < rows, two_j = j + 1 < M;
        // (the rows of B and of the first columns are consecutive; c0 > 0: later columns, alone)
        const int4* B = reinterpret_cast<const int4*>(sm.T + (M + i + c0) * ldm);
        const int4* A = reinterpret_cast<const int4*>(sm.T + j);
        const int lc = ldm >> 1, db = two_i ? lc : 0;
        LimbSum a0, a1, b0, b1;
#pragma unroll 1
        for (int k = 0; 2 * k < M; ++k) {
            const int4 x = B[k], y = B[k + db], u = A[0], v = A[lc];
            A += 2 * lc;
            const int2 x0 = make_int2(x.x, x.y), x1 = make_int2(x.z, x.w);
            const int2 y0 = make_int2(y.x, y.y), y1 = make_int2(y.z, y.w);
            const int2 u0 = make_int2(u.x, u.y), u1 = make_int2(u.z, u.w);
            const int2 v0 = make_int2(v.x, v.y), v1 = make_int2(v.z, v.w);
            a0.mac(x0, u0); a1.mac(x0, u1); b0.mac(y0, u0); b1.mac(y0, u1);
            a0.mac(x1, v0); a1.mac(x1, v1); b0.mac(y1, v0); b1.mac(y1, v1);
            if ((k & 7) == 7) { a0.fold(); a1.fold(); b0.fold(); b1.fold(); }
        }
        auto put = [&](int r, long long t0, long long t1) {
            long long* d = fixed((r < s ? sm.C + r * ldm : sm.X + (r - s) * sm.ldx) + j);
            t0 = d[0] - t0;
            t1 = two_j ? d[1] - t1 : 0;
            d[0] = t0;
            if (two_j) d[1] = t1;
            if (r < s) top |= (t0 ^ (t0 >> 63)) | (t1 ^ (t1 >> 63));
        };
        put(i, a0.total(), a1.total());
        if (two_i) put(i + 1, b0.total(), b1.total());
    }
    if (i0 < s) {  // the scale of C (one for all its rows)
        const int e = __reduce_max_sync(0xffffffffu, int_exp(top)) + eA + s_ns_eb + kSumUnit - 1;
        if ((threadIdx.x & 31) == 0) atomicMax(&s_ns_ec, e);
    }
}

template <int NT>
__device__ __forceinline__ void ns_c_to_limbs(int s, int M, int eA, const NullSmem& sm) {
    const int Mp = (M + 1) & ~1, sh = eA + s_ns_eb + kSumUnit - 1 - s_ns_ec + kFixBits;
#pragma unroll 1
    for (int t = threadIdx.x; t < s * Mp; t += NT) {
        const int r = small_div(t, Mp), c = t - r * Mp;
        double* d = sm.C + r * sm.ldm + c;
        *limbs(d) = c < M ? split_limbs(shift_fixed(*fixed(d), sh)) : make_int2(0, 0);
    }
}

// The columns' rows: f1 - A11 ghat / 2 to limbs at a scale 2^ef that covers the row, with
// ef + eB = eg + eC (both products of a column's sums in one unit), for which ghat may move to a
// larger scale; f2 to the unit of those sums.  A warp per column.
template <int NT>
__device__ __forceinline__ void ns_columns_to_limbs(int n, int M, int c0, int qk, int eA, int eF, const NullSmem& sm) {
    const int lane = threadIdx.x & 31, s = n - M, Mp = (M + 1) & ~1;
    const int eB = s_ns_eb, eC = s_ns_ec;
#pragma unroll 1
    for (int c = threadIdx.x >> 5; c < qk; c += NT / 32) {
        double* X = sm.X + c * sm.ldx;
        const int eg = sm.eg[c0 + c];
        const int u1 = eA + eg + kSumUnit - 1, u2 = eF - kPowerBits;
        int e1 = 0;
#pragma unroll 1
        for (int t = lane; t < M; t += 32) e1 = max(e1, int_exp(fixed(X)[t]));
        const int e = __reduce_max_sync(0xffffffffu, e1) + u1;
        const int ef = max(max(e, eF - eB - 2), eg + eC - eB);  // (f2 fits the sums' unit)
        const int up = ef + eB - eC - eg;  // >= 0
        double* G = sm.T + (n + c0 + c) * sm.ldm;
#pragma unroll 1
        for (int t = lane; t < Mp; t += 32) {
            *limbs(X + t) = t < M ? split_limbs(shift_fixed(fixed(X)[t], u1 - ef + kFixBits)) : make_int2(0, 0);
            if (up > 0) {
                const int k = min(up, 62);
                *limbs(G + t) = split_limbs((join_limbs(*limbs(G + t)) + (1ll << (k - 1))) >> k);
            }
        }
#pragma unroll 1
        for (int t = lane; t < s; t += 32) {
            long long* f = fixed(X) + sm.x2 + t;
            *f = shift_fixed(*f, u2 - (ef + eB + kSumUnit));
        }
        __syncwarp();
        if (lane == 0) sm.eg[c0 + c] = eg + up;
    }
}

// C B^T + B C^T (lower triangle; rows < s) into S, and taken off the columns' f2: the tiles I >= J
// of 2 x 2 entries, then the columns' tiles, in integers of the sums' units (ns_finish adds A22).
template <int NT>
__device__ void ns_product_s(int n, int M, bool triangle, int c0, int qk, const NullSmem& sm) {
    const int s = n - M, ldm = sm.ldm, nt = (s + 1) >> 1;
    const int half = (nt + 1) >> 1;
    const int tri_tiles = triangle ? half * (nt + 1) : 0;
    const int all = tri_tiles + ((qk + 1) >> 1) * nt;
#pragma unroll 1
    for (int e = threadIdx.x; e < all; e += NT) {
        const bool column = e >= tri_tiles;
        int I, J;
        if (!column) {
            const int p = small_div(e, nt + 1), o = e - p * (nt + 1);
            const bool first = o <= p;
            I = first ? p : nt - 1 - p;
            J = first ? o : o - p - 1;
            if (!first && I == p) continue;  // an odd middle row of tiles pairs with itself
        } else {
            I = small_div(e - tri_tiles, nt);
            J = e - tri_tiles - I * nt;
        }
        const int i = 2 * I, j = 2 * J;
        const bool two_i = i + 1 < (column ? qk : s), two_j = j + 1 < s;
        // the rows' first 16-byte words and the steps to their second rows
        const int4* Bi = reinterpret_cast<const int4*>(sm.T + ((column ? n + c0 : M) + i) * ldm);
        const int4* Ci = reinterpret_cast<const int4*>(column ? sm.X + i * sm.ldx : sm.C + i * ldm);
        const int4* Bj = reinterpret_cast<const int4*>(sm.T + (M + j) * ldm);
        const int4* Cj = reinterpret_cast<const int4*>(sm.C + j * ldm);
        const int db = two_i ? ldm >> 1 : 0, dc = two_i ? (column ? sm.ldx : ldm) >> 1 : 0;
        const int dj = two_j ? ldm >> 1 : 0;
        LimbSum aa, ab, ba, bb;
#pragma unroll 1
        for (int k = 0; 2 * k < M; ++k) {
            auto half_step = [&](int4 bi, int4 bk, int4 cj, int4 ck) {
                const int2 x0 = make_int2(bi.x, bi.y), x1 = make_int2(bi.z, bi.w);
                const int2 y0 = make_int2(bk.x, bk.y), y1 = make_int2(bk.z, bk.w);
                const int2 u0 = make_int2(cj.x, cj.y), u1 = make_int2(cj.z, cj.w);
                const int2 v0 = make_int2(ck.x, ck.y), v1 = make_int2(ck.z, ck.w);
                aa.mac(x0, u0); ab.mac(x0, v0); ba.mac(y0, u0); bb.mac(y0, v0);
                aa.mac(x1, u1); ab.mac(x1, v1); ba.mac(y1, u1); bb.mac(y1, v1);
            };
            half_step(Bi[k], Bi[k + db], Cj[k], Cj[k + dj]);
            half_step(Ci[k], Ci[k + dc], Bj[k], Bj[k + dj]);
            if ((k & 3) == 3) { aa.fold(); ab.fold(); ba.fold(); bb.fold(); }
        }
        // entry (i, j) and the steps to (i + 1, j) and (i, j + 1)
        long long* d = column ? fixed(sm.X) + i * sm.ldx + sm.x2 + j : fixed(sm.S) + col_start(j, s) + i;
        const int di = column ? sm.ldx : 1, dd = column ? 1 : s - j - 1;
        const long long keep = column ? -1 : 0;  // S starts here
        d[0] = (d[0] & keep) - aa.total();
        if (two_j && (column || j < i)) d[dd] = (d[dd] & keep) - ab.total();
        if (two_i) {
            d[di] = (d[di] & keep) - ba.total();
            if (two_j) d[di + dd] = (d[di + dd] & keep) - bb.total();
        }
    }
}

// ------------------------------------------------------------------ the definite system
// S = L D L^T without pivoting, with the columns' forward substitution (rows of X): w_ij = L_ij d_j,
// the unscaled entries, replace S column by column.  Every entry gets fma(-w_ij, L_pj, .) for
// j = 0, 1, ... (L_pj = w_pj / d_j), in two forms with the same operations: a single warp goes
// left-looking, a row (of S or of a column) per lane and one dot product per column, which takes
// three instructions per FMA; larger teams, which hold large systems, go right-looking, all
// threads sharing each update.  Returns false on a pivot below 2^-kSpanBits of the largest one (S is
// definite, so that is rounding: nodes too near each other).
// s_ns_ratio: floor(log2) of the largest over that of the smallest pivot, a lower bound of S's
// condition number (read after a barrier).
__shared__ int s_ns_ratio;
constexpr int kSpanBits = 49;

// (d_max: the largest key so far, d among them)
__device__ __forceinline__ bool pivot_lost(double d, unsigned d_max) {
    return abs_bits(d) == 0ull || (int)(d_max >> 20) - (int)(mag_key(d) >> 20) > kSpanBits;
}

template <int NT>
__device__ bool ns_factor(int s, int qk, const NullSmem& sm) {
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    double* S = sm.S;
    double* Y = sm.X + sm.x2;
    const int ldx = sm.ldx;
    unsigned d_max = 0u, d_min = ~0u;  // (warp 0) magnitude keys of the pivots
    if constexpr (NT == 32) {
#pragma unroll 1
        for (int p = 0; p < s; ++p) {
#pragma unroll 1
            for (int j = lane; j < p; j += 32) sm.wb[j] = S[col_start(j, s) + p] * sm.rd[j];
            __syncwarp();
            double d = 0.0;
#pragma unroll 1
            for (int r = lane; r < s - p + qk; r += 32) {  // rows p .. s-1, then the columns
                const bool col = r >= s - p;
                double* t = col ? Y + (r - (s - p)) * ldx : S + p + r;
                const int t1 = col ? 1 : s - 1;  // w_ij at t[j t1 - (j (j - 1) / 2 for rows of S)]
                int off = 0, step = t1;
                double v = t[col ? p : col_start(p, s)];
#pragma unroll 1
                for (int j = 0; j < p; ++j) {
                    v = fma(-t[off], sm.wb[j], v);
                    off += step;
                    step -= col ? 0 : 1;
                }
                t[col ? p : col_start(p, s)] = v;
                if (r == lane) d = v;
            }
            d = __shfl_sync(0xffffffffu, d, 0);
            d_max = max(d_max, mag_key(d));
            if (pivot_lost(d, d_max)) return false;
            const double rcp = rcp_fixed(d);
            d_min = min(d_min, mag_key(d));
            if (lane == 0) sm.rd[p] = rcp;
            __syncwarp();
        }
    } else {
#pragma unroll 1
        for (int p = 0; p < s; ++p) {
            if (wid == 0) {
                const double d = S[col_start(p, s) + p];
                const double rcp = rcp_fixed(d);
                d_max = max(d_max, mag_key(d));
                d_min = min(d_min, mag_key(d));
                if (lane == 0) { sm.rd[p] = rcp; s_ns_ok = !pivot_lost(d, d_max); }
#pragma unroll 1
                for (int i = p + 1 + lane; i < s; i += 32) sm.wb[i] = S[col_start(p, s) + i] * rcp;
            }
            __syncthreads();
            if (!s_ns_ok) return false;
            const int rows = s - p - 1;
            const int L2 = rows + 1 + 2 * qk;
            const int total = ((rows + 1) >> 1) * L2;
            const double* Sp = S + col_start(p, s);
            // row i has its triangle entries, then its entry of every column; rows r and
            // rows-1-r are paired into one of constant length
            if (tid < total) {
                int pr = small_div(tid, L2), off = tid - pr * L2;
                const int di = small_div(NT, L2), dj = NT - di * L2;
#pragma unroll 1
                for (int e = tid; e < total; e += NT) {
                    const int len0 = pr + 1 + qk;
                    const bool first = off < len0;
                    const int r = first ? pr : rows - 1 - pr;
                    const int t = first ? off : off - len0;
                    if (first || r != pr) {
                        const int i = p + 1 + r;
                        const bool trin = t <= r;
                        const int jj = p + 1 + t, c = t - (r + 1);
                        double* dst = trin ? S + col_start(jj, s) + i : Y + c * ldx + i;
                        const double* src = trin ? Sp + i : Y + c * ldx + p;
                        *dst = fma(-*src, sm.wb[trin ? jj : i], *dst);
                    }
                    pr += di;
                    off += dj;
                    if (off >= L2) { off -= L2; ++pr; }
                }
            }
            __syncthreads();
        }
    }
    if (tid == 0) s_ns_ratio = (int)(d_max >> 20) - (int)(d_min >> 20);
    return true;
}

// Forward substitution of later columns with the stored factors: the same operations on every
// entry, in the same order, as in ns_factor.
template <int NT>
__device__ void ns_forward(int s, int qk, const NullSmem& sm) {
    double* Y = sm.X + sm.x2;
#pragma unroll 1
    for (int p = 0; p < s; ++p) {
        const int rows = s - p - 1;
        const double rcp = sm.rd[p];
        const double* Sp = sm.S + col_start(p, s);
#pragma unroll 1
        for (int e = threadIdx.x; e < rows * qk; e += NT) {
            const int c = small_div(e, rows), i = p + 1 + e - c * rows;
            Y[c * sm.ldx + i] = fma(-Y[c * sm.ldx + p], Sp[i] * rcp, Y[c * sm.ldx + i]);
        }
        team_sync<NT>();
    }
}

// Back substitution of the columns, v_j = (y_j - sum over i > j of w_ij v_i) / d_j, then v to limbs
// (in the words of f1) and its scale.  With more columns than warps a team shares each step,
// (column, row) pairs flattened over its lanes; else a warp per column.  (The same operations.)
template <int NT>
__device__ void ns_back(int s, int qk, const NullSmem& sm) {
    constexpr int NW = NT / 32;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    double* Y = sm.X + sm.x2;
    const bool shared_steps = qk > NW;
    const int c0 = shared_steps ? 0 : wid, nc = shared_steps ? qk : min(qk, wid + 1);
    const int l0 = shared_steps ? (int)threadIdx.x : lane, L = shared_steps ? NT : 32;
#pragma unroll 1
    for (int i = s - 1; i >= 0; --i) {
        const double rd = sm.rd[i];
        const int total = i * (nc - c0);
        const int k = small_div(l0, max(i, 1)), dc = small_div(L, max(i, 1)), dj = L - dc * i;
        int c = c0 + k, j = l0 - k * i;
#pragma unroll 1
        for (int e = l0; e < total; e += L) {
            double* y = Y + c * sm.ldx;
            y[j] = fma(-sm.S[col_start(j, s) + i], y[i] * rd, y[j]);
            j += dj;
            c += dc;
            if (j >= i) { j -= i; ++c; }
        }
        if (shared_steps) team_sync<NT>();
        else __syncwarp();
    }
#pragma unroll 1
    for (int c = wid; c < qk; c += NW) {
        double* y = Y + c * sm.ldx;
        int e = -200;
#pragma unroll 1
        for (int i = lane; i < s; i += 32) {
            const double v = y[i] * sm.rd[i];
            y[i] = v;
            e = max(e, scale_exp(v));
        }
        e = __reduce_max_sync(0xffffffffu, e) + 4;  // (16 times its largest entry: a sum of s <= 128
                                                     //  products with B stays inside 64 bits)
        int2* V = limbs(sm.X + c * sm.ldx);
#pragma unroll 1
        for (int i = lane; i < s; i += 32) V[i] = to_limbs(y[i], e);
        if (lane == 0) sm.ev[c] = (short)e;
    }
}

// w_basic = ghat - B^T v, in place of ghat: two entries of a column per thread.
template <int NT>
__device__ void ns_basic_weights(int n, int M, int c0, int qk, const NullSmem& sm) {
    const int s = n - M, ldm = sm.ldm, nc = (M + 1) >> 1, eB = s_ns_eb;
#pragma unroll 1
    for (int e = threadIdx.x; e < qk * nc; e += NT) {
        const int c = small_div(e, nc), l = 2 * (e - c * nc);
        const int2* V = limbs(sm.X + c * sm.ldx);
        const int4* B = reinterpret_cast<const int4*>(sm.T + M * ldm + l);
        LimbSum a, b;
#pragma unroll 1
        for (int k = 0; k < s; ++k) {
            const int2 v = V[k];
            const int4 x = B[k * (ldm >> 1)];
            a.mac(make_int2(x.x, x.y), v);
            b.mac(make_int2(x.z, x.w), v);
            if ((k & 15) == 15) { a.fold(); b.fold(); }
        }
        double* G = sm.T + (n + c0 + c) * ldm + l;
        const int eg = sm.eg[c0 + c], unit = eB + sm.ev[c] + kSumUnit;
        G[0] = from_fixed(join_limbs(limbs(G)[0]), eg - kFixBits) - from_fixed(a.total(), unit);
        if (l + 1 < M)
            G[1] = from_fixed(join_limbs(limbs(G)[1]), eg - kFixBits) - from_fixed(b.total(), unit);
    }
}

// The correction's share of the basic weights: w_basic -= B^T dv, with the limbs of dv in place.
template <int NT>
__device__ void ns_basic_correction(int n, int M, int c0, int qk, const NullSmem& sm) {
    const int s = n - M, ldm = sm.ldm, eB = s_ns_eb;
#pragma unroll 1
    for (int e = threadIdx.x; e < qk * M; e += NT) {
        const int c = small_div(e, M), l = e - c * M;
        const int2* V = limbs(sm.X + c * sm.ldx);
        LimbSum a;
#pragma unroll 1
        for (int k = 0; k < s; ++k) {
            a.mac(limbs(sm.T + (M + k) * ldm)[l], V[k]);
            if ((k & 15) == 15) a.fold();
        }
        sm.T[(n + c0 + c) * ldm + l] -= from_fixed(a.total(), eB + sm.ev[c] + kSumUnit);
    }
}

// Weight of stencil position r in column c0 + c of the current chunk.
__device__ __forceinline__ double ns_weight(int n, int M, int r, int c0, int c, const NullSmem& sm) {
    const int p = sm.pos[r];
    return p < M ? sm.T[(n + c0 + c) * sm.ldm + p] : sm.X[c * sm.ldx + sm.x2 + p - M];
}

}  // namespace rbffd

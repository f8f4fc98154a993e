// spectrum.cu -- full-system spectrum of a configuration (Sec. VI): all 2N
// eigenvalues of the whole lattice's one-body Hamiltonian, where the paper
// diagonalises saved configurations with ScaLAPACK.  Everything runs in this
// library's kernels, off the sweep's hot path (step 2 in FP64 for FP64
// contexts and in double-float on the FP32 pipe for PTCA_MIXED contexts):
//   1. the dense matrix is built as its packed lower triangle (row-major:
//      element (i, j <= i) at i(i+1)/2 + j) in global memory;
//   2. a Householder reduction to real tridiagonal form spread over the whole
//      GPU: per reflector, one pass applies the previous reflector's deferred
//      rank-2 update to the trailing block and accumulates the Hermitian
//      matrix-vector product with the current reflector (row and column partial
//      sums per strip of 64 columns, in a fixed order), and one thread-block
//      cluster adds the partials up and forms w, the explicit update of the
//      next pivot column and the next reflector -- the algorithm of the
//      cluster kernels (cluster_solve.cuh), with the matrix too large for one
//      SM;
//   3. one thread per eigenvalue: FP32 bisection on the FP32-rounded
//      tridiagonal, then the cluster solver's double-float Sturm counts and
//      safeguarded Newton on the exact (FP64) tridiagonal.
#include <algorithm>
#include <cfloat>
#include <cmath>
#include <string>
#include <vector>

#include "../../include/ptca.h"
#include "context.h"
#include "kernels.cuh"
#include "launch.h"

namespace ptca {

__host__ __device__ __forceinline__ int64_t tri64(int64_t r) { return r * (r + 1) / 2; }

constexpr int FS_TB = 64;            // columns of a strip of the reduction pass
constexpr int FS_PASS_THREADS = 256, FS_PASS_WARPS = FS_PASS_THREADS / 32;
constexpr int FS_PASS_CTAS = 2;      // resident per SM
constexpr int FS_GROUP = 4;          // rows that a warp loads and reduces at a time
constexpr int FS_MIN_ROWS = 16, FS_MAX_ROWS = 128;  // rows of a chunk
constexpr int FS_RED_THREADS = 256;  // 8 warps; each CTA sums the partials of FS_RED_ROWS rows
constexpr int FS_RED_ROWS = 32;
constexpr int FS_CL = 8;             // CTAs of the step cluster (the portable size)
constexpr int FS_STEP_THREADS = 1024, FS_STEP_PARTS = 4, FS_STEP_ROWS = FS_STEP_THREADS / FS_STEP_PARTS;
constexpr int FS_SCALAR_THREADS = 1024;
constexpr int FS_EIG_THREADS = 128;

// One thread per lattice site: its on-site 2x2 block and its bonds to the
// +x, +y, +z neighbours, hopping added atomically so that an axis of extent 2
// on a torus gets both of its bonds (-2t).  H: packed lower triangle of order
// 2N, zeroed by the caller.
__global__ void k_full_hamiltonian(Model m, const double* __restrict__ S, int N, double2* __restrict__ H) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const int x = i % m.Lx, y = (i / m.Lx) % m.Ly, z = i / (m.Lx * m.Ly);
    const double sx = S[3 * i], sy = S[3 * i + 1], sz = S[3 * i + 2];
    const double dg = m.e0 + m.lam * sx, J = m.JH;
    const int64_t a = 2 * (int64_t)i, b = a + 1;
    H[tri64(a) + a] = make_double2(dg - J * sz, 0.0);
    H[tri64(b) + b] = make_double2(dg + J * sz, 0.0);
    H[tri64(b) + a] = make_double2(-J * sx, -J * sy);  // element (b, a) = -J (S_x + i S_y)
    const int L[3] = {m.Lx, m.Ly, m.Lz};
    const int c[3] = {x, y, z};
    for (int d = 0; d < 3; ++d) {
        if (L[d] == 1) continue;
        int cc[3] = {c[0], c[1], c[2]};
        cc[d] += 1;
        if (cc[d] == L[d]) {
            if (!m.lattice_periodic) continue;
            cc[d] = 0;
        }
        const int j = (cc[2] * m.Ly + cc[1]) * m.Lx + cc[0];
        for (int sg = 0; sg < 2; ++sg) {
            const int64_t p = 2 * (int64_t)i + sg, q = 2 * (int64_t)j + sg;
            const int64_t hi = p > q ? p : q, lo = p > q ? q : p;
            atomicAdd(&H[tri64(hi) + lo].x, -m.t);
        }
    }
}

// The reduction runs in the real arithmetic R: double, or dfl (double-float:
// about 48 significant bits on the FP32 pipe, which runs 64 times the FP64
// rate).  A complex entry takes 16 bytes and a real one 8 in either, so the
// buffers are the same.
__device__ __forceinline__ double fs_d(double x) { return x; }
__device__ __forceinline__ double fs_d(dfl x) { return (double)x; }
template <typename R> __device__ __forceinline__ R fs_r(float x);
template <> __device__ __forceinline__ double fs_r<double>(float x) { return (double)x; }
template <> __device__ __forceinline__ dfl fs_r<dfl>(float x) { return dfl(x, 0.f); }
__device__ __forceinline__ double shfl_xor_r(double v, int o) { return __shfl_xor_sync(FULL_MASK, v, o); }
__device__ __forceinline__ dfl shfl_xor_r(dfl v, int o) { return shfl_xor_dfl(v, o); }

// Pairs of floats for the two-wide FP32 instructions.
using fs_f2 = unsigned long long;
__device__ __forceinline__ fs_f2 f2_pack(float a, float b) {
    fs_f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 f2_split(fs_f2 v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ fs_f2 f2_dup(float a) { return f2_pack(a, a); }
__device__ __forceinline__ fs_f2 f2_add(fs_f2 a, fs_f2 b) {
    fs_f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ fs_f2 f2_sub(fs_f2 a, fs_f2 b) {
    fs_f2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ fs_f2 f2_mul(fs_f2 a, fs_f2 b) {
    fs_f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ fs_f2 f2_fma(fs_f2 a, fs_f2 b, fs_f2 c) {
    fs_f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// A complex double-float in memory: the leading parts of (re, im), then the
// trailing ones, so that the pass works on pairs; and its accumulators.
struct __align__(16) DfPair { fs_f2 hi, lo; };
// c += p + (the product's error and cross terms), not renormalised: TwoSum on the
// leading parts, everything below into the trailing ones.
__device__ __forceinline__ void df_add(DfPair& c, fs_f2 hi, fs_f2 lo) {
    const fs_f2 s = f2_add(c.hi, hi), t = f2_sub(s, c.hi);
    const fs_f2 e = f2_add(f2_sub(c.hi, f2_sub(s, t)), f2_sub(hi, t));
    c.hi = s;
    c.lo = f2_add(c.lo, f2_add(e, lo));
}
// a b elementwise: the rounded product, and its error and cross terms in lo.
__device__ __forceinline__ fs_f2 df_mul(const DfPair& a, const DfPair& b, fs_f2& lo) {
    const fs_f2 p = f2_mul(a.hi, b.hi);
    const float2 x = f2_split(a.hi), y = f2_split(b.hi), q = f2_split(p);
    lo = f2_fma(a.lo, b.hi, f2_fma(a.hi, b.lo, f2_pack(__fmaf_rn(x.x, y.x, -q.x), __fmaf_rn(x.y, y.y, -q.y))));
    return p;
}
__device__ __forceinline__ void df_fma(DfPair& c, const DfPair& a, const DfPair& b) {
    fs_f2 lo;
    const fs_f2 p = df_mul(a, b, lo);
    df_add(c, p, lo);
}
__device__ __forceinline__ DfPair df_norm(const DfPair& c) {
    DfPair r;
    r.hi = f2_add(c.hi, c.lo);
    r.lo = f2_sub(c.lo, f2_sub(r.hi, c.hi));
    return r;
}
__device__ __forceinline__ DfPair df_dup(dfl v) { return {f2_dup(v.hi), f2_dup(v.lo)}; }
__device__ __forceinline__ DfPair df_pack(dfl x, dfl y) { return {f2_pack(x.hi, y.hi), f2_pack(x.lo, y.lo)}; }

// The memory form of a complex entry and its conversions.
template <typename R> struct FsMem { using type = cplx_t<R>; };
template <> struct FsMem<dfl> { using type = DfPair; };
template <typename R> using fs_mem = typename FsMem<R>::type;
__device__ __forceinline__ double2 fs_get(const double2& v) { return v; }
__device__ __forceinline__ dfl2 fs_get(const DfPair& v) {
    const float2 h = f2_split(v.hi), l = f2_split(v.lo);
    return mk(dfl(h.x, l.x), dfl(h.y, l.y));
}
// s += v on memory forms, without the renormalisation (fs_sum does it once).
__device__ __forceinline__ void fs_acc(double2& s, const double2& v) { s = cadd(s, v); }
__device__ __forceinline__ void fs_acc(DfPair& s, const DfPair& v) { df_add(s, v.hi, v.lo); }
__device__ __forceinline__ double2 fs_sum(const double2& s) { return s; }
__device__ __forceinline__ dfl2 fs_sum(const DfPair& s) { return fs_get(df_norm(s)); }
__device__ __forceinline__ void fs_acc(double& s, double v) { s += v; }
__device__ __forceinline__ void fs_acc(dfl& s, dfl v) {
    const dfl t = two_sum(s.hi, v.hi);
    s = dfl(t.hi, __fadd_rn(__fadd_rn(t.lo, v.lo), s.lo));
}
__device__ __forceinline__ double fs_sum(double s) { return s; }
__device__ __forceinline__ dfl fs_sum(dfl s) { return fast_two_sum(s.hi, s.lo); }
__device__ __forceinline__ double2 fs_xor(const double2& v, int o) { return cshfl_xor(v, o); }
__device__ __forceinline__ DfPair fs_xor(const DfPair& v, int o) {
    return {__shfl_xor_sync(FULL_MASK, v.hi, o), __shfl_xor_sync(FULL_MASK, v.lo, o)};
}
__device__ __forceinline__ void fs_put(double2& m, double2 v) { m = v; }
__device__ __forceinline__ void fs_put(DfPair& m, dfl2 v) { m = df_pack(v.x, v.y); }

// The pass's arithmetic on one element x of row i and a column c: the update
// x - u_i w_c^* - w_i u_c^*, the row sum of x v_c and the column sum of x^* v_i.
// `Row` and `Col` hold the operands in the form that the products take, `Sum` is
// an accumulator; save() leaves a row sum's parts in two places of shared memory
// and total() reads them.
template <typename R> struct FsOps;
template <> struct FsOps<double> {
    struct Row { double2 u, w, v; };
    struct Col { double2 u, w, v; };
    using Sum = double2;
    static __device__ __forceinline__ Sum zero() { return make_double2(0.0, 0.0); }
    static __device__ __forceinline__ Row row(const double2* m) { return {m[0], m[1], m[2]}; }
    static __device__ __forceinline__ Col col(double2 u, double2 w, double2 v) { return {u, w, v}; }
    static __device__ __forceinline__ double2 update(double2 x, const Row& r, const Col& c) {
        return cfms_conj_b(r.w, c.u, cfms_conj_b(r.u, c.w, x));
    }
    static __device__ __forceinline__ void real(double2& x) { x.y = 0.0; }
    static __device__ __forceinline__ void row_add(Sum& s, double2 x, const Col& c, bool) { s = cfma(x, c.v, s); }
    static __device__ __forceinline__ void col_add(Sum& s, double2 x, const Row& r) { s = cfma_conj_a(x, r.v, s); }
    static __device__ __forceinline__ void save_row(double2* m, const Sum& s) { *m = s; }
    static __device__ __forceinline__ double2 row_total(const double2* m, int n, int stride) {
        double2 s = m[0];
        for (int j = 1; j < n; ++j) s = cadd(s, m[j * stride]);
        return s;
    }
    static __device__ __forceinline__ double2 col_total(const Sum& s) { return s; }
};
template <> struct FsOps<dfl> {
    // Scalars of the row, both halves alike; the column's u and w as (-re, im) and
    // (-im, -re), so that the update is four products into the element; v's parts
    // alike.  The sums keep the products with v.x and v.y apart and combine them
    // at the end: nothing is swapped or negated per element.  51 + 16 + 24
    // two-wide operations an element (216 scalar ones before).
    struct Row { DfPair ux, uy, wx, wy, vx, vy; };
    struct Col { DfPair u1, u2, w1, w2, vx, vy; };
    struct Sum { DfPair x, y; };
    static __device__ __forceinline__ Sum zero() { return {{0, 0}, {0, 0}}; }
    static __device__ __forceinline__ Row row(const DfPair* m) {
        const dfl2 u = fs_get(m[0]), w = fs_get(m[1]), v = fs_get(m[2]);
        return {df_dup(u.x), df_dup(u.y), df_dup(w.x), df_dup(w.y), df_dup(v.x), df_dup(v.y)};
    }
    static __device__ __forceinline__ Col col(dfl2 u, dfl2 w, dfl2 v) {
        return {df_pack(-u.x, u.y), df_pack(-u.y, -u.x), df_pack(-w.x, w.y), df_pack(-w.y, -w.x), df_dup(v.x), df_dup(v.y)};
    }
    static __device__ __forceinline__ DfPair update(DfPair x, const Row& r, const Col& c) {
        df_fma(x, r.ux, c.w1);
        df_fma(x, r.uy, c.w2);
        df_fma(x, r.wx, c.u1);
        df_fma(x, r.wy, c.u2);
        return df_norm(x);
    }
    static __device__ __forceinline__ void real(DfPair& x) {
        x.hi &= 0xffffffffull;
        x.lo &= 0xffffffffull;
    }
    static __device__ __forceinline__ void row_add(Sum& s, const DfPair& x, const Col& c, bool first) {
        if (first) {
            s.x.hi = df_mul(x, c.vx, s.x.lo);
            s.y.hi = df_mul(x, c.vy, s.y.lo);
        } else {
            df_fma(s.x, x, c.vx);
            df_fma(s.y, x, c.vy);
        }
    }
    static __device__ __forceinline__ void col_add(Sum& s, const DfPair& x, const Row& r) {
        df_fma(s.x, x, r.vx);
        df_fma(s.y, x, r.vy);
    }
    static __device__ __forceinline__ void save_row(DfPair* m, const Sum& s) {
        m[0] = s.x;
        m[32] = s.y;
    }
    static __device__ __forceinline__ dfl2 row_total(const DfPair* m, int n, int stride) {
        Sum s{m[0], m[32]};
        for (int j = 1; j < n; ++j) {
            const DfPair a = m[j * stride], b = m[j * stride + 32];
            df_add(s.x, a.hi, a.lo);
            df_add(s.y, b.hi, b.lo);
        }
        const dfl2 x = fs_get(df_norm(s.x)), y = fs_get(df_norm(s.y));
        return mk(x.x - y.y, x.y + y.x);
    }
    static __device__ __forceinline__ dfl2 col_total(const Sum& s) {
        const dfl2 x = fs_get(df_norm(s.x)), y = fs_get(df_norm(s.y));
        return mk(x.x + y.y, y.x - x.y);
    }
};

// The built FP64 matrix rewritten in place as double-float pairs.
__global__ void k_fs_to_dfl(double2* A, int64_t count) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x) {
        const double2 x = A[i];
        fs_put(reinterpret_cast<DfPair*>(A)[i], mk(dfl(x.x), dfl(x.y)));
    }
}

// Buffers of the reduction.  Reflector k acts on rows/columns k+1 .. n-1;
// its first entry is stored at index k+1 like the others.
template <typename R>
struct FsArgs {
    using C = fs_mem<R>;
    int n;
    C* A;
    const C* U;   // v_{k-1} (zero at k = 0)
    const C* V;   // v_k
    C* Vn;        // v_{k+1}, written by the scalar phase of step k
    const C* W;   // w_{k-1} (zero at k = 0)
    C* Wn;        // w_k, written by the scalar phase of step k
    C* pr;        // [strips][n]  row partial sums of A v_k, by strip
    C* pc;        // [chunks][n]  column partial sums, by chunk of the column's strip
    C* p;         // [n]    tau A v_k
    R* tau;       // [2]    tau_k in tau[k & 1]
    double* d;    // [n]
    double* e2;   // [n]
};

// Chunks of a strip (64 columns) of `rows` rows, q rows each.
__host__ __device__ __forceinline__ int fs_chunks(int rows, int q) { return (rows + q - 1) / q; }

__device__ __forceinline__ void fs_copy16(void* smem, const void* gmem) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(gmem) : "memory");
}

// Step k's pass over the trailing block (rows and columns j0 = k+1 .. n-1): A <-
// A - u w^H - w u^H with step k-1's (u, w), then row sums of A v (into
// pr[strip][row]) and, below the diagonal, column sums of A^H v (into
// pc[chunk][column]).  The lower triangle is cut into strips of 64 columns and
// each strip into chunks of q rows, one per CTA; q is the smallest multiple of
// eight for which the chunks fit on the chip at once, so that every step is one
// wave of nearly equal CTAs however large its block is (64 x 64 tiles left a
// second wave of 40 tiles at order 1950, and one tile per SM at order 1050).
// Warp w takes rows w, w+8, ... of its chunk; lanes take columns lane and lane +
// 32.  A warp copies its rows' elements and their entries of u, w and v to its
// own part of shared memory two groups of four rows ahead; a consumed element's
// place takes the lane's row partial, and eight lanes per row add these up, in a
// fixed order.
// In double-float bound by the FP32 pipe (55 % issue, most of it two-wide): 232
// instructions an element, 362 with scalar arithmetic, 23 against 29 us at order
// 1950; 10 us at order 1050 and 5.5 at 150, most of it latency.  Two CTAs per SM
// leave the 128 registers that the columns' operands take.
template <typename R> struct FsPassBuf {
    fs_mem<R> x[2][FS_GROUP][FS_TB];
    fs_mem<R> uwv[2][FS_GROUP][3];
};
template <typename R>
__global__ void __launch_bounds__(FS_PASS_THREADS, FS_PASS_CTAS) k_fs_pass(FsArgs<R> a, int k, int q) {
    using C = cplx_t<R>;
    using M = fs_mem<R>;
    using Op = FsOps<R>;
    extern __shared__ __align__(16) unsigned char fs_smem[];
    FsPassBuf<R>* const bufs = reinterpret_cast<FsPassBuf<R>*>(fs_smem);
    const int n = a.n, j0 = k + 1, m = n - j0;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    launch_next();
    // strip and chunk of this CTA: a scan over the strips' chunk counts
    int strip = 0, chunk = 0;
    for (int base = 0, before = 0;; base += 32) {
        const int rows = m - FS_TB * (base + lane);
        int incl = rows > 0 ? fs_chunks(rows, q) : 0;
        const int own = incl;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(FULL_MASK, incl, o);
            if (lane >= o) incl += t;
        }
        const unsigned hit = __ballot_sync(FULL_MASK, (int)blockIdx.x < before + incl);
        const int f = hit ? __ffs(hit) - 1 : 31;
        if (hit) {
            strip = base + f;
            chunk = (int)blockIdx.x - before - __shfl_sync(FULL_MASK, incl - own, f);
            break;
        }
        before += __shfl_sync(FULL_MASK, incl, 31);
        if (base > m) return;  // past the last strip: not reached with the host's grid
    }
    const int c0 = FS_TB * strip, r0 = c0 + chunk * q, r1 = min(m, r0 + q);
    FsPassBuf<R>& buf = bufs[warp];
    const R z = fs_r<R>(0.f);
    const C zero = mk(z, z);
    M zero_m;
    fs_put(zero_m, zero);
    int cr[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) cr[h] = c0 + lane + 32 * h;
    const int nrow = r0 + warp < r1 ? (r1 - r0 - warp + FS_PASS_WARPS - 1) / FS_PASS_WARPS : 0;
    // offset of row ri (of the block) in A: below 2^32 elements for every order
    auto row_at = [&](int ri) { return (uint32_t)(j0 + ri) * (uint32_t)(j0 + ri + 1) / 2 + j0; };
    // group g of this warp's rows: warp + 8 (4 g + r) of the chunk
    auto fetch = [&](int g) {
#pragma unroll
        for (int r = 0; r < FS_GROUP; ++r) {
            const int ri = r0 + warp + FS_PASS_WARPS * (FS_GROUP * g + r);
            if (ri < r1) {
                const M* row = a.A + row_at(ri);
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    if (cr[h] <= ri) fs_copy16(&buf.x[g & 1][r][lane + 32 * h], row + cr[h]);
                if (lane < 3) fs_copy16(&buf.uwv[g & 1][r][lane], (lane == 0 ? a.U : lane == 1 ? a.W : a.V) + j0 + ri);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    wait_previous();
    fetch(0);
    fetch(1);
    typename Op::Col col[2];
    typename Op::Sum csum[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const bool in = cr[h] < m;
        const int j = j0 + cr[h];
        col[h] = Op::col(in ? fs_get(a.U[j]) : zero, in ? fs_get(a.W[j]) : zero, in ? fs_get(a.V[j]) : zero);
        csum[h] = Op::zero();
    }
    for (int g = 0; FS_GROUP * g < nrow; ++g) {
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncwarp();
        const int nr = min(FS_GROUP, nrow - FS_GROUP * g);
        for (int r = 0; r < nr; ++r) {
            const int ri = r0 + warp + FS_PASS_WARPS * (FS_GROUP * g + r);
            const typename Op::Row rw = Op::row(buf.uwv[g & 1][r]);
            M* row = a.A + row_at(ri);
            typename Op::Sum rsum = Op::zero();
            if (ri >= c0 + FS_TB) {  // below the strip's diagonal block: every lane, no conditions
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const M x = Op::update(buf.x[g & 1][r][lane + 32 * h], rw, col[h]);
                    row[cr[h]] = x;
                    Op::row_add(rsum, x, col[h], h == 0);
                    Op::col_add(csum[h], x, rw);
                }
            } else {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if (cr[h] <= ri) {
                        M x = Op::update(buf.x[g & 1][r][lane + 32 * h], rw, col[h]);
                        if (cr[h] == ri) Op::real(x);  // the diagonal stays real
                        row[cr[h]] = x;
                        Op::row_add(rsum, x, col[h], h == 0);
                        if (cr[h] < ri) Op::col_add(csum[h], x, rw);
                    }
                }
            }
            Op::save_row(&buf.x[g & 1][r][lane], rsum);
        }
        __syncwarp();
        {
            const int r = lane >> 3, part = lane & 7;
            M sum = zero_m;
            if (r < nr) fs_put(sum, Op::row_total(&buf.x[g & 1][r][part], 4, 8));
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) fs_acc(sum, fs_xor(sum, o));
            if (part == 0 && r < nr)
                fs_put(a.pr[(int64_t)strip * n + r0 + warp + FS_PASS_WARPS * (FS_GROUP * g + r)], fs_sum(sum));
        }
        __syncwarp();
        fetch(g + 2);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();
#pragma unroll
    for (int h = 0; h < 2; ++h) fs_put(buf.x[0][0][lane + 32 * h], Op::col_total(csum[h]));
    __syncthreads();
    if (threadIdx.x < FS_TB) {
        M sum = bufs[0].x[0][0][threadIdx.x];
#pragma unroll
        for (int w = 1; w < FS_PASS_WARPS; ++w) fs_acc(sum, bufs[w].x[0][0][threadIdx.x]);
        const int c = c0 + threadIdx.x;
        if (c < m) fs_put(a.pc[(int64_t)chunk * n + c], fs_sum(sum));
    }
}

// Partial `j` of row ri of A v: the row partials of strips 0 .. band (the row's own
// band), then the column partials of the band's chunks (a diagonal block's column
// sums hold the elements below the diagonal).
template <typename R> __device__ __forceinline__ fs_mem<R> fs_partial(const FsArgs<R>& a, int j, int band, int ri) {
    const fs_mem<R>* src = j <= band ? a.pr + (int64_t)j * a.n : a.pc + (int64_t)(j - band - 1) * a.n;
    return src[ri];
}

// p = tau (A v) of large blocks, spread over the chip.  A CTA takes 32 consecutive
// rows, one per lane; warp q adds the partials q, q+8, ..., and warp 0 adds the
// eight warps' sums, in a fixed order.
template <typename R>
__global__ void __launch_bounds__(FS_RED_THREADS) k_fs_reduce(FsArgs<R> a, int k, int q) {
    using C = cplx_t<R>;
    using M = fs_mem<R>;
    __shared__ M part[FS_RED_THREADS / 32][FS_RED_ROWS];
    const int n = a.n, j0 = k + 1, m = n - j0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ri = blockIdx.x * FS_RED_ROWS + lane;
    const R z = fs_r<R>(0.f);
    M s;
    fs_put(s, mk(z, z));
    launch_next();
    wait_previous();
    if (ri < m) {
        const int band = ri / FS_TB, np = band + 1 + fs_chunks(m - FS_TB * band, q);
#pragma unroll 4
        for (int j = warp; j < np; j += FS_RED_THREADS / 32) fs_acc(s, fs_partial(a, j, band, ri));
    }
    part[warp][lane] = s;
    __syncthreads();
    if (warp != 0 || ri >= m) return;
#pragma unroll
    for (int w = 1; w < FS_RED_THREADS / 32; ++w) fs_acc(s, part[w][lane]);
    const R tau = a.tau[k & 1];
    const C t = fs_sum(s);
    fs_put(a.p[j0 + ri], mk(t.x * tau, t.y * tau));
}

// Sum over the FS_SCALAR_THREADS threads of a scalar-phase CTA; every thread
// receives the same value (each warp's butterfly, then a butterfly over the
// 32 warp sums).  `red` holds 32 entries and is not read by another
// reduction until a later __syncthreads.
static_assert(FS_SCALAR_THREADS == 32 * 32, "fs_block_sum adds one value per warp in one warp");
template <typename R> __device__ __forceinline__ R fs_block_sum(R v, R* red) {
    v = warp_sum<R>(v);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    return warp_sum<R>(red[threadIdx.x & 31]);
}

// Column 0: d_0, ||x||^2 and the first reflector (one CTA).
template <typename R>
__global__ void __launch_bounds__(FS_SCALAR_THREADS) k_fs_setup(FsArgs<R> a) {
    using C = cplx_t<R>;
    __shared__ R red[FS_SCALAR_THREADS / 32];
    __shared__ C s_x0;
    const int n = a.n;
    R s2 = fs_r<R>(0.f);
    for (int i = 1 + threadIdx.x; i < n; i += blockDim.x) {
        const C x = fs_get(a.A[tri64(i)]);
        s2 = s2 + cabs2(x);
        if (i >= 2) fs_put(a.Vn[i], x);
        if (i == 1) s_x0 = x;
    }
    s2 = fs_block_sum<R>(s2, red);
    if (threadIdx.x == 0) {
        a.d[0] = fs_d(fs_get(a.A[0]).x);
        a.e2[0] = fs_d(s2);
        C f;
        R tau;
        reflector_head<R>(s2, s_x0, f, tau);
        fs_put(a.Vn[1], f);
        a.tau[0] = tau;
    }
}

// Step k's scalar phase: p = tau A v (its partials added up here, or by
// k_fs_reduce: `reduced`); w = p - (tau/2)(v^H p) v; the explicit update of pivot
// column j0 = k+1 with (v_k, w_k); d_j0, e2_j0 and, unless this was the last
// reflector, the next reflector v_{k+1} and tau_{k+1}.
// One cluster of eight CTAs: the two sums over all rows that it needs (v^H p and
// the next column's norm) cross between the CTAs through distributed shared memory
// and the hardware's cluster barrier.  Bound by latency: the loads of the partials
// (1 MB at order 1950, in flight at once), two barriers and the reflector's head.
// 9.3 us at order 1950, 7.4 at 150, where a reduction over the chip and one CTA
// took 16.
// CTA r takes blocks r, r + 8, ... of 256 rows: four threads of four warps add a
// row's partials, one of them keeps the row.
template <typename R> struct FsXch {
    R sum[2][FS_CL];
    cplx_t<R> p0;
};
__device__ __forceinline__ void fs_cluster_arrive() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void fs_cluster_wait() {
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// 16 or 8 bytes into the same place of CTA `rank`'s shared memory.
__device__ __forceinline__ unsigned fs_remote(const void* p, int rank) {
    unsigned d;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
    return d;
}
__device__ __forceinline__ void fs_remote_store(void* p, int rank, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(fs_remote(p, rank)), "d"(v) : "memory");
}
__device__ __forceinline__ void fs_remote_store(void* p, int rank, dfl v) {
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(fs_remote(p, rank)), "f"(v.hi), "f"(v.lo) : "memory");
}
// Sum over the cluster's row-keeping threads (warps 0 .. 7 of each CTA) of v, into
// every CTA's x.sum[which]; the caller passes the cluster barrier before it reads it.
template <typename R> __device__ __forceinline__ void fs_cluster_sum(R v, R* red, FsXch<R>& x, int which, int rank) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp < FS_STEP_ROWS / 32) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) fs_acc(v, shfl_xor_r(v, o));
        if (lane == 0) red[warp] = v;
    }
    __syncthreads();
    if (warp == 0) {
        v = red[lane % (FS_STEP_ROWS / 32)];
#pragma unroll
        for (int o = FS_STEP_ROWS / 64; o > 0; o >>= 1) fs_acc(v, shfl_xor_r(v, o));
        if (lane < FS_CL) fs_remote_store(&x.sum[which][rank], lane, fs_sum(v));
    }
}
template <typename R> __device__ __forceinline__ R fs_sum8(const R* s) {
    R a = s[0], b = s[2], c = s[4], d = s[6];
    fs_acc(a, s[1]);
    fs_acc(b, s[3]);
    fs_acc(c, s[5]);
    fs_acc(d, s[7]);
    fs_acc(a, b);
    fs_acc(c, d);
    fs_acc(a, c);
    return fs_sum(a);
}
template <typename R>
__global__ void __cluster_dims__(FS_CL, 1, 1) __launch_bounds__(FS_STEP_THREADS) k_fs_step(FsArgs<R> a, int k, int q,
                                                                                         bool reduced) {
    using C = cplx_t<R>;
    using M = fs_mem<R>;
    __shared__ M part[FS_STEP_PARTS][FS_STEP_ROWS];
    __shared__ R red[2][FS_STEP_ROWS / 32];
    __shared__ FsXch<R> xch;
    __shared__ C s_p0;
    const int n = a.n, j0 = k + 1, m = n - j0, rank = blockIdx.x;
    const int slot = threadIdx.x % FS_STEP_ROWS, pt = threadIdx.x / FS_STEP_ROWS;
    const bool keeper = pt == 0;
    const R z = fs_r<R>(0.f);
    const C zero = mk(z, z);
    // (no launch_next(): the next pass's CTAs would take their places while this
    // cluster still holds eight SMs; 1 % slower)
    fs_cluster_arrive();  // every CTA runs before any writes into another's memory
    wait_previous();
    const R tau = a.tau[k & 1];
    // the first block's entries, loaded ahead of the partials
    const int ri0 = rank * FS_STEP_ROWS + slot;
    C v1 = zero, x1 = zero, p1 = zero;
    if (keeper && ri0 < m) {
        v1 = fs_get(a.V[j0 + ri0]);
        x1 = fs_get(a.A[tri64(j0 + ri0) + j0]);
    }
    const C vf = fs_get(a.V[j0]);
    R sp = z;
    for (int rb = ri0 - slot; rb < m; rb += FS_CL * FS_STEP_ROWS) {
        const int ri = rb + slot;
        const bool first = ri == ri0;
        C s = zero;
        M acc;
        fs_put(acc, zero);
        if (!reduced) {
            if (ri < m) {
                const int band = ri / FS_TB, np = band + 1 + fs_chunks(m - FS_TB * band, q);
#pragma unroll 4
                for (int j = pt; j < np; j += FS_STEP_PARTS) fs_acc(acc, fs_partial(a, j, band, ri));
            }
            part[pt][slot] = acc;
            __syncthreads();
        }
        if (keeper && ri < m) {
            if (reduced) {
                s = fs_get(a.p[j0 + ri]);
            } else {
#pragma unroll
                for (int t = 1; t < FS_STEP_PARTS; ++t) fs_acc(acc, part[t][slot]);
                s = fs_sum(acc);
                s = mk(s.x * tau, s.y * tau);
                if (!first) fs_put(a.p[j0 + ri], s);
            }
            const C v = first ? v1 : fs_get(a.V[j0 + ri]);
            sp = sp + (v.x * s.x + v.y * s.y);
            if (first) p1 = s;
            if (ri == 0) s_p0 = s;
        }
        if (!reduced) __syncthreads();
    }
    fs_cluster_wait();
    fs_cluster_sum<R>(sp, red[0], xch, 0, rank);  // (its __syncthreads covers s_p0)
    if (rank == 0 && threadIdx.x < 2 * FS_CL) {
        const int to = threadIdx.x >> 1;
        if (threadIdx.x & 1) fs_remote_store(&xch.p0.y, to, s_p0.y);
        else fs_remote_store(&xch.p0.x, to, s_p0.x);
    }
    fs_cluster_arrive();
    fs_cluster_wait();
    const R K = fs_r<R>(0.5f) * tau * fs_sum8(xch.sum[0]);
    const C p0 = xch.p0;
    const C w0 = mk(p0.x - K * vf.x, p0.y - K * vf.y);
    R s2 = z;
    C w1 = zero;
    if (keeper) {
        for (int ri = ri0; ri < m; ri += FS_CL * FS_STEP_ROWS) {
            const bool first = ri == ri0;
            const int i = j0 + ri;
            const C v = first ? v1 : fs_get(a.V[i]), pi = first ? p1 : fs_get(a.p[i]);
            const C w = mk(pi.x - K * v.x, pi.y - K * v.y);
            if (first) w1 = w;
            else fs_put(a.Wn[i], w);
            C x = first ? x1 : fs_get(a.A[tri64(i) + j0]);
            x = cfms_conj_b(v, w0, x);
            x = cfms_conj_b(w, vf, x);
            if (ri >= 1) s2 = s2 + cabs2(x);
            if (first) x1 = x;
            else fs_put(a.Vn[i], x);
        }
    }
    fs_cluster_sum<R>(s2, red[1], xch, 1, rank);
    fs_cluster_arrive();
    // the first block's results go out while the barrier fills (ahead of it, its
    // release would wait for them)
    if (keeper && ri0 < m) {
        fs_put(a.Wn[j0 + ri0], w1);
        if (ri0 >= 2) fs_put(a.Vn[j0 + ri0], x1);
        if (ri0 == 0) a.d[j0] = fs_d(x1.x);
    }
    // row j0 + 1's keeper forms the reflector's head (reflector_head), the part
    // without the norm first
    const bool head = rank == 0 && threadIdx.x == 1;
    R ax0 = z;
    C ph = zero;
    if (head) {
        ax0 = sqroot(cabs2(x1));
        ph = ax0 > z ? mk(x1.x / ax0, x1.y / ax0) : mk(fs_r<R>(1.f), z);
    }
    fs_cluster_wait();
    if (head) {
        s2 = fs_sum8(xch.sum[1]);
        a.e2[j0] = fs_d(s2);
        if (k + 1 <= n - 3) {
            const R sigma = sqroot(s2);
            fs_put(a.Vn[j0 + 1], mk(x1.x + ph.x * sigma, x1.y + ph.y * sigma));
            a.tau[(k + 1) & 1] = sigma > z ? fs_r<R>(1.f) / (sigma * (sigma + ax0)) : z;
        }
    }
}

// The last diagonal entry: step n-3's update of A_{n-1,n-1} (V = v_{n-3},
// W = w_{n-3}).
template <typename R>
__global__ void k_fs_finish(FsArgs<R> a) {
    const int n = a.n;
    const auto v = fs_get(a.V[n - 1]), w = fs_get(a.W[n - 1]);
    a.d[n - 1] = fs_d(fs_get(a.A[tri64(n - 1) + n - 1]).x - fs_r<R>(2.f) * (v.x * w.x + v.y * w.y));
}

// Gershgorin bracket and Sturm-count guards of the tridiagonal (d, e2), and
// its float pairs (hi + lo = the FP64 entries exactly).  One CTA.
// prm: [0] lo, [1] hi, [2] pivmin (float), [3] nrm.
__global__ void __launch_bounds__(FS_SCALAR_THREADS) k_fs_eig_prep(int n, const double* __restrict__ d,
                                                                  const double* __restrict__ e2, float* df,
                                                                  float* dlo, float* e2f, float* e2lo, double* prm) {
    __shared__ double smin[FS_SCALAR_THREADS / 32], smax[FS_SCALAR_THREADS / 32], semax[FS_SCALAR_THREADS / 32];
    double lo = 1e300, hi = -1e300, em = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const double el = i > 0 ? sqrt(e2[i - 1]) : 0.0, er = i < n - 1 ? sqrt(e2[i]) : 0.0;
        lo = fmin(lo, d[i] - el - er);
        hi = fmax(hi, d[i] + el + er);
        const double ee = i < n - 1 ? e2[i] : 0.0;
        em = fmax(em, ee);
        df[i] = (float)d[i];
        dlo[i] = (float)(d[i] - (double)df[i]);
        e2f[i] = (float)ee;
        e2lo[i] = (float)(ee - (double)e2f[i]);
    }
    lo = warp_min(lo);
    hi = warp_max(hi);
    em = warp_max(em);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    if (lane == 0) { smin[warp] = lo; smax[warp] = hi; semax[warp] = em; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 0; w < nw; ++w) { lo = fmin(lo, smin[w]); hi = fmax(hi, smax[w]); em = fmax(em, semax[w]); }
        const double wdt = hi - lo, nrm = fmax(fabs(lo), fabs(hi));
        prm[0] = lo - (1e-12 * (wdt + nrm) + 1e-300);
        prm[1] = hi + (1e-12 * (wdt + nrm) + 1e-300);
        prm[2] = (double)(FLT_MIN * fmaxf(1.0f, (float)em));
        prm[3] = fmax(fabs(prm[0]), fabs(prm[1]));
    }
}

// Eigenvalue k (ascending), one thread each: FP32 bisection to a few FP32
// ulps of ||T||, then the widened bracket confirmed by double-float Sturm
// counts and finished by safeguarded double-float Newton (eig_df_bracketed).
__global__ void __launch_bounds__(FS_EIG_THREADS) k_fs_eig(int n, const float* __restrict__ df,
                                                          const float* __restrict__ dlo, const float* __restrict__ e2f,
                                                          const float* __restrict__ e2lo, const double* __restrict__ prm,
                                                          double* __restrict__ eig) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const double lo = prm[0], hi = prm[1], nrm = prm[3];
    const float pivminf = (float)prm[2];
    float a = (float)lo * (lo < 0 ? 1.0000002f : 0.9999998f) - 1e-30f;
    float b = (float)hi * (hi > 0 ? 1.0000002f : 0.9999998f) + 1e-30f;
    const float atolf = fmaxf(2.0f * FLT_EPSILON * (float)nrm, 1e-30f);
    for (int it = 0; it < 96 && b - a > atolf; ++it) {
        const float mid = 0.5f * (a + b);
        if (!(mid > a && mid < b)) break;
        if (sturm_count_f32(n, df, e2f, mid, pivminf) <= k) a = mid;
        else b = mid;
    }
    eig[k] = eig_df_bracketed(n, df, dlo, e2f, e2lo, k, a, b, 8.0 * FLT_EPSILON * nrm, lo, hi, pivminf, nrm);
}

// Rows of a chunk of the pass over a block of order m, and the chunks' number.
struct FsPlan { int q, chunks; };
static FsPlan fs_plan(int m, int slots) {
    auto count = [&](int q) {
        int c = 0;
        for (int rows = m; rows > 0; rows -= FS_TB) c += fs_chunks(rows, q);
        return c;
    };
    const int64_t rows = (int64_t)m * ((m + FS_TB - 1) / FS_TB) / 2;
    int q = std::clamp((int)(rows / slots) / 8 * 8, FS_MIN_ROWS, FS_MAX_ROWS), c = count(q);
    while (q < FS_MAX_ROWS && c > slots) c = count(q += 8);
    return {q, c};
}
// Blocks above this order have their partials added up by k_fs_reduce: the step
// cluster's eight SMs read 16 bytes per row and partial, 1 MB at order 2000.
constexpr int FS_FUSED_MAX = 4096;

// Reduction of the packed matrix A (in R's complex form) to the real
// tridiagonal (d, e2), enqueued on st.  The buffers are those of FsArgs, as
// raw device memory; v_k sits in vb[k mod 3] and w_k in wb[k mod 2], and
// v_{-1} = vb[2] and w_{-1} = wb[1] start at zero.
template <typename R>
static cudaError_t fs_tridiagonalise(int n, int slots, void* A, void* vb_, void* wb_, void* pr, void* pc, void* p, void* tau,
                                     double* d, double* e2, cudaStream_t st) {
    using C = fs_mem<R>;
    FsArgs<R> a;
    a.n = n;
    a.A = static_cast<C*>(A);
    a.pr = static_cast<C*>(pr);
    a.pc = static_cast<C*>(pc);
    a.p = static_cast<C*>(p);
    a.tau = static_cast<R*>(tau);
    a.d = d;
    a.e2 = e2;
    C* vb = static_cast<C*>(vb_);
    C* wb = static_cast<C*>(wb_);
    if (n == 2) {
        // d_0, d_1 and |e_0|^2 straight from the 2x2 matrix
        a.U = a.V = vb; a.Vn = vb; a.W = wb; a.Wn = wb;
        k_fs_setup<R><<<1, FS_SCALAR_THREADS, 0, st>>>(a);
        a.V = vb + n; a.W = wb;  // zero vectors: the finish reads A_11 unchanged
        k_fs_finish<R><<<1, 1, 0, st>>>(a);
        return cudaGetLastError();
    }
    a.Vn = vb;
    a.U = vb + 2 * (size_t)n;
    a.W = wb + n;
    a.V = vb;
    a.Wn = wb;
    const size_t smem = FS_PASS_WARPS * sizeof(FsPassBuf<R>);
    cudaError_t e = cudaFuncSetAttribute(k_fs_pass<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_fs_setup<R><<<1, FS_SCALAR_THREADS, 0, st>>>(a);
    e = cudaGetLastError();
    for (int k = 0; k <= n - 3 && e == cudaSuccess; ++k) {
        const int mm = n - k - 1;
        const FsPlan pl = fs_plan(mm, slots);
        const bool reduced = mm > FS_FUSED_MAX;
        a.U = vb + (size_t)((k + 2) % 3) * n;
        a.V = vb + (size_t)(k % 3) * n;
        a.Vn = vb + (size_t)((k + 1) % 3) * n;
        a.W = wb + (size_t)((k + 1) & 1) * n;
        a.Wn = wb + (size_t)(k & 1) * n;
        e = launch_chained(k_fs_pass<R>, (unsigned)pl.chunks, FS_PASS_THREADS, smem, st, a, k, pl.q);
        if (e == cudaSuccess && reduced)
            e = launch_chained(k_fs_reduce<R>, (unsigned)((mm + FS_RED_ROWS - 1) / FS_RED_ROWS), FS_RED_THREADS, 0, st, a, k, pl.q);
        if (e == cudaSuccess) e = launch_chained(k_fs_step<R>, FS_CL, FS_STEP_THREADS, 0, st, a, k, pl.q, reduced);
    }
    if (e != cudaSuccess) return e;
    a.V = vb + (size_t)((n - 3) % 3) * n;
    a.W = wb + (size_t)((n - 3) & 1) * n;
    k_fs_finish<R><<<1, 1, 0, st>>>(a);
    return cudaGetLastError();
}

}  // namespace ptca

ptca_status ptca_internal_fail(ptca_status s, const char* msg);
ptca::Model ptca_context_model(const ptca_ctx* ctx);

extern "C" ptca_status ptca_full_spectrum(ptca_ctx* ctx, double* eig_out, void* stream) {
    using namespace ptca;
    if (!ctx || !eig_out) return ptca_internal_fail(PTCA_ERR_INVALID, "null argument");
    const int N = ctx->N;
    if (N > 16384) return ptca_internal_fail(PTCA_ERR_INVALID, "ptca_full_spectrum covers lattices of up to 16384 sites");
    const int n = 2 * N;
    const int Tmax = std::max((n - 1 + FS_TB - 1) / FS_TB, 1), slots = FS_PASS_CTAS * ctx->sms;
    int cmax = 1;  // most chunks of a strip (its first) in any step
    for (int mm = n - 1; mm >= 2; --mm) cmax = std::max(cmax, fs_chunks(mm, fs_plan(mm, slots).q));
    cudaError_t es = ptca_internal_settle(ctx, static_cast<cudaStream_t>(stream), true);
    if (es != cudaSuccess) return ptca_internal_fail(PTCA_ERR_CUDA, cudaGetErrorString(es));
    cudaStream_t st = static_cast<cudaStream_t>(stream);

    std::vector<void*> owned;
    auto alloc = [&](size_t bytes) -> void* {
        void* q = nullptr;
        if (cudaMalloc(&q, bytes) != cudaSuccess) return nullptr;
        owned.push_back(q);
        return q;
    };
    auto release = [&]() {
        cudaStreamSynchronize(st);
        for (void* q : owned) cudaFree(q);
    };
    // + 64 elements of padding past the packed triangle
    double2* A = static_cast<double2*>(alloc(((size_t)tri64(n) + 64) * sizeof(double2)));
    double2* vb = static_cast<double2*>(alloc(3 * (size_t)n * sizeof(double2)));
    double2* wb = static_cast<double2*>(alloc(2 * (size_t)n * sizeof(double2)));
    double2* p = static_cast<double2*>(alloc((size_t)n * sizeof(double2)));
    double2* pr = static_cast<double2*>(alloc((size_t)Tmax * n * sizeof(double2)));
    double2* pc = static_cast<double2*>(alloc((size_t)cmax * n * sizeof(double2)));
    double* tau = static_cast<double*>(alloc(2 * sizeof(double)));
    double* d = static_cast<double*>(alloc((size_t)n * sizeof(double)));
    double* e2 = static_cast<double*>(alloc((size_t)n * sizeof(double)));
    float* f32 = static_cast<float*>(alloc(4 * (size_t)n * sizeof(float)));
    double* prm = static_cast<double*>(alloc(4 * sizeof(double)));
    for (void* q : {(void*)A, (void*)vb, (void*)wb, (void*)p, (void*)pr, (void*)pc, (void*)tau, (void*)d,
                    (void*)e2, (void*)f32, (void*)prm})
        if (!q) {
            release();
            return ptca_internal_fail(PTCA_ERR_OOM, "ptca_full_spectrum: not enough device memory for the matrix");
        }
    auto fail = [&](cudaError_t e, const char* where) {
        release();
        cudaGetLastError();
        return ptca_internal_fail(PTCA_ERR_CUDA, (std::string("ptca_full_spectrum: ") + where + ": " +
                                                  cudaGetErrorString(e)).c_str());
    };
    cudaError_t e = cudaMemsetAsync(A, 0, ((size_t)tri64(n) + 64) * sizeof(double2), st);
    if (e == cudaSuccess) e = cudaMemsetAsync(vb, 0, 3 * (size_t)n * sizeof(double2), st);
    if (e == cudaSuccess) e = cudaMemsetAsync(wb, 0, 2 * (size_t)n * sizeof(double2), st);
    if (e == cudaSuccess) e = cudaMemsetAsync(e2, 0, (size_t)n * sizeof(double), st);
    if (e != cudaSuccess) return fail(e, "clearing the buffers");
    const Model m = ptca_context_model(ctx);
    k_full_hamiltonian<<<(N + 255) / 256, 256, 0, st>>>(m, ctx->d_S[0], N, A);
    if ((e = cudaGetLastError()) != cudaSuccess) return fail(e, "building the matrix");

    if (ctx->prec == 1) {
        // PTCA_MIXED: the reduction in double-float
        const int64_t cnt = tri64(n) + 64;
        k_fs_to_dfl<<<(unsigned)std::min<int64_t>((cnt + 255) / 256, 152 * 16), 256, 0, st>>>(A, cnt);
        e = fs_tridiagonalise<dfl>(n, slots, A, vb, wb, pr, pc, p, tau, d, e2, st);
    } else {
        e = fs_tridiagonalise<double>(n, slots, A, vb, wb, pr, pc, p, tau, d, e2, st);
    }
    if (e != cudaSuccess) return fail(e, "reducing to tridiagonal form");
    float* df = f32;
    float* dlo = f32 + n;
    float* e2f = f32 + 2 * (size_t)n;
    float* e2lo = f32 + 3 * (size_t)n;
    k_fs_eig_prep<<<1, FS_SCALAR_THREADS, 0, st>>>(n, d, e2, df, dlo, e2f, e2lo, prm);
    k_fs_eig<<<(n + FS_EIG_THREADS - 1) / FS_EIG_THREADS, FS_EIG_THREADS, 0, st>>>(n, df, dlo, e2f, e2lo, prm, eig_out);
    if ((e = cudaGetLastError()) != cudaSuccess) return fail(e, "eigenvalues");
    e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return fail(e, "synchronising");
    release();
    return PTCA_OK;
}

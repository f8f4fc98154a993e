// resolvent.cuh -- free energies of a visit from determinants of its cluster
// matrix, without an eigenvalue.
//
// F = -T sum_k ln(1 + e^(-x_k)), x = (eps - mu)/T, is a short sum of
// ln|det(mu - H + i T y_j)| over nodes y_j plus Tr H and Tr H^2
// (fermi_nodes.cuh); the phases of the same determinants give the filling.
// The window's hopping couples only neighbouring layers of sites, by a
// multiple of the identity.  So the matrix is eliminated layer by layer with
// blocks of order B = 2 (sites per layer), the update site last:
//   A = (mu - H)/(T y) + i,   D_0 = A_00,
//   X_k = D_k^-1,  D_{k+1} = A_{k+1,k+1} - t'^2 X_k        (t' = t/(T y)),
// and, on a ring of layers, with the border blocks C_k, E_k that couple layer
// k to the last one: C_{k+1} = -t' X_k C_k, E_{k+1} = -t' E_k X_k,
// S -= E_k X_k C_k.  Every Schur complement of A keeps an imaginary part
// of at least 1, so its 2x2 (one site's) pivots are never small, no pivoting is
// needed, and the phases of their determinants add up without a branch cut.
// H_new differs from H_old in the update site's 2x2 block alone: both visits'
// determinants share every pivot but the last, dF comes from the last one, and
// the rounding of the elimination cancels in it.
//
// Work per node: about (4 (L - 2) + 2) B^3 complex multiply-adds on a ring of L
// layers, (L - 1) B^3 on an open one, against (4/3) n^3 for a Householder
// reduction of each of the two matrices (n = B L): 0.10 M against 5.6 M at
// n = 128, times 13 nodes at |x| <= 512.
//
// Short rings pay three products per layer for little.  Where every bond joins
// sites of opposite parity the parity that the update site does not have can
// go first: its 2x2 pivots are independent, and what is left is a dense matrix of
// half the order, done as two blocks with two inversions and two products
// (RsPairs).  It is taken on rings of four layers (4x4 and 4x4x4 clusters):
// 4 b^3 multiply-adds instead of 9 b^3.
//
// One node is eliminated by LPN lanes of a warp, which holds 32 / LPN nodes: the
// larger the tile per lane, the fewer shuffles and loads per multiply-add.
// Lane (r, c) of a GR x GC grid holds the rows of sites r + GR i and the columns of
// sites c + GC j (both spins) in registers.  The pivot block, row and column
// travel by shuffles (Gauss-Jordan in place, one site's two rows at a time);
// the products read their operands from shared memory, where a matrix row is
// padded by two elements so that the row groups hit different banks.
#pragma once

#include "fermi_nodes.cuh"
#include "kernels.cuh"

namespace ptca {

__device__ __forceinline__ dfl2 cfms(dfl2 a, dfl2 b, dfl2 acc) {
    return mk(dot2_acc(acc.x, -a.x, b.x, a.y, b.y), dot2_acc(acc.y, -a.x, b.y, -a.y, b.x));
}
__device__ __forceinline__ float2 shfl_c(float2 v, int src) {
    v.x = __shfl_sync(FULL_MASK, v.x, src);
    v.y = __shfl_sync(FULL_MASK, v.y, src);
    return v;
}
// Two consecutive elements of a matrix row (the first at an even index).
__device__ __forceinline__ void ld2(const float2* p, float2& a, float2& b) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    a = make_float2(v.x, v.y);
    b = make_float2(v.z, v.w);
}
__device__ __forceinline__ void st2(float2* p, float2 a, float2 b) {
    *reinterpret_cast<float4*>(p) = make_float4(a.x, a.y, b.x, b.y);
}

// Scalar helpers of the two arithmetics.
__device__ __forceinline__ float rs_rcp(float x) { return __fdividef(1.f, x); }
// Newton correction r (1 + e + e^2) of the FP32 reciprocal, e = 1 - x r from one
// fused multiply-add each for the two parts of x: relative error a few 2^-48.
__device__ __forceinline__ dfl rs_rcp(dfl x) {
    const float r = __fdividef(1.f, x.hi);
    const float e = __fmaf_rn(-x.lo, r, __fmaf_rn(-x.hi, r, 1.f));
    return fast_two_sum(r, r * __fmaf_rn(e, e, e));
}
__device__ __forceinline__ float rs_log1p(float q) { return log1pf(q); }
__device__ __forceinline__ double rs_log1p(dfl q) { return log1p(double(q)); }
__device__ __forceinline__ float rs_phase(float y, float x) { return atan2f(y, x); }
__device__ __forceinline__ double rs_phase(dfl y, dfl x) { return atan2(double(y), double(x)); }

__device__ __forceinline__ float2 cmulp(float2 a, float2 b) {
    return make_float2(__fmaf_rn(-a.y, b.y, a.x * b.x), __fmaf_rn(a.y, b.x, a.x * b.y));
}
// g with 1 + g = -det(P + i): the determinant of a pivot block (stored without
// its i) against i^2.
template <typename V> __device__ __forceinline__ V rs_det_g(V p00, V p01, V p10, V p11) {
    V m;
    m.x = p00.x * p11.x; m.y = p00.x * p11.y;
    m.x = m.x - p00.y * p11.y;
    m.y = m.y + p00.y * p11.x;
    m = cfms(p01, p10, m);
    m = mk(p00.y + p11.y - m.x, -(p00.x + p11.x + m.y));
    return m;
}

__device__ __forceinline__ void rs_get(float& x, const volatile float* p) { x = *p; }
__device__ __forceinline__ void rs_get(dfl& x, const volatile dfl* p) { x = dfl(p->hi, p->lo); }

// Running sum of a lane's logarithms or phases: a float pair in FP32 (the
// pivots' own rounding is all that is left), FP64 in double-float.
template <typename T> struct RsSum;
template <> struct RsSum<float> {
    dfl v = dfl(0.f, 0.f);
    __device__ __forceinline__ void add(float x) {
        const dfl s = two_sum(v.hi, x);
        v = dfl(s.hi, v.lo + s.lo);
    }
    __device__ __forceinline__ void merge(int o) { v = v + shfl_xor_dfl(v, o); }
    __device__ __forceinline__ double value() const { return double(v); }
};
template <> struct RsSum<dfl> {
    double v = 0.0;
    __device__ __forceinline__ void add(double x) { v += x; }
    __device__ __forceinline__ void merge(int o) { v += __shfl_xor_sync(FULL_MASK, v, o); }
    __device__ __forceinline__ double value() const { return v; }
};

// On-site terms of a window site: mu - H = [[d + z, x - iy], [x + iy, d - z]], in
// units of |t| (RsUnit), so that the scaled hopping is the scale s itself.
template <typename T> struct RsSite { T d, x, y, z; };
// P: the last pivot block, without its i; s = unit / (T y), rounded; eta: its relative rounding error.
template <typename T> struct RsOut { double lnd, th; T P[8], s; float eta; };

// Window of a visit in layer order.
struct RsVisit {
    int c, site, n, L, ns, u, us;   // stage index, lattice site, order, layers, sites per layer, update layer and site
    int per, cls;                   // cluster periodic; node class (-1: |x| beyond the last class)
};
// A window split by parity: kept sites (of the update site's parity) in two
// blocks, block 1 ending with the update site; eliminated sites; for each kept
// site the set of its eliminated neighbours.
struct RsPairs {
    int na, nb, ne;                 // sites of block 0, of block 1, eliminated
    int kept[32], gone[32];         // window sites (layer order); kept: block 0, then block 1
    uint32_t near[32], place[32];   // place: coordinates of the eliminated sites, packed
};
constexpr int kPairSites = 64;      // largest window

// Sums over the window, FP64.
struct RsTerms { double x1, x2, cl, sn[3], lnu; float dv[4]; };  // dv: change of (d, x, y, z) of RsSite, rounded

template <int GR_, int GC_, int SR_, int SC_, int MAXT_, int MINB_> struct RsTile {
    static constexpr int GR = GR_, GC = GC_, SR = SR_, SC = SC_;
    static constexpr int MAXT = MAXT_, MINB = MINB_;       // launch bounds of the stage kernels
    static constexpr int NS = GR * SR, B = 2 * NS, RS = B + 2;
    static constexpr int LPN = GR * GC, NPW = 32 / LPN;
    // Elements of a node's buffers: padded so that the nodes of a warp start in
    // different banks.
    static constexpr int PAD = NPW == 1 ? 0 : LPN >= 16 ? 8 : LPN > 1 ? 2 * LPN : 2;
    static constexpr int node(bool pairs) { return (pairs ? 2 * B * RS + 8 * NS : 3 * B * RS) + PAD; }
    static_assert(GR * SR == GC * SC && GR % GC == 0 && 32 % LPN == 0, "square blocks");
};
using RsT1 = RsTile<1, 1, 1, 1, 256, 2>;    // chains: a node per lane
using RsT4 = RsTile<2, 2, 2, 2, 256, 2>;    // up to 4 sites per layer: 4x4 per lane, eight nodes per warp
using RsT8 = RsTile<4, 4, 2, 2, 224, 2>;    // two nodes per warp
using RsT12 = RsTile<4, 4, 3, 3, 224, 1>;   // 6x6 per lane
using RsT16 = RsTile<8, 4, 2, 4, 256, 1>;   // 4x8 per lane, one node per warp
// Stages of few visits: more lanes per node.
using RsL4 = RsTile<4, 4, 1, 1, 256, 1>;
using RsL8 = RsTile<8, 4, 1, 2, 256, 1>;

template <class Tl> struct RsNode {
    using V = float2;
    static constexpr int GR = Tl::GR, GC = Tl::GC, SR = Tl::SR, SC = Tl::SC, NS = Tl::NS, RS = Tl::RS;
    using Tile = V[2 * SR][2 * SC];

    // Tile row a: spin a / SR of site r + GR (a % SR); column likewise.  In
    // memory rows are grouped by spin and columns by site (the two spins of a
    // site in one 16-byte load), so that a row of the left operand and the
    // matching row of the right one are col = 2 site + spin apart.
    static __device__ __forceinline__ int row(int r, int a) { return (a / SR) * NS + r + GR * (a % SR); }
    static __device__ __forceinline__ int csite(int c, int s) { return c + GC * s; }
    static __device__ __forceinline__ V shfl(V v, int src) { return Tl::LPN == 1 ? v : shfl_c(v, src); }

    static __device__ __forceinline__ void store(V* M, const Tile& a, int r, int c) {
#pragma unroll
        for (int i = 0; i < 2 * SR; ++i) {
            V* p = M + row(r, i) * RS;
#pragma unroll
            for (int j = 0; j < SC; ++j) st2(p + 2 * csite(c, j), a[i][j], a[i][SC + j]);
        }
    }

    static __device__ __forceinline__ void load(Tile& a, const V* M, int r, int c) {
#pragma unroll
        for (int i = 0; i < 2 * SR; ++i)
#pragma unroll
            for (int j = 0; j < SC; ++j) ld2(M + row(r, i) * RS + 2 * csite(c, j), a[i][j], a[i][SC + j]);
    }

    // o = P Q
    static __device__ __forceinline__ void mul(Tile& o, const V* P, const V* Q, int ns, int r, int c) {
#pragma unroll
        for (int i = 0; i < 2 * SR; ++i)
#pragma unroll
            for (int j = 0; j < 2 * SC; ++j) o[i][j] = make_float2(0.f, 0.f);
#pragma unroll 2
        for (int k = 0; k < ns; ++k) {   // site k: its two columns of P, its two rows of Q
            V p[2 * SR][2];
#pragma unroll
            for (int i = 0; i < 2 * SR; ++i) ld2(P + row(r, i) * RS + 2 * k, p[i][0], p[i][1]);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const V* q = Q + (h * NS + k) * RS;
                V b[2 * SC];
#pragma unroll
                for (int j = 0; j < SC; ++j) ld2(q + 2 * csite(c, j), b[j], b[SC + j]);
#pragma unroll
                for (int i = 0; i < 2 * SR; ++i)
#pragma unroll
                    for (int j = 0; j < 2 * SC; ++j) o[i][j] = cfma(p[i][h], b[j], o[i][j]);
            }
        }
    }
    // M = f o, between the warp's last read of the operands and the next
    static __device__ __forceinline__ void put(V* M, Tile& o, float f, int r, int c) {
#pragma unroll
        for (int i = 0; i < 2 * SR; ++i)
#pragma unroll
            for (int j = 0; j < 2 * SC; ++j) o[i][j] = make_float2(f * o[i][j].x, f * o[i][j].y);
        __syncwarp();
        store(M, o, r, c);
        __syncwarp();
    }

    // The block of layer l without its i on the diagonal, minus t'^2 X (X in a); t'
    // is applied twice, since a rounded t'^2 would be off by as much on every bond.
    static __device__ __forceinline__ void layer(Tile& a, const RsSite<float>* site, const float* hop, float s, float tp,
                                                 int ns, int r, int c, bool chain) {
#pragma unroll
        for (int i = 0; i < SR; ++i) {
            const int sr = r + GR * i;
            const float f = sr < ns ? tp : 0.f;
#pragma unroll
            for (int j = 0; j < SC; ++j) {
                const int sc = csite(c, j);
                const float h = hop[sr * NS + sc] * s;
                V uu = make_float2(h, 0.f), dd = uu, ud = make_float2(0.f, 0.f), du = ud;
                if (sr == sc && sr < ns) {
                    const RsSite<float> o = site[sr];
                    const float x = o.x * s, y = o.y * s;
                    uu.x = (o.d + o.z) * s;
                    dd.x = (o.d - o.z) * s;
                    ud = make_float2(x, -y);
                    du = make_float2(x, y);
                }
                if (chain) {
                    const V x00 = a[i][j], x01 = a[i][SC + j], x10 = a[SR + i][j], x11 = a[SR + i][SC + j];
                    uu = make_float2(uu.x - f * (f * x00.x), -(f * (f * x00.y)));
                    dd = make_float2(dd.x - f * (f * x11.x), -(f * (f * x11.y)));
                    ud = make_float2(ud.x - f * (f * x01.x), ud.y - f * (f * x01.y));
                    du = make_float2(du.x - f * (f * x10.x), du.y - f * (f * x10.y));
                }
                a[i][j] = uu;
                a[SR + i][SC + j] = dd;
                a[i][SC + j] = ud;
                a[SR + i][j] = du;
            }
        }
    }

    // Gauss-Jordan inversion in place of the block a + i, one site at a time;
    // site `skip` and the padding from ns on are left out.  The sums of
    // ln|det|^2 and of the phases of the 2x2 pivots (against i^2) go to lnd, th.
    // The pivots of one round lie in tile row 0 and columns 0 .. GR/GC - 1;
    // the tile is turned by a round's worth afterwards (SR rounds are a full
    // turn), so that the body exists once: unrolled over the rounds it
    // overflowed the instruction cache (1.45 no-instruction stalls per issue).
    static __device__ __forceinline__ void invert(Tile& a, RsSum<float>& lnd, RsSum<float>& th, int skip, int ns, int r, int c,
                                                  int nl, int base) {
        constexpr int QR = GR / GC;
        static_assert(NS <= Tl::LPN || NS == 1, "a lane per pivot");
        const V zero = make_float2(0.f, 0.f);
        V g = zero;
#pragma unroll 1
        for (int p0 = 0; p0 < ns; p0 += GR) {
#pragma unroll
            for (int s = 0; s < QR; ++s) {
#pragma unroll 1
                for (int cp = 0; cp < GC; ++cp) {
                    const int rp = s * GC + cp, p = p0 + rp;
                    if (p == skip || p >= ns) continue;
                    const int src = base + rp * GC + cp;
                    const V p00 = shfl(a[0][s], src), p01 = shfl(a[0][SC + s], src);
                    const V p10 = shfl(a[SR][s], src), p11 = shfl(a[SR][SC + s], src);
                    const V gp = rs_det_g(p00, p01, p10, p11);
                    if (nl == p) g = gp;
                    // inverse of P + i: -(adj) conj(1 + g)/|1 + g|^2
                    const float gr = 1.f + gp.x, rq = rs_rcp(gr * gr + gp.y * gp.y);
                    const V w = make_float2(-(gr * rq), gp.y * rq), wn = make_float2(-w.x, -w.y);   // 1/det
                    const V i00 = cmulp(make_float2(p11.x, p11.y + 1.f), w), i11 = cmulp(make_float2(p00.x, p00.y + 1.f), w);
                    const V i01 = cmulp(p01, wn), i10 = cmulp(p10, wn);
                    const bool pr = r == rp, pc = c == cp;
                    V q0[2 * SR], q1[2 * SR];
                    const int csrc = base + r * GC + cp, rsrc = base + rp * GC + c;
#pragma unroll
                    for (int k = 0; k < 2 * SR; ++k) {
                        const V c0 = shfl(a[k][s], csrc), c1 = shfl(a[k][SC + s], csrc);
                        q0[k] = cfma(c1, i10, cmulp(c0, i00));
                        q1[k] = cfma(c1, i11, cmulp(c0, i01));
                    }
                    if (pr) {
                        q0[0] = make_float2(-i00.x, -i00.y);
                        q1[0] = make_float2(-i01.x, -i01.y);
                        q0[SR] = make_float2(-i10.x, -i10.y);
                        q1[SR] = make_float2(-i11.x, -i11.y);
                    }
#pragma unroll
                    for (int j = 0; j < 2 * SC; ++j) {
                        const V r0 = shfl(a[0][j], rsrc), r1 = shfl(a[SR][j], rsrc);
                        if (pr) { a[0][j] = zero; a[SR][j] = zero; }
#pragma unroll
                        for (int k = 0; k < 2 * SR; ++k) a[k][j] = cfms(q1[k], r1, cfms(q0[k], r0, a[k][j]));
                    }
                    if (pc) {
#pragma unroll
                        for (int k = 0; k < 2 * SR; ++k) {
                            a[k][s] = make_float2(-q0[k].x, -q0[k].y);
                            a[k][SC + s] = make_float2(-q1[k].x, -q1[k].y);
                        }
                    }
                }
            }
            turn(a);
        }
        // padding shorter than a full turn
#pragma unroll 1
        for (int p0 = (ns + GR - 1) / GR; p0 < SR; ++p0) turn(a);
        if (nl < NS) {
            lnd.add(log1pf((g.x + g.x) + (g.x * g.x + g.y * g.y)));
            th.add(atan2f(g.y, 1.f + g.x));
        }
    }
    static __device__ __forceinline__ void turn(Tile& a) {
        if constexpr (SR > 1) {
            Tile b;
#pragma unroll
            for (int i = 0; i < 2 * SR; ++i)
#pragma unroll
                for (int j = 0; j < 2 * SC; ++j)
                    b[i][j] = a[(i / SR) * SR + (i % SR + 1) % SR][(j / SC) * SC + (j % SC + GR / GC) % SC];
#pragma unroll
            for (int i = 0; i < 2 * SR; ++i)
#pragma unroll
                for (int j = 0; j < 2 * SC; ++j) a[i][j] = b[i][j];
        }
    }

    // o = P^t Q with P^t the block transpose of P (2x2 blocks stay as they are)
    static __device__ __forceinline__ void mul_t(Tile& o, const V* P, const V* Q, int ns, int r, int c) {
#pragma unroll
        for (int i = 0; i < 2 * SR; ++i)
#pragma unroll
            for (int j = 0; j < 2 * SC; ++j) o[i][j] = make_float2(0.f, 0.f);
#pragma unroll 2
        for (int k = 0; k < ns; ++k) {
            V p[2 * SR][2];
#pragma unroll
            for (int i = 0; i < 2 * SR; ++i) ld2(P + ((i / SR) * NS + k) * RS + 2 * (r + GR * (i % SR)), p[i][0], p[i][1]);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const V* q = Q + (h * NS + k) * RS;
                V b[2 * SC];
#pragma unroll
                for (int j = 0; j < SC; ++j) ld2(q + 2 * csite(c, j), b[j], b[SC + j]);
#pragma unroll
                for (int i = 0; i < 2 * SR; ++i)
#pragma unroll
                    for (int j = 0; j < 2 * SC; ++j) o[i][j] = cfma(p[i][h], b[j], o[i][j]);
            }
        }
    }

    // Block (row0, col0) of the kept sites' matrix after the eliminated parity:
    // on-site terms (without i) minus t'^2 times the pivot inverses of common
    // neighbours (inv: 4 elements per eliminated site).
    static __device__ __forceinline__ void pair_block(Tile& a, const RsPairs& pt, int row0, int nr, int col0, int nc,
                                                      const RsSite<float>* site, const V* inv, float s, float tp, int r, int c) {
#pragma unroll 1
        for (int i = 0; i < SR; ++i)
#pragma unroll 1
            for (int j = 0; j < SC; ++j) {
                const int x = r + GR * i, y = csite(c, j);
                V uu = make_float2(0.f, 0.f), ud = uu, du = uu, dd = uu;
                if (x < nr && y < nc) {
                    uint32_t both = pt.near[row0 + x] & pt.near[col0 + y];
                    while (both) {
                        const int e = __ffs(both) - 1;
                        both &= both - 1;
                        V p, q;
                        ld2(inv + 4 * e, p, q);
                        uu = csub(uu, p);
                        ud = csub(ud, q);
                        ld2(inv + 4 * e + 2, p, q);
                        du = csub(du, p);
                        dd = csub(dd, q);
                    }
                    uu = make_float2(tp * (tp * uu.x), tp * (tp * uu.y));
                    ud = make_float2(tp * (tp * ud.x), tp * (tp * ud.y));
                    du = make_float2(tp * (tp * du.x), tp * (tp * du.y));
                    dd = make_float2(tp * (tp * dd.x), tp * (tp * dd.y));
                    if (row0 + x == col0 + y) {
                        const RsSite<float> o = site[pt.kept[row0 + x]];
                        uu.x += (o.d + o.z) * s;
                        dd.x += (o.d - o.z) * s;
                        ud = make_float2(ud.x + o.x * s, ud.y - o.y * s);
                        du = make_float2(du.x + o.x * s, du.y + o.y * s);
                    }
                }
#pragma unroll
                for (int k = 0; k < SR; ++k)
#pragma unroll
                    for (int l = 0; l < SC; ++l)
                        if (k == i && l == j) {
                            a[k][l] = uu;
                            a[k][SC + l] = ud;
                            a[SR + k][l] = du;
                            a[SR + k][SC + l] = dd;
                        }
            }
    }

    static __device__ __forceinline__ void finish(const Tile& a, int us, float s, RsSum<float>& lnd, RsSum<float>& th, int r,
                                                  int c, int nl, RsOut<float>* out) {
        // last pivot block: the lane holding rows and columns of the update site
#pragma unroll
        for (int i = 0; i < SR; ++i)
#pragma unroll
            for (int j = 0; j < SC; ++j)
                if (r + GR * i == us && csite(c, j) == us) {
                    out->P[0] = a[i][j].x; out->P[1] = a[i][j].y;
                    out->P[2] = a[i][SC + j].x; out->P[3] = a[i][SC + j].y;
                    out->P[4] = a[SR + i][j].x; out->P[5] = a[SR + i][j].y;
                    out->P[6] = a[SR + i][SC + j].x; out->P[7] = a[SR + i][SC + j].y;
                }
#pragma unroll
        for (int o = Tl::LPN / 2; o > 0; o >>= 1) {
            lnd.merge(o);
            th.merge(o);
        }
        if (nl == 0) {
            out->lnd = 0.5 * lnd.value();
            out->th = th.value();
            out->s = s;
        }
        __syncwarp();
    }

    // run() for a window split by parity.
    static __device__ __forceinline__ void run_pairs(const RsPairs& pt, const RsSite<float>* site, float s, float tp, V* buf,
                                                     int lane, RsOut<float>* out) {
        const int base = lane & ~(Tl::LPN - 1), nl = lane - base;
        const int r = nl / GC, c = nl % GC;
        V *X = buf, *C = buf + Tl::B * RS, *inv = C + Tl::B * RS;
        RsSum<float> lnd, th;
        for (int e = nl; e < pt.ne; e += Tl::LPN) {
            const RsSite<float> o = site[pt.gone[e]];
            const V p00 = make_float2((o.d + o.z) * s, 0.f), p11 = make_float2((o.d - o.z) * s, 0.f);
            const V p01 = make_float2(o.x * s, -(o.y * s)), p10 = make_float2(o.x * s, o.y * s);
            const V g = rs_det_g(p00, p01, p10, p11);
            const float gr = 1.f + g.x, rq = rs_rcp(gr * gr + g.y * g.y);
            const V w = make_float2(-(gr * rq), g.y * rq), wn = make_float2(-w.x, -w.y);
            st2(inv + 4 * e, cmulp(make_float2(p11.x, 1.f), w), cmulp(p01, wn));
            st2(inv + 4 * e + 2, cmulp(p10, wn), cmulp(make_float2(p00.x, 1.f), w));
            lnd.add(log1pf((g.x + g.x) + (g.x * g.x + g.y * g.y)));
            th.add(atan2f(g.y, 1.f + g.x));
        }
        __syncwarp();
        Tile a, S;
        pair_block(a, pt, 0, pt.na, 0, pt.na, site, inv, s, tp, r, c);
#pragma unroll 1
        for (int o = 0;; ++o) {
            invert(a, lnd, th, o == 0 ? -1 : pt.nb - 1, o == 0 ? pt.na : pt.nb, r, c, nl, base);
            if (o) break;
            store(X, a, r, c);
            pair_block(a, pt, 0, pt.na, pt.na, pt.nb, site, inv, s, tp, r, c);
            store(C, a, r, c);
            pair_block(S, pt, pt.na, pt.nb, pt.na, pt.nb, site, inv, s, tp, r, c);
            __syncwarp();
            mul(a, X, C, pt.na, r, c);
            put(X, a, 1.f, r, c);
            mul_t(a, C, X, pt.na, r, c);
#pragma unroll
            for (int i = 0; i < 2 * SR; ++i)
#pragma unroll
                for (int j = 0; j < 2 * SC; ++j) a[i][j] = csub(S[i][j], a[i][j]);
        }
        finish(a, pt.nb - 1, s, lnd, th, r, c, nl, out);
    }

    // One node of one visit: the sums over all pivots but the update site's,
    // and that site's last pivot block.  s: unit / (T y), tp: t / (T y) = +-s.
    static __device__ __forceinline__ void run(const RsVisit& v, const RsSite<float>* site, const float* hop, float s, float tp,
                                               V* buf, int lane, RsOut<float>* out) {
        const int base = lane & ~(Tl::LPN - 1), nl = lane - base;
        const int r = nl / GC, c = nl % GC;
        const int L = v.L, ns = v.ns;
        V *X = buf, *C = buf + Tl::B * RS, *E = C + Tl::B * RS;
        const bool ring = v.per && L >= 3;
        Tile a, S;
        RsSum<float> lnd, th;
        layer(S, site + v.u * ns, hop, s, tp, ns, r, c, false);
#pragma unroll 1
        for (int o = 0; o < L; ++o) {
            const bool last = o == L - 1;
            if (last) {
#pragma unroll
                for (int i = 0; i < 2 * SR; ++i)
#pragma unroll
                    for (int j = 0; j < 2 * SC; ++j) a[i][j] = S[i][j];
            } else {
                // elimination order: round the ring from the update layer, or
                // from both ends of an open window towards it
                int l;
                if (v.per) { l = v.u + 1 + o; if (l >= L) l -= L; }
                else l = o < v.u ? o : L - 1 - (o - v.u);
                layer(a, site + l * ns, hop, s, tp, ns, r, c, o > 0 && (v.per || o != v.u));
            }
            invert(a, lnd, th, last ? v.us : -1, ns, r, c, nl, base);
            if (last) break;
            if (ring && o > 0) {
                // Stored: W_k = E_k X_k and Y_k = X_k C_k; the next border
                // blocks are -t' times these, and at the last eliminated layer the
                // direct bond t' is added (-t' (Y - 1)).  X leaves the registers
                // meanwhile (they hold S and one product).
                if (o == L - 2)
                    for (int k = nl; k < 2 * ns; k += Tl::LPN) {
                        const int d = ((k & 1) * NS + (k >> 1)) * RS + k;
                        C[d].x -= 1.f;
                        E[d].x -= 1.f;
                    }
                store(X, a, r, c);
                __syncwarp();
                Tile w;
#pragma unroll 1
                for (int q = 0; q < (o < L - 2 ? 3 : 2); ++q) {   // E X -> E, S += t' E C, X C -> C
                    mul(w, q == 2 ? X : E, q == 0 ? X : C, ns, r, c);
                    if (q == 1) {
#pragma unroll
                        for (int i = 0; i < 2 * SR; ++i)
#pragma unroll
                            for (int j = 0; j < 2 * SC; ++j)
                                S[i][j] = make_float2(S[i][j].x + tp * w[i][j].x, S[i][j].y + tp * w[i][j].y);
                    } else {
                        put(q == 0 ? E : C, w, -tp, r, c);
                    }
                }
                load(a, X, r, c);
                __syncwarp();
                continue;
            }
            if (!ring && !(o == L - 2 || (!v.per && o == v.u - 1))) continue;
            // S -= (coupling)^2 X, on real sites; the ring's first layer also
            // starts the border blocks with t' X.
            const float cc = v.per && L == 2 ? 2.f * tp : tp;
#pragma unroll
            for (int i = 0; i < 2 * SR; ++i) {
                const float f = (r + GR * (i % SR)) < ns ? cc : 0.f;
#pragma unroll
                for (int j = 0; j < 2 * SC; ++j) S[i][j] = make_float2(S[i][j].x - f * (f * a[i][j].x), S[i][j].y - f * (f * a[i][j].y));
            }
            if (ring) {
                Tile w;
#pragma unroll
                for (int i = 0; i < 2 * SR; ++i) {
                    const float f = (r + GR * (i % SR)) < ns ? tp : 0.f;
#pragma unroll
                    for (int j = 0; j < 2 * SC; ++j) w[i][j] = make_float2(f * a[i][j].x, f * a[i][j].y);
                }
                store(C, w, r, c);
                store(E, w, r, c);
                __syncwarp();
            }
        }
        finish(a, v.us, s, lnd, th, r, c, nl, out);
    }
};

// ---------------------------------------------------------------------------
// The same elimination by a group of GR x GC threads per node, for the
// double-float re-solve: the next stage waits for it, so the time of one node
// counts.  Thread (r, c) holds rows r + GR i of column c (a row is 2 site + spin);
// one row is pivoted at a time, its row, column and inverse pivot broadcast
// through double-buffered shared memory (one barrier of the group per pivot),
// and nothing is padded.  One column per thread: the scaled pivot row element
// serves all its rows, so that a step is one product and R updates.  (In FP32
// one warp per node is faster: 49 against 66 us for a stage of 16 visits of 8x8
// clusters -- the barriers and the broadcast outweigh the arithmetic.)
// ---------------------------------------------------------------------------
template <int GR_, int GC_, int R_, int DFG_> struct RsGroupShape {
    static constexpr int GR = GR_, GC = GC_, R = R_, C = 1, TPN = GR * GC;
    static constexpr int DFG = DFG_;                              // groups per CTA
    static constexpr int B = GC, RS = B + 1;                      // largest block order, elements per matrix row
    static_assert(GR * R == GC, "square blocks");
};
using RsG8 = RsGroupShape<4, 8, 2, 3>;       // one warp, up to 4 sites per layer
using RsG16 = RsGroupShape<8, 16, 2, 3>;     // four warps, up to 8 sites
using RsG24 = RsGroupShape<8, 24, 3, 2>;     // six warps, 12 sites
using RsG32 = RsGroupShape<8, 32, 4, 2>;     // eight warps, 16 sites

template <typename T, class Gp> struct RsGroup {
    using V = cplx_t<T>;
    static constexpr int GR = Gp::GR, GC = Gp::GC, R = Gp::R, C = Gp::C, RS = Gp::RS;
    using Tile = V[R][C];
    // Shared memory of a group: three matrices, two broadcast buffers of a pivot
    // row and column; the node's pivots follow (bytes() with n of them).
    struct Smem { V X[Gp::B * RS], C[Gp::B * RS], E[Gp::B * RS], row[2][Gp::B], col[2][Gp::B], inv[2]; };
    static __host__ __device__ constexpr size_t bytes(int n) { return sizeof(Smem) + (size_t)n * sizeof(V); }

    static __device__ __forceinline__ void sync(int id) {
        if constexpr (Gp::TPN == 32) __syncwarp();
        else asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(Gp::TPN) : "memory");
    }
    static __device__ __forceinline__ void store(V* M, const Tile& a, T f, int b, int r, int c) {
#pragma unroll
        for (int i = 0; i < R; ++i)
#pragma unroll
            for (int j = 0; j < C; ++j) {
                const int x = r + GR * i, y = c + GC * j;
                if (x < b && y < b) M[x * RS + y] = mk(f * a[i][j].x, f * a[i][j].y);
            }
    }
    static __device__ __forceinline__ void mul(Tile& o, const V* P, const V* Q, int b, int bc, int r, int c) {
#pragma unroll
        for (int i = 0; i < R; ++i)
#pragma unroll
            for (int j = 0; j < C; ++j) o[i][j] = mk(T(0.f), T(0.f));
        // rows and columns past the block read the last one and are not used
#pragma unroll 2
        for (int k = 0; k < b; ++k) {
            V p[R];
#pragma unroll
            for (int i = 0; i < R; ++i) p[i] = P[(r + GR * i < b ? r + GR * i : b - 1) * RS + k];
#pragma unroll
            for (int j = 0; j < C; ++j) {
                const V q = Q[k * RS + (c + GC * j < bc ? c + GC * j : bc - 1)];
#pragma unroll
                for (int i = 0; i < R; ++i) o[i][j] = cfma(p[i], q, o[i][j]);
            }
        }
    }
    // The block of a layer without its i, minus tt X (X in a).
    static __device__ __forceinline__ void layer(Tile& a, const RsSite<T>* site, const T* hop, int hs, T s, T tt, int b,
                                                 int r, int c, bool chain) {
#pragma unroll
        for (int i = 0; i < R; ++i)
#pragma unroll
            for (int j = 0; j < C; ++j) {
                const int x = r + GR * i, y = c + GC * j, sx = x >> 1, sy = y >> 1;
                V e = mk(T(0.f), T(0.f));
                if (x < b && y < b) {
                    if (sx == sy) {
                        const RsSite<T> o = site[sx];
                        if (x == y) e.x = ((x & 1) ? o.d - o.z : o.d + o.z) * s;
                        else { e.x = o.x * s; e.y = (x & 1) ? o.y * s : -(o.y * s); }
                    } else if (((x ^ y) & 1) == 0) {
                        e.x = hop[sx * hs + sy] * s;
                    }
                    if (chain) { e.x = e.x - tt * a[i][j].x; e.y = e.y - tt * a[i][j].y; }
                }
                a[i][j] = e;
            }
    }
    // Gauss-Jordan inversion in place of a + i; rows 2 skip and 2 skip + 1 are
    // left out.  The pivots go to piv (without their i).
    static __device__ __forceinline__ void invert(Tile& a, Smem& sm, V* piv, int skip, int b, int r, int c, int id) {
#pragma unroll 1
        for (int p = 0; p < b; ++p) {
            if ((p >> 1) == skip) continue;
            V* row = sm.row[p & 1];
            V* col = sm.col[p & 1];
            const V zero = mk(T(0.f), T(0.f));
            const bool pc = c == p;
#pragma unroll
            for (int i = 0; i < R; ++i) {
                const int x = r + GR * i;
                if (x == p) {
                    if (c < b) row[c] = a[i][0];
                    if (pc) {
                        const V pv = a[i][0];
                        piv[p] = pv;
                        const T im = pv.y + T(1.f), rq = rs_rcp(pv.x * pv.x + im * im);
                        sm.inv[p & 1] = mk(pv.x * rq, -(im * rq));     // 1/(pivot + i)
                    }
                }
                if (pc && x < b) col[x] = a[i][0];
            }
            sync(id);
            const V w = sm.inv[p & 1];
            const V s = pc ? w : c < b ? cfma(row[c], w, zero) : zero;
#pragma unroll
            for (int i = 0; i < R; ++i) {
                const int x = r + GR * i;
                const V q = x < b ? col[x] : zero;
                a[i][0] = x == p ? s : cfms(q, s, pc ? zero : a[i][0]);
            }
        }
    }

    static __device__ __forceinline__ void run(const RsVisit& v, const RsSite<T>* site, const T* hop, int hs, T s, T tp,
                                               Smem& sm, int t, int id, RsOut<T>* out) {
        V* const piv = reinterpret_cast<V*>(&sm + 1);
        const int r = t / GC, c = t % GC, L = v.L, ns = v.ns, b = 2 * ns;
        const bool ring = v.per && L >= 3;
        const T tt = tp * tp, tau2 = (v.per && L == 2) ? T(4.f) * tt : tt, one = T(1.f);
        Tile a, S;
        RsSum<T> lnd, th;
        layer(S, site + v.u * ns, hop, hs, s, tt, b, r, c, false);
#pragma unroll 1
        for (int o = 0; o < L; ++o) {
            const bool last = o == L - 1;
            if (last) {
#pragma unroll
                for (int i = 0; i < R; ++i)
#pragma unroll
                    for (int j = 0; j < C; ++j) a[i][j] = S[i][j];
            } else {
                int l;
                if (v.per) { l = v.u + 1 + o; if (l >= L) l -= L; }
                else l = o < v.u ? o : L - 1 - (o - v.u);
                layer(a, site + l * ns, hop, hs, s, tt, b, r, c, o > 0 && (v.per || o != v.u));
            }
            invert(a, sm, piv + o * b, last ? v.us : -1, b, r, c, id);
            if (last) break;
            sync(id);
            if (ring && o > 0) {
                if (o == L - 2 && t < b) {
                    sm.C[t * RS + t].x = sm.C[t * RS + t].x - one;
                    sm.E[t * RS + t].x = sm.E[t * RS + t].x - one;
                }
                store(sm.X, a, one, b, r, c);
                sync(id);
                Tile w;
                mul(w, sm.E, sm.X, b, b, r, c);
                sync(id);
                store(sm.E, w, -tp, b, r, c);
                sync(id);
                mul(w, sm.E, sm.C, b, b, r, c);
#pragma unroll
                for (int i = 0; i < R; ++i)
#pragma unroll
                    for (int j = 0; j < C; ++j) S[i][j] = mk(S[i][j].x + tp * w[i][j].x, S[i][j].y + tp * w[i][j].y);
                if (o < L - 2) {
                    mul(w, sm.X, sm.C, b, b, r, c);
                    sync(id);
                    store(sm.C, w, -tp, b, r, c);
                }
                sync(id);
                continue;
            }
            if (!ring && !(o == L - 2 || (!v.per && o == v.u - 1))) continue;
            const T cc = ring ? tt : tau2;
#pragma unroll
            for (int i = 0; i < R; ++i)
#pragma unroll
                for (int j = 0; j < C; ++j) S[i][j] = mk(S[i][j].x - cc * a[i][j].x, S[i][j].y - cc * a[i][j].y);
            if (ring) {
                store(sm.C, a, tp, b, r, c);
                store(sm.E, a, tp, b, r, c);
                sync(id);
            }
        }
        finish(a, sm, piv, b * L, b * (L - 1) + 2 * v.us, v.us, s, lnd, th, r, c, t, id, out);
    }

    // o = P^t Q with P^t the block transpose of P (2x2 blocks stay as they are)
    static __device__ __forceinline__ void mul_t(Tile& o, const V* P, const V* Q, int b, int nrow, int r, int c) {
#pragma unroll
        for (int i = 0; i < R; ++i)
#pragma unroll
            for (int j = 0; j < C; ++j) o[i][j] = mk(T(0.f), T(0.f));
#pragma unroll 2
        for (int k = 0; k < b; ++k) {
            V p[R];
#pragma unroll
            for (int i = 0; i < R; ++i) {
                const int x = r + GR * i < nrow ? r + GR * i : nrow - 1;
                p[i] = P[((k & ~1) + (x & 1)) * RS + (x & ~1) + (k & 1)];
            }
#pragma unroll
            for (int j = 0; j < C; ++j) {
                const V q = Q[k * RS + (c + GC * j < nrow ? c + GC * j : nrow - 1)];
#pragma unroll
                for (int i = 0; i < R; ++i) o[i][j] = cfma(p[i], q, o[i][j]);
            }
        }
    }
    // Block of the kept sites' matrix after the eliminated parity (RsNode::pair_block).
    static __device__ __forceinline__ void pair_block(Tile& a, const RsPairs& pt, int row0, int nr, int col0, int nc,
                                                      const RsSite<T>* site, const V* inv, T s, T tt, int r, int c) {
#pragma unroll
        for (int i = 0; i < R; ++i)
#pragma unroll
            for (int j = 0; j < C; ++j) {
                const int x = r + GR * i, y = c + GC * j, sx = x >> 1, sy = y >> 1;
                V e = mk(T(0.f), T(0.f));
                if (sx < nr && sy < nc) {
                    uint32_t both = pt.near[row0 + sx] & pt.near[col0 + sy];
                    const int q = 2 * (x & 1) + (y & 1);
                    while (both) {
                        const int k = __ffs(both) - 1;
                        both &= both - 1;
                        e = csub(e, inv[4 * k + q]);
                    }
                    e = mk(tt * e.x, tt * e.y);
                    if (row0 + sx == col0 + sy) {
                        const RsSite<T> o = site[pt.kept[row0 + sx]];
                        if (x == y) e.x = e.x + ((x & 1) ? o.d - o.z : o.d + o.z) * s;
                        else { e.x = e.x + o.x * s; e.y = e.y + ((x & 1) ? o.y * s : -(o.y * s)); }
                    }
                }
                a[i][j] = e;
            }
    }
    // run() for a window split by parity.
    static __device__ __forceinline__ void run_pairs(const RsPairs& pt, const RsSite<T>* site, T s, T tp, Smem& sm, int t,
                                                     int id, RsOut<T>* out) {
        V* const piv = reinterpret_cast<V*>(&sm + 1);
        const int r = t / GC, c = t % GC;
        const T tt = tp * tp, one = T(1.f);
        V* const inv = sm.E;
        RsSum<T> lnd, th;
        for (int e = t; e < pt.ne; e += Gp::TPN) {
            const RsSite<T> o = site[pt.gone[e]];
            const V zero = mk(T(0.f), T(0.f));
            const V p00 = mk((o.d + o.z) * s, T(0.f)), p11 = mk((o.d - o.z) * s, T(0.f));
            const V p01 = mk(o.x * s, -(o.y * s)), p10 = mk(o.x * s, o.y * s);
            const V g = rs_det_g(p00, p01, p10, p11);
            const T gr = one + g.x, rq = rs_rcp(gr * gr + g.y * g.y);
            const V w = mk(-(gr * rq), g.y * rq);
            inv[4 * e] = cfma(mk(p11.x, one), w, zero);
            inv[4 * e + 1] = cfms(p01, w, zero);
            inv[4 * e + 2] = cfms(p10, w, zero);
            inv[4 * e + 3] = cfma(mk(p00.x, one), w, zero);
            lnd.add(rs_log1p((g.x + g.x) + (g.x * g.x + g.y * g.y)));
            th.add(rs_phase(g.y, one + g.x));
        }
        sync(id);
        Tile a, S;
        const int ba = 2 * pt.na, bb = 2 * pt.nb;
        pair_block(a, pt, 0, pt.na, 0, pt.na, site, inv, s, tt, r, c);
#pragma unroll 1
        for (int o = 0;; ++o) {
            invert(a, sm, piv + (o ? ba : 0), o ? pt.nb - 1 : -1, o ? bb : ba, r, c, id);
            if (o) break;
            store(sm.X, a, one, ba, r, c);
            pair_block(a, pt, 0, pt.na, pt.na, pt.nb, site, inv, s, tt, r, c);
#pragma unroll
            for (int i = 0; i < R; ++i)
#pragma unroll
                for (int j = 0; j < C; ++j)
                    if (r + GR * i < ba && c + GC * j < bb) sm.C[(r + GR * i) * RS + c + GC * j] = a[i][j];
            pair_block(S, pt, pt.na, pt.nb, pt.na, pt.nb, site, inv, s, tt, r, c);
            sync(id);
            mul(a, sm.X, sm.C, ba, bb, r, c);
            sync(id);
#pragma unroll
            for (int i = 0; i < R; ++i)
#pragma unroll
                for (int j = 0; j < C; ++j)
                    if (r + GR * i < ba && c + GC * j < bb) sm.X[(r + GR * i) * RS + c + GC * j] = a[i][j];
            sync(id);
            mul_t(a, sm.C, sm.X, ba, bb, r, c);
#pragma unroll
            for (int i = 0; i < R; ++i)
#pragma unroll
                for (int j = 0; j < C; ++j) a[i][j] = csub(S[i][j], a[i][j]);
            sync(id);
        }
        finish(a, sm, piv, ba + bb, ba + bb - 2, pt.nb - 1, s, lnd, th, r, c, t, id, out);
    }

    // Results of a node: the last pivot block, and the sums over the np pivots
    // but the update site's two, on top of what lnd and th hold already.
    static __device__ __forceinline__ void finish(const Tile& a, Smem& sm, const V* piv, int np, int skip, int us, T s, RsSum<T>& lnd,
                                                  RsSum<T>& th, int r, int c, int t, int id, RsOut<T>* out) {
        const T one = T(1.f);
#pragma unroll
        for (int i = 0; i < R; ++i)
#pragma unroll
            for (int j = 0; j < C; ++j) {
                const int x = r + GR * i, y = c + GC * j;
                if ((x >> 1) == us && (y >> 1) == us) {
                    const int k = 4 * (x & 1) + 2 * (y & 1);
                    out->P[k] = a[i][j].x;
                    out->P[k + 1] = a[i][j].y;
                }
            }
        sync(id);
        // Logarithm and phase of two pivots at a time (their product against i^2
        // has a phase within (-pi, pi)), all at the end: FP64 logarithms of a few
        // lanes after each layer took longer than the eliminations of a chain.
        for (int p = 2 * t; p < np; p += 2 * Gp::TPN) {
            if (p == skip) continue;
            const V u = piv[p], w = piv[p + 1];
            // (1 - i u)(1 - i w) = 1 + g
            const V g = mk(u.y + w.y - (u.x * w.x - u.y * w.y), -(u.x + w.x) - (u.x * w.y + u.y * w.x));
            lnd.add(rs_log1p((g.x + g.x) + (g.x * g.x + g.y * g.y)));
            th.add(rs_phase(g.y, one + g.x));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) { lnd.merge(o); th.merge(o); }
        double2* part = reinterpret_cast<double2*>(sm.row[0]);   // per-warp partial sums
        if (Gp::TPN > 32) sync(id);
        if ((t & 31) == 0) part[t >> 5] = make_double2(lnd.value(), th.value());
        sync(id);
        if (t == 0) {
            double l = part[0].x, h = part[0].y;
            for (int k = 1; k < Gp::TPN / 32; ++k) { l += part[k].x; h += part[k].y; }
            out->lnd = 0.5 * l;
            out->th = h;
            out->s = s;
        }
        sync(id);
    }
};

// ---------------------------------------------------------------------------
// A CTA's share of a stage: up to VB visits.  Shared memory (byte offsets):
// the visits' headers, FP64 terms, node results, window sites, in-layer
// hopping, and one set of block buffers per concurrently eliminated node.
// ---------------------------------------------------------------------------
struct RsLayout { size_t terms, out, site, hop, buf, total; };

// kOut: nodes kept per visit.  One hopping table when all windows have one shape.
template <class Tl>
__host__ __device__ inline RsLayout rs_layout(int vb, int max_sites, int nw, bool uniform, bool pairs) {
    RsLayout L;
    size_t o = align16((size_t)vb * sizeof(RsVisit)) + (pairs ? align16(sizeof(RsPairs)) : 0);
    L.terms = o; o = align16(o + (size_t)vb * sizeof(RsTerms));
    L.out = o;   o = align16(o + (size_t)vb * kFermiOut * sizeof(RsOut<float>));
    L.site = o;  o = align16(o + (size_t)vb * max_sites * sizeof(RsSite<float>));
    L.hop = o;   o = align16(o + (size_t)(uniform ? 1 : vb) * Tl::NS * Tl::NS * sizeof(float));
    L.buf = o;   o = align16(o + (size_t)nw * Tl::NPW * Tl::node(pairs) * sizeof(float2));
    L.total = o;
    return L;
}

static __constant__ float c_fermi_x[kFermiClasses] = {PTCA_FERMI_X};
static __constant__ FermiNodes c_fermi[kFermiClasses] = {PTCA_FERMI_NODES};
static __constant__ FermiNodes c_fermi_df[kFermiClasses] = {PTCA_FERMI_NODES_DF};
static __constant__ FermiSlopes c_slope = fermi_slopes();

// The nodes of an arithmetic: their approximation error is below its rounding.
template <typename T> struct RsFermi {
    static __device__ __forceinline__ const FermiNodes& tab(int cls) { return sizeof(T) == 4 ? c_fermi[cls] : c_fermi_df[cls]; }
};

// A window in layer order: layers along its longest axis (a layer then has the
// fewest sites), e0 x e1 sites each; window site k is site k % ns of layer k / ns.
struct RsFrame {
    Window win;
    int ax, L, e0, e1, ns, u, us;   // u, us: layer and in-layer index of the update site
    __device__ __forceinline__ int site(const Model& m, int k) const {
        const int l = k / ns, q = k % ns, q0 = q % e0, q1 = q / e0;
        return window_site(m, win, ax == 0 ? l : q0, ax == 1 ? l : (ax == 0 ? q0 : q1), ax == 2 ? l : q1);
    }
};
__device__ __forceinline__ RsFrame rs_frame(const Model& m, int site) {
    RsFrame f;
    f.win = make_window(m, site);
    const Window& w = f.win;
    f.ax = w.ez > max(w.ex, w.ey) ? 2 : w.ey > w.ex ? 1 : 0;
    f.L = f.ax == 0 ? w.ex : f.ax == 1 ? w.ey : w.ez;
    f.e0 = f.ax == 0 ? w.ey : w.ex;                 // the other axes, in order
    f.e1 = f.ax == 2 ? w.ey : w.ez;
    f.ns = f.e0 * f.e1;
    f.u = f.ax == 0 ? w.uwx : f.ax == 1 ? w.uwy : w.uwz;
    f.us = (f.ax == 2 ? w.uwy : w.uwz) * f.e0 + (f.ax == 0 ? w.uwy : w.uwx);
    return f;
}

// Tr x, Tr x^2 (on-site sums x1, x2 plus the hopping) and the classical energy.
__device__ __forceinline__ void rs_terms_out(const StageArgs& a, const RsFrame& f, double x1, double x2, double cl, RsTerms& w) {
    const int per = a.m.cluster_periodic, nsite = f.ns * f.L;
    int pairs = 0;
    for (int e : {f.L, f.e0, f.e1}) pairs += e < 2 ? 0 : nsite / e * (per ? (e == 2 ? 4 : e) : e - 1);
    w.x1 = x1 * a.unit.T1;
    w.x2 = (x2 + 4.0 * a.unit.t * a.unit.t * (double)pairs) * a.unit.T1 * a.unit.T1;
    w.cl = cl;
}

// A visit's window, gathered by GL lanes of a warp: the on-site terms, the node
// class from Gershgorin's bound on |mu - H|, and (kTerms) rs_terms.
template <typename T, int GL, bool kTerms>
__device__ __forceinline__ void rs_gather(const StageArgs& a, const double* S, int c, int site, RsVisit& h, RsTerms& w,
                                          RsSite<T>* sites, int gl) {
    const Model& m = a.m;
    const RsFrame f = rs_frame(m, site);
    const int nsite = f.ns * f.L, per = m.cluster_periodic;
    const RsUnit& u = a.unit;
    double x1 = 0.0, x2 = 0.0, cl = 0.0;
    float bound = 0.f;
    for (int k = gl; k < nsite; k += GL) {
        const double* v = S + 3 * (int64_t)f.site(m, k);
        const double v0 = v[0], v1 = v[1], v2 = v[2], d = u.mu - u.lam * v0;
        sites[k].d = T(d); sites[k].x = T(u.J * v0); sites[k].y = T(u.J * v1); sites[k].z = T(u.J * v2);
        if constexpr (kTerms) {
            const double m2 = v0 * v0 + v1 * v1 + v2 * v2;
            x1 -= 2.0 * d;
            x2 += 2.0 * (d * d + u.J * u.J * m2);
            if (m.cls_on) cl += m.ca * m2 + m.cb * v0 + m.cc;
        }
        const float g0 = (float)v0, g1 = (float)v1, g2 = (float)v2;
        bound = fmaxf(bound, fabsf((float)d) + fabsf((float)u.J) * sqrtf(g0 * g0 + g1 * g1 + g2 * g2));
    }
#pragma unroll
    for (int o = GL / 2; o > 0; o >>= 1) {
        if constexpr (kTerms) {
            x1 += __shfl_xor_sync(FULL_MASK, x1, o);
            x2 += __shfl_xor_sync(FULL_MASK, x2, o);
            if (m.cls_on) cl += __shfl_xor_sync(FULL_MASK, cl, o);
        }
        bound = fmaxf(bound, __shfl_xor_sync(FULL_MASK, bound, o));
    }
    if (gl == 0) {
        float deg = 0.f;
        for (int e : {f.L, f.e0, f.e1}) deg += e < 2 ? 0.f : e == 2 && !per ? 1.f : 2.f;
        const float X = (bound + deg * fabsf((float)u.t)) * (float)u.T1 * (1.f + 1e-6f);
        int cls = 0;
        while (cls < kFermiClasses && !(X <= c_fermi_x[cls])) ++cls;
        h.c = c; h.site = site; h.n = 2 * nsite; h.L = f.L; h.ns = f.ns; h.per = per;
        h.u = f.u;
        h.us = f.us;
        h.cls = cls < kFermiClasses ? cls : -1;
        if constexpr (kTerms) rs_terms_out(a, f, x1, x2, cl, w);
    }
}

// rs_terms_out of a window, by one warp.
__device__ __forceinline__ void rs_terms(const StageArgs& a, const double* S, int site, RsTerms& w, int lane) {
    const Model& m = a.m;
    const RsFrame f = rs_frame(m, site);
    const RsUnit& u = a.unit;
    double x1 = 0.0, x2 = 0.0, cl = 0.0;
    for (int k = lane; k < f.ns * f.L; k += 32) {
        const double* v = S + 3 * (int64_t)f.site(m, k);
        const double v0 = v[0], d = u.mu - u.lam * v0, m2 = v0 * v0 + v[1] * v[1] + v[2] * v[2];
        x1 -= 2.0 * d;
        x2 += 2.0 * (d * d + u.J * u.J * m2);
        if (m.cls_on) cl += m.ca * m2 + m.cb * v0 + m.cc;
    }
    x1 = warp_sum(x1);
    x2 = warp_sum(x2);
    if (m.cls_on) cl = warp_sum(cl);
    if (lane == 0) rs_terms_out(a, f, x1, x2, cl, w);
}

// The proposal and ln u of a visit (one thread): drawn here, or from the sweep's
// table where the caller drew them all at once.
__device__ __forceinline__ void rs_proposal(const StageArgs& a, const StageVar& v, int site, RsTerms& w) {
    if (a.prop) {
        const double4 p = a.prop[site];
        w.sn[0] = p.x; w.sn[1] = p.y; w.sn[2] = p.z;
        w.lnu = p.w;
        return;
    }
    double u0, u1;
    propose(a.m, v.sweep, (uint32_t)site, v.S_in + 3 * (int64_t)site, w.sn);
    uniform2(a.m.seed, v.sweep, (uint32_t)site, RNG_ACCEPT, u0, u1);
    w.lnu = log(u0);
}

// In-layer hopping of a window between sites i and j of a layer, at [i hs + j]
// (an axis of extent 2 of a periodic cluster has two bonds), by one warp.
template <typename T> __device__ __forceinline__ void rs_hopping(const StageArgs& a, int site, T* hop, int hs, int lane) {
    const Model& m = a.m;
    const RsFrame f = rs_frame(m, site);
    const int e0 = f.e0, e1 = f.e1, ns = f.ns, per = m.cluster_periodic;
    for (int k = lane; k < hs * hs; k += 32) {
        const int i = k / hs, j = k % hs;
        double bonds = 0.0;
        if (i < ns && j < ns) {
            const int d0 = abs(i % e0 - j % e0), d1 = abs(i / e0 - j / e0);
            if (d1 == 0 && d0 > 0) bonds = (d0 == 1) + (per && d0 == e0 - 1);
            if (d0 == 0 && d1 > 0) bonds = (d1 == 1) + (per && d1 == e1 - 1);
        }
        hop[k] = T(a.unit.t * bonds);
    }
}

// The parity split of a periodic lattice's windows (all alike), by one warp.
// Window sites in layer order, as rs_gather places them.
__device__ __forceinline__ void rs_pairs(const Model& m, int site, RsPairs& t, int lane) {
    const RsFrame f = rs_frame(m, site);
    const int e0 = f.e0, e1 = f.e1, e2 = f.L, ns = f.ns, n = ns * e2, per = m.cluster_periodic, u = f.u * ns + f.us;
    // coordinates of a window site, packed (8 bits each); parity; bonds
    auto place = [&](int k) { return (uint32_t)(k % e0) | (uint32_t)(k / e0 % e1) << 8 | (uint32_t)(k / ns) << 16; };
    auto parity = [&](int k) {
        const uint32_t x = place(k);
        return (int)((x ^ (x >> 8) ^ (x >> 16)) & 1u);
    };
    auto next = [&](int d, int e) { return d == 1 || (per && d == e - 1); };
    auto bond = [&](uint32_t x, uint32_t y) {
        const int d0 = abs((int)(x & 255) - (int)(y & 255)), d1 = abs((int)(x >> 8 & 255) - (int)(y >> 8 & 255)),
                  d2 = abs((int)(x >> 16) - (int)(y >> 16));
        return (d0 && !d1 && !d2 && next(d0, e0)) || (!d0 && d1 && !d2 && next(d1, e1)) || (!d0 && !d1 && d2 && next(d2, e2));
    };
    const int pu = parity(u);
    // kept and eliminated sites in order, the update site last
    int nk = 0, ne = 0;
    for (int k0 = 0; k0 < n; k0 += 32) {
        const int k = k0 + lane;
        const bool in = k < n, keep = in && k != u && parity(k) == pu, drop = in && parity(k) != pu;
        const unsigned bk = __ballot_sync(FULL_MASK, keep), bd = __ballot_sync(FULL_MASK, drop), below = (1u << lane) - 1u;
        if (keep) t.kept[nk + __popc(bk & below)] = k;
        if (drop) {
            t.gone[ne + __popc(bd & below)] = k;
            t.place[ne + __popc(bd & below)] = place(k);
        }
        nk += __popc(bk);
        ne += __popc(bd);
    }
    if (lane == 0) {
        t.kept[nk] = u;
        t.na = (nk + 1) / 2;
        t.nb = nk + 1 - t.na;
        t.ne = ne;
    }
    __syncwarp();
    if (lane <= nk) {
        const uint32_t x = place(t.kept[lane]);
        uint32_t near = 0;
        for (int e = 0; e < ne; ++e) near |= (uint32_t)bond(x, t.place[e]) << e;
        t.near[lane] = near;
    }
}

// What a visit's free energies are for: the stage's decision, with decisions
// near the threshold left to the re-solve; the re-solve's decision; or the
// precision checker, which takes the two free energies alone (Fbuf[2c],
// Fbuf[2c + 1]).
enum RsMode : int { RS_STAGE, RS_RESOLVE, RS_CHECK };

// Metropolis on dF and the visit's records (one thread).  fine: the free
// energies are valid (the window lies within the node classes).
__device__ __forceinline__ void rs_commit(RsMode mode, const StageArgs& a, const StageVar& v, const RsVisit& h,
                                          const RsTerms& w, bool fine, double Fo, double dF, double fo, double fn) {
    const Model& m = a.m;
    const double Fn = Fo + dF;
    const double* so = v.S_in + 3 * (int64_t)h.site;
    const int c = h.c, site = h.site;
    if (mode == RS_CHECK) {
        if (fine) { a.Fbuf[2 * c] = Fo; a.Fbuf[2 * c + 1] = Fn; }
        return;
    }
    if (fine && !isfinite(dF)) atomicExch(a.err, 1);
    const double dFe = stage2_dF(a, c, dF);
    if (mode == RS_STAGE) {
        // near the threshold, or a window beyond the last node class
        if (!fine || (a.margin > 0.0 && fabs(w.lnu + dFe * a.invT) < a.margin)) {
            a.flag_list[atomicAdd(a.flag_count, 1u)] = c;
            atomicAdd(&a.counters[2], 1ull);
            return;
        }
    }
    const bool acc = w.lnu < -dFe * a.invT;
    if (a.sg_feat) collect_sample(a, v.S_in, make_window(m, site), v.rec_base + c, w.sn, dF);
    double* dst = v.S_out + 3 * (int64_t)site;
#pragma unroll
    for (int k = 0; k < 3; ++k) dst[k] = acc ? w.sn[k] : so[k];
    const int r = v.rec_base + c;
    a.rec_site[r] = site;
    a.rec_Fold[r] = Fo;
    a.rec_Fnew[r] = Fn;
    a.rec_lnu[r] = w.lnu;
    a.rec_acc[r] = acc ? 1 : 0;
    a.rec_Facc[r] = acc ? Fn : Fo;
    a.rec_fill[r] = acc ? fn : fo;
    a.rec_n[r] = h.n;
    if (acc) atomicAdd(&a.counters[0], 1ull);
    atomicAdd(&a.counters[1], 2ull);
}

// A node's results, past the L1 (another SM may have written them).
template <typename T> __device__ __forceinline__ void rs_load(RsOut<T>& r, const RsOut<T>* p) {
    const volatile RsOut<T>* q = p;
    r.lnd = q->lnd;
    r.th = q->th;
#pragma unroll
    for (int k = 0; k < 8; ++k) rs_get(r.P[k], &q->P[k]);
    rs_get(r.s, &q->s);
    r.eta = q->eta;
}

// The last pivot of a node: lq = ln|det| and t0 = phase (against i^2) of the
// update site's block, and dl, dt their changes under the proposal, which adds
// [[dd + jz, jx - i jy], [jx + i jy, dd - jz]] (times s already) to the block.
template <typename T, typename L>
__device__ __forceinline__ void rs_last_pivot(const RsOut<T>& r, T dd, T jx, T jy, T jz, L& lq, L& t0, L& dl, L& dt) {
    const auto p00 = mk(r.P[0], r.P[1]), p01 = mk(r.P[2], r.P[3]), p10 = mk(r.P[4], r.P[5]), p11 = mk(r.P[6], r.P[7]);
    const auto g = rs_det_g(p00, p01, p10, p11);
    const auto gn = rs_det_g(mk(p00.x + dd + jz, p00.y), mk(p01.x + jx, p01.y - jy), mk(p10.x + jx, p10.y + jy),
                             mk(p11.x + dd - jz, p11.y));
    const T q = (g.x + g.x) + (g.x * g.x + g.y * g.y), qn = (gn.x + gn.x) + (gn.x * gn.x + gn.y * gn.y);
    // det_new / det_old = 1 + z, with det_new - det_old formed from the
    // change of the block (no cancellation between the two determinants)
    const auto zero = mk(T(0.f), T(0.f));
    const T ax = dd + jz, bx = dd - jz;
    auto num = cfma(p11, mk(ax, T(0.f)), cfma(p00, mk(bx, T(0.f)), zero));
    num = cfms(p01, mk(jx, jy), num);
    num = cfms(p10, mk(jx, -jy), num);
    // (P + i): the i of the two diagonal entries; minus det of the change
    num = mk(num.x + ax * bx - (jx * jx + jy * jy), num.y + ax + bx);
    const T gr = T(1.f) + g.x, rq = rs_rcp(gr * gr + g.y * g.y);
    // z = num / det_old, det_old = -(1 + g)
    const auto z = cfms(num, mk(gr * rq, -(g.y * rq)), zero);
    const T zq = (z.x + z.x) + (z.x * z.x + z.y * z.y);
    const L l0 = rs_log1p(q), half = (L)0.5;
    lq = half * l0;
    dl = zq < T(1.f) && T(-0.5f) < zq ? half * rs_log1p(zq) : half * (rs_log1p(qn) - l0);
    t0 = rs_phase(g.y, T(1.f) + g.x);
    dt = rs_phase(gn.y, T(1.f) + gn.x) - t0;
}

// Free energies, filling and decision of a visit (one thread) from its weighted
// sums over the nodes: ln|det| and phases of the old matrix, and their changes.
__device__ __forceinline__ void rs_final(RsMode mode, const StageArgs& a, const StageVar& v, const RsVisit& h, const RsTerms& w,
                                         const FermiNodes& f, double Lo, double Th, double dL, double dT) {
    const Model& m = a.m;
    const double* so = v.S_in + 3 * (int64_t)h.site;
    const bool fine = h.cls >= 0;
    const double invT = a.invT, dx = w.sn[0] - so[0];
    // |v|^2 of the site, new minus old
    const double dn = (w.sn[0] - so[0]) * (w.sn[0] + so[0]) + (w.sn[1] - so[1]) * (w.sn[1] + so[1]) +
                      (w.sn[2] - so[2]) * (w.sn[2] + so[2]);
    const double dx1 = 2.0 * m.lam * dx * invT;
    // d(d^2 + J^2 |v|^2) of the site's two rows, d = mu - e0 - lam v_x
    const double mus = m.mu - m.e0, d0 = mus - m.lam * so[0], d1 = mus - m.lam * w.sn[0];
    const double dx2 = 2.0 * ((d1 - d0) * (d1 + d0) + m.JH * m.JH * dn) * invT * invT;
    const double Fo = -m.T * (h.n * (0.69314718055994530942 + f.c) + 0.5 * f.e * w.x2 + Lo - 0.5 * w.x1) + w.cl;
    double dF = -m.T * (0.5 * f.e * dx2 + dL - 0.5 * dx1);
    if (m.cls_on) dF += m.ca * dn + m.cb * dx;
    const double fo = 0.5 * h.n - Th;
    rs_commit(mode, a, v, h, w, fine, Fo, dF, fo, fo - dT);
}

// One visit by one warp, lane = node.
template <typename T>
__device__ __forceinline__ void rs_decide(RsMode mode, const StageArgs& a, const StageVar& v, const RsVisit& h, const RsTerms& w,
                                          const RsOut<T>* out, int lane) {
    const RsUnit& u = a.unit;
    const double* so = v.S_in + 3 * (int64_t)h.site;
    const FermiNodes& f = RsFermi<T>::tab(h.cls >= 0 ? h.cls : 0);
    double Lo = 0.0, Th = 0.0, dL = 0.0, dT = 0.0;
    float ln = 0.f, th = 0.f, dln = 0.f, dth = 0.f, eta = 0.f;   // FP32: logarithm, phase, changes, rounding of the scale
    if (h.cls >= 0 && lane < f.M) {
        RsOut<T> r;
        rs_load(r, out + lane);
        const T dd = T(-u.lam * (w.sn[0] - so[0])) * r.s, jx = T(u.J * (w.sn[0] - so[0])) * r.s,
                jy = T(u.J * (w.sn[1] - so[1])) * r.s, jz = T(u.J * (w.sn[2] - so[2])) * r.s;
        decltype(rs_log1p(r.s)) lq, t0, dl, dt;
        rs_last_pivot(r, dd, jx, jy, jz, lq, t0, dl, dt);
        Lo = f.a[lane] * (r.lnd + (double)lq);
        Th = f.b[lane] * (r.th + (double)t0);
        dL = f.a[lane] * (double)dl;
        dT = f.b[lane] * (double)dt;
        if constexpr (sizeof(T) == 4) {
            ln = (float)r.lnd + (float)lq;
            th = (float)r.th + (float)t0;
            dln = (float)dl;
            dth = (float)dt;
            eta = r.eta;
        }
    }
    if constexpr (sizeof(T) == 4) {
        const int mid = fermi_middle(lane, f.M);
        const FermiSlope& w = c_slope.of[h.cls >= 0 ? h.cls : 0][lane < f.M ? lane : 0];
        float cl = 0.f, ct = 0.f, cdl = 0.f, cdt = 0.f;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            cl += w.a[i] * __shfl_sync(FULL_MASK, ln, mid + i - 1);
            ct += w.b[i] * __shfl_sync(FULL_MASK, th, mid + i - 1);
            cdl += w.a[i] * __shfl_sync(FULL_MASK, dln, mid + i - 1);
            cdt += w.b[i] * __shfl_sync(FULL_MASK, dth, mid + i - 1);
        }
        Lo += (double)(eta * cl);
        Th += (double)(eta * ct);
        dL += (double)(eta * cdl);
        dT += (double)(eta * cdt);
    }
    Lo = warp_sum(Lo);
    Th = warp_sum(Th);
    dL = warp_sum(dL);
    dT = warp_sum(dT);
    if (lane == 0) rs_final(mode, a, v, h, w, f, Lo, Th, dL, dT);
}

// A window beyond the last node class (fields thousands of T long): both
// matrices reduced and solved in FP64 by the CTA, the matrix in its global
// re-solve slot.  Reached only by configurations that a caller sets far from
// any the chain visits, so plain: one thread per row, no blocking.
inline size_t rs_exact_bytes(int n) { return (size_t)n * 48 + ((size_t)n * 12 > 512 ? (size_t)n * 12 : 512); }
static __device__ __noinline__ void rs_exact(const StageArgs& a, const StageVar& v, const RsVisit& h, RsTerms& w, int slot,
                                      unsigned char* smem) {
    const int n = h.n, tid = threadIdx.x, nt = blockDim.x;
    double2* vk = reinterpret_cast<double2*>(smem);
    double2* p = vk + n;
    double* d = reinterpret_cast<double*>(p + n);
    double* e2 = d + n;
    double* sp = e2 + n;                // window spins (12 n bytes); later the block sums
    double2* A = a.gA + (int64_t)slot * a.gA_stride;
    const Model& m = a.m;
    const Window win = make_window(m, h.site);
    double F[2], fill[2];
    for (int var = 0; var < 2; ++var) {
        __syncthreads();
        build_cluster<double>(m, win, v.S_in, var ? w.sn : nullptr, sp, A);
        __syncthreads();
        const double cl = window_classical(m, sp, n / 2);
        __syncthreads();
        for (int k = 0; k < n; ++k) {
            const int q = n - 1 - k;     // order of the trailing block
            double s = 0.0;
            for (int i = tid; i < q; i += nt) {
                vk[i] = A[tri(k + 1 + i) + k];
                s += cabs2(vk[i]);
            }
            __syncthreads();
            const double s2 = block_sum<double>(s, sp);
            if (tid == 0) {
                d[k] = A[tri(k) + k].x;
                if (q > 0) e2[k] = s2;
            }
            if (q < 2 || !(s2 > 0.0)) { __syncthreads(); continue; }
            double2 first;
            double tau;
            reflector_head<double>(s2, vk[0], first, tau);
            __syncthreads();
            if (tid == 0) vk[0] = first;
            __syncthreads();
            s = 0.0;
            for (int i = tid; i < q; i += nt) {
                double2 r = make_double2(0.0, 0.0);
                for (int j = 0; j < q; ++j) {
                    if (j <= i) r = cfma(A[tri(k + 1 + i) + k + 1 + j], vk[j], r);
                    else r = cfma_conj_a(A[tri(k + 1 + j) + k + 1 + i], vk[j], r);
                }
                r.x *= tau; r.y *= tau;
                p[i] = r;
                s += vk[i].x * r.x + vk[i].y * r.y;
            }
            const double K = 0.5 * tau * block_sum<double>(s, sp + 32);
            for (int i = tid; i < q; i += nt) p[i] = make_double2(p[i].x - K * vk[i].x, p[i].y - K * vk[i].y);
            __syncthreads();
            for (int i = tid; i < q; i += nt)
                for (int j = 0; j <= i; ++j) {
                    double2& x = A[tri(k + 1 + i) + k + 1 + j];
                    x = cfms_conj_b(p[i], vk[j], cfms_conj_b(vk[i], p[j], x));
                }
            __syncthreads();
        }
        __syncthreads();
        double lo = 1e300, hi = -1e300, em = 0.0;
        for (int i = 0; i < n; ++i) {
            const double el = i > 0 ? sqrt(e2[i - 1]) : 0.0, er = i < n - 1 ? sqrt(e2[i]) : 0.0;
            lo = fmin(lo, d[i] - el - er);
            hi = fmax(hi, d[i] + el + er);
            if (i < n - 1) em = fmax(em, e2[i]);
        }
        const double nrm = fmax(fabs(lo), fabs(hi)), pad = 1e-12 * (hi - lo + nrm) + 1e-300;
        double sf = 0.0, sn = 0.0;
        for (int k = tid; k < n; k += nt) {
            const double lam = eig_f64(n, d, e2, k, lo - pad, hi + pad, DBL_MIN * fmax(1.0, em), nrm);
            const double x = -(lam - (m.mu - m.e0)) / m.T;
            sf += softplus(x);
            sn += 1.0 / (1.0 + exp(-x));
        }
        __syncthreads();
        F[var] = -m.T * block_sum<double>(sf, sp) + cl;
        fill[var] = block_sum<double>(sn, sp + 32);
        __syncthreads();
    }
    if (tid == 0) rs_commit(RS_RESOLVE, a, v, h, w, true, F[0], F[1] - F[0], fill[0], fill[1]);
    __syncthreads();
}

// Relative rounding error of s > 0 as a float; none where that is zero or below the
// normal floats (T above 1e36 |t|: levels and phases are then zero as well), where the
// quotient would be 0 / 0.
__device__ __forceinline__ float rs_rounding(double s) {
    const float f = (float)s;
    return f > 1e-37f ? __fdividef((float)((double)f - s), f) : 0.f;
}

// Visits [first, first + nv) of the work list (nv <= vb <= 32), by the CTA.
// uniform: all windows have one shape (periodic lattices), so that a warp may
// hold nodes of several visits.  kPairs: windows split by parity (uniform).
template <class Tl, bool kPairs>
__device__ __forceinline__ void rs_visits(RsMode mode, const StageArgs& a, const StageVar& v, const int32_t* list, int first, int nv,
                                          int vb, int max_sites, bool uniform, unsigned char* smem, int* s_task) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const RsLayout lay = rs_layout<Tl>(vb, max_sites, nw, uniform, kPairs);
    RsVisit* hd = reinterpret_cast<RsVisit*>(smem);
    RsPairs& pt = *reinterpret_cast<RsPairs*>(smem + align16((size_t)vb * sizeof(RsVisit)));
    RsTerms* tm = reinterpret_cast<RsTerms*>(smem + lay.terms);
    RsOut<float>* out = reinterpret_cast<RsOut<float>*>(smem + lay.out);
    RsSite<float>* sites = reinterpret_cast<RsSite<float>*>(smem + lay.site);
    float* hop = reinterpret_cast<float*>(smem + lay.hop);
    float2* buf = reinterpret_cast<float2*>(smem + lay.buf) + (size_t)(warp * Tl::NPW + lane / Tl::LPN) * Tl::node(kPairs);
    // Small windows: several visits per warp, so that its FP64 instructions
    // serve them together.
    constexpr int GL = Tl::NS == 1 ? 8 : Tl::NS <= 4 ? 16 : 32;
    for (int k0 = warp * (32 / GL); k0 < nv; k0 += nw * (32 / GL)) {
        const int k = k0 + lane / GL < nv ? k0 + lane / GL : nv - 1;   // lanes past the end repeat the last visit
        const int c = list ? list[first + k] : first + k;
        rs_gather<float, GL, true>(a, v.S_in, c, v.sites[c], hd[k], tm[k], sites + k * max_sites, lane % GL);
    }
    if (!kPairs)
        for (int k = nw - 1 - warp; k < (uniform ? 1 : nv); k += nw)
            rs_hopping(a, v.sites[list ? list[first + k] : first + k], hop + k * Tl::NS * Tl::NS, Tl::NS, lane);
    if (kPairs && warp == nw - 1) rs_pairs(a.m, v.sites[list ? list[first] : first], pt, lane);
    if (threadIdx.x == 0) *s_task = 0;
    __syncthreads();
    if (warp == nw - 1 && lane < nv) {
        // proposals and uniforms of the CTA's visits, one lane each, beside
        // the other warps' eliminations
        const int site = hd[lane].site;
        rs_proposal(a, v, site, tm[lane]);
        const double* so = v.S_in + 3 * (int64_t)site;
        const double dx = tm[lane].sn[0] - so[0];
        tm[lane].dv[0] = (float)(-a.unit.lam * dx);
        tm[lane].dv[1] = (float)(a.unit.J * dx);
        tm[lane].dv[2] = (float)(a.unit.J * (tm[lane].sn[1] - so[1]));
        tm[lane].dv[3] = (float)(a.unit.J * (tm[lane].sn[2] - so[2]));
    }
    __syncwarp();
    // Tasks: NPW nodes per warp, of one visit unless the windows are uniform.
    for (;;) {
        int task = 0;
        if (lane == 0) task = atomicAdd(s_task, 1);
        task = __shfl_sync(FULL_MASK, task, 0);
        int k = 0, j = uniform ? task * Tl::NPW + lane / Tl::LPN : task;
        for (; k < nv; ++k) {
            const int cls = hd[k].cls, M = cls < 0 ? 0 : c_fermi[cls].M;
            const int nt = uniform ? M : (M + Tl::NPW - 1) / Tl::NPW;
            if (j < nt) break;
            j -= nt;
        }
        bool idle = k >= nv;
        if (__all_sync(FULL_MASK, idle)) break;
        if (uniform) {
            // lanes past the last node repeat the warp's first one, unrecorded
            const int k0 = __shfl_sync(FULL_MASK, k, 0), j0 = __shfl_sync(FULL_MASK, j, 0);
            if (idle) { k = k0; j = j0; }
        } else {
            const int M = c_fermi[hd[k].cls].M;
            j = j * Tl::NPW + lane / Tl::LPN;
            idle = j >= M;
            if (idle) j = M - 1;
        }
        const double s = a.unit.T1 / c_fermi[hd[k].cls].y[j];
        RsOut<float> spare;
        RsOut<float>* const to = idle ? &spare : out + k * kFermiOut + j;
        if (lane % Tl::LPN == 0) to->eta = rs_rounding(s);
        if constexpr (kPairs) RsNode<Tl>::run_pairs(pt, sites + k * max_sites, (float)s, (float)(a.unit.t * s), buf, lane, to);
        else RsNode<Tl>::run(hd[k], sites + k * max_sites, hop + (uniform ? 0 : k * Tl::NS * Tl::NS), (float)s,
                             (float)(a.unit.t * s), buf, lane, to);
    }
    __syncthreads();
    if constexpr (Tl::NS <= 4) {
        // Many visits: the nodes' last pivots spread over the CTA in FP32, then a
        // lane per visit for the FP64 sums (a warp's FP64 instruction holds the
        // pipe for 17 cycles, whatever its lanes: one visit per warp took half
        // the time of a chain's stage).
        for (int q = threadIdx.x; q < nv * kFermiOut; q += blockDim.x) {
            const int k = q / kFermiOut, j = q % kFermiOut;
            if (hd[k].cls < 0 || j >= c_fermi[hd[k].cls].M) continue;
            RsOut<float>& r = out[q];
            float lq, t0, dl, dt;
            rs_last_pivot(r, tm[k].dv[0] * r.s, tm[k].dv[1] * r.s, tm[k].dv[2] * r.s, tm[k].dv[3] * r.s, lq, t0, dl, dt);
            r.P[0] = lq; r.P[1] = t0; r.P[2] = dl; r.P[3] = dt;
        }
        __syncthreads();
        // corrections for the rounding of the scales (FermiSlope)
        for (int q = threadIdx.x; q < nv * kFermiOut; q += blockDim.x) {
            const int k = q / kFermiOut, j = q % kFermiOut, cls = hd[k].cls;
            if (cls < 0 || j >= c_fermi[cls].M) continue;
            const RsOut<float>* near = out + k * kFermiOut + fermi_middle(j, c_fermi[cls].M) - 1;
            const FermiSlope& w = c_slope.of[cls][j];
            float cl = 0.f, ct = 0.f, cdl = 0.f, cdt = 0.f;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                cl += w.a[i] * ((float)near[i].lnd + near[i].P[0]);
                ct += w.b[i] * ((float)near[i].th + near[i].P[1]);
                cdl += w.a[i] * near[i].P[2];
                cdt += w.b[i] * near[i].P[3];
            }
            RsOut<float>& r = out[q];
            r.P[4] = r.eta * cl; r.P[5] = r.eta * ct; r.P[6] = r.eta * cdl; r.P[7] = r.eta * cdt;
        }
        __syncthreads();
        if (warp == 0 && lane < nv) {
            const FermiNodes& f = c_fermi[hd[lane].cls >= 0 ? hd[lane].cls : 0];
            double Lo = 0.0, Th = 0.0, dL = 0.0, dT = 0.0;
            float cl = 0.f, ct = 0.f, cdl = 0.f, cdt = 0.f;
            if (hd[lane].cls >= 0)
                for (int j = 0; j < f.M; ++j) {
                    const RsOut<float>& r = out[lane * kFermiOut + j];
                    Lo += f.a[j] * (r.lnd + (double)r.P[0]);
                    Th += f.b[j] * (r.th + (double)r.P[1]);
                    dL += f.a[j] * (double)r.P[2];
                    dT += f.b[j] * (double)r.P[3];
                    cl += r.P[4];
                    ct += r.P[5];
                    cdl += r.P[6];
                    cdt += r.P[7];
                }
            rs_final(mode, a, v, hd[lane], tm[lane], f, Lo + (double)cl, Th + (double)ct, dL + (double)cdl, dT + (double)cdt);
        }
    } else {
        for (int k = warp; k < nv; k += nw) rs_decide<float>(mode, a, v, hd[k], tm[k], out + k * kFermiOut, lane);
    }
}

// One visit, its nodes dealt to `parts` CTAs: each leaves its nodes' results in
// out (global memory), and the CTA that arrives last (the visit's ticket)
// decides.  Nobody waits for another CTA.  The CTA's last warp draws the
// proposal meanwhile.  Nodes are done by RsNode's lanes (FP32) or by RsGroup's
// threads (double-float): RsWarps and RsGroups below say how.
struct RsPartLayout { size_t terms, site, hop, buf, total; };
template <class E> __host__ __device__ inline RsPartLayout rs_part_layout(int max_sites, int max_layer, int threads) {
    RsPartLayout L;
    size_t o = align16(sizeof(RsVisit)) + align16(sizeof(RsPairs));
    L.terms = o; o = align16(o + sizeof(RsTerms));
    L.site = o;  o = align16(o + (size_t)max_sites * sizeof(RsSite<typename E::Real>));
    L.hop = o;   o = align16(o + (size_t)E::hop_stride(max_layer) * E::hop_stride(max_layer) * sizeof(typename E::Real));
    L.buf = o;   o = align16(o + (size_t)(threads - 32) / E::LANES * E::bytes(max_sites));
    L.total = o;
    return L;
}

// FP32 nodes on LPN lanes of a warp.  LANES: threads that share one `unit`
// index; a unit takes one node.
template <class Tl, bool kPairs> struct RsWarps {
    using Real = float;
    static constexpr int LANES = Tl::LPN;
    static constexpr bool kFullWarp = true;   // the warp's nodes run together
    static __host__ __device__ constexpr int hop_stride(int) { return Tl::NS; }
    static __host__ __device__ constexpr size_t bytes(int) { return Tl::node(kPairs) * sizeof(float2); }
    static __device__ __forceinline__ void run(const RsVisit& h, const RsPairs& pt, const RsSite<float>* site, const float* hop,
                                               int, float s, float tp, unsigned char* buf, int, RsOut<float>* out) {
        if constexpr (kPairs) RsNode<Tl>::run_pairs(pt, site, s, tp, reinterpret_cast<float2*>(buf), threadIdx.x & 31, out);
        else RsNode<Tl>::run(h, site, hop, s, tp, reinterpret_cast<float2*>(buf), threadIdx.x & 31, out);
    }
};
template <class Gp, bool kPairs> struct RsGroups {
    using Real = dfl;
    static constexpr int LANES = Gp::TPN;
    static constexpr bool kFullWarp = false;
    static __host__ __device__ constexpr int hop_stride(int max_layer) { return max_layer; }
    static __host__ __device__ constexpr size_t bytes(int max_sites) { return RsGroup<dfl, Gp>::bytes(2 * max_sites); }
    static __device__ __forceinline__ void run(const RsVisit& h, const RsPairs& pt, const RsSite<dfl>* site, const dfl* hop,
                                               int hs, dfl s, dfl tp, unsigned char* buf, int unit, RsOut<dfl>* out) {
        using G = RsGroup<dfl, Gp>;
        auto& sm = *reinterpret_cast<typename G::Smem*>(buf);
        const int t = threadIdx.x % Gp::TPN;
        if constexpr (kPairs) G::run_pairs(pt, site, s, tp, sm, t, 1 + unit, out);
        else G::run(h, site, hop, hs, s, tp, sm, t, 1 + unit, out);
    }
};

template <class E, bool kPairs>
__device__ __forceinline__ void rs_visit_part(RsMode mode, const StageArgs& a, const StageVar& v, int c, int part, int parts,
                                              RsOut<typename E::Real>* out, int max_sites, int max_layer, unsigned char* smem) {
    using T = typename E::Real;
    __shared__ int s_last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, units = (blockDim.x - 32) / E::LANES;
    const bool extra = threadIdx.x >= blockDim.x - 32;
    const auto lay = rs_part_layout<E>(max_sites, max_layer, blockDim.x);
    RsVisit& h = *reinterpret_cast<RsVisit*>(smem);
    RsPairs& pt = *reinterpret_cast<RsPairs*>(smem + align16(sizeof(RsVisit)));
    RsTerms& tm = *reinterpret_cast<RsTerms*>(smem + lay.terms);
    RsSite<T>* sites = reinterpret_cast<RsSite<T>*>(smem + lay.site);
    T* hop = reinterpret_cast<T*>(smem + lay.hop);
    const int hs = E::hop_stride(max_layer), site = v.sites[c];
    if (warp == 0) rs_gather<T, 32, false>(a, v.S_in, c, site, h, tm, sites, lane);
    if (extra) {
        if constexpr (kPairs) rs_pairs(a.m, site, pt, lane);
        else rs_hopping(a, site, hop, hs, lane);
    }
    __syncthreads();
    if (extra) {
        if (lane == 0) rs_proposal(a, v, site, tm);
        rs_terms(a, v.S_in, site, tm, lane);
    } else if (h.cls >= 0) {
        const FermiNodes& f = RsFermi<T>::tab(h.cls);
        // nodes part, part + parts, ... of the visit, in turn over the units
        const int unit = threadIdx.x / E::LANES, mine = (f.M - part + parts - 1) / parts;
        for (int u0 = 0; u0 < mine; u0 += units) {
            int u = u0 + unit;
            const bool idle = u >= mine;
            if (idle && !E::kFullWarp) break;
            if (idle) u = mine - 1;
            if (E::kFullWarp && __all_sync(FULL_MASK, idle)) break;
            const int j = part + parts * u;
            const double s = a.unit.T1 / f.y[j];
            RsOut<T> spare;
            RsOut<T>* const to = idle ? &spare : out + j;
            if (sizeof(T) == 4 && threadIdx.x % E::LANES == 0) to->eta = rs_rounding(s);
            E::run(h, pt, sites, hop, hs, T(s), T(a.unit.t * s), smem + lay.buf + (size_t)unit * E::bytes(max_sites), unit, to);
        }
    }
    if constexpr (sizeof(T) == 8) {   // the re-solve
        if (h.cls < 0) {
            __syncthreads();
            if (part == 0) rs_exact(a, v, h, tm, blockIdx.x, smem + lay.site);
            __syncthreads();
            return;
        }
    }
    __threadfence();   // this thread's node results, before the ticket
    __syncthreads();
    if (threadIdx.x == 0) {
        s_last = parts == 1 || atomicAdd(&a.ticket[c], 1) == parts - 1;
        if (parts > 1 && s_last) a.ticket[c] = 0;
        __threadfence();
    }
    __syncthreads();
    if (s_last && warp == 0) rs_decide<T>(mode, a, v, h, tm, out, lane);
    __syncthreads();
}

}  // namespace ptca

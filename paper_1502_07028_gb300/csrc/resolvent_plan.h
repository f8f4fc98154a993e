// resolvent_plan.h -- host rules of the determinant sweeps (resolvent.cuh):
// which problems they serve and how a window is laid out.
#pragma once

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "resolvent.cuh"

namespace ptca {

inline int lattice_dims(const Model& m) { return (m.Lx > 1) + (m.Ly > 1) + (m.Lz > 1); }
// Sites per layer of the largest window (layers along its longest axis).
inline int layer_sites(const Model& m) {
    const int d = lattice_dims(m);
    return d <= 1 ? 1 : d == 2 ? m.Lc : m.Lc * m.Lc;
}
inline int window_sites(const Model& m) { return layer_sites(m) * m.Lc; }

// Sites per block where the windows are split by parity, else 0: a ring of
// layers of even extents above 2 (every bond, all of them single, joins opposite
// parities), at most 64 sites, and the two blocks' 4 b^3 multiply-adds at
// most two thirds of the layers' (4 L - 7) b^3 -- rings of four layers.  Measured
// on 4x4x4 clusters: 8.4 -> 3.8 ms for a stage of 8000 visits.
inline int pair_sites(const Model& m) {
    if (!m.lattice_periodic || !m.cluster_periodic || (m.Lc & 1) || m.Lc < 4 || window_sites(m) > kPairSites) return 0;
    const int nb = (window_sites(m) / 2 + 1) / 2, ns = layer_sites(m);
    return 6.0 * nb * nb * nb <= (4.0 * m.Lc - 7.0) * ns * ns * ns ? nb : 0;
}

// Gershgorin's bound on |x| for windows of unit vectors.
inline double unit_bound(const Model& m) {
    return (fabs(m.mu - m.e0) + fabs(m.lam) + fabs(m.JH) + 2.0 * lattice_dims(m) * fabs(m.t)) / m.T;
}
inline int class_nodes(const FermiNodes* tab, double X) {
    int c = 0;
    while (c + 1 < kFermiClasses && X > tab[c].X) ++c;
    return tab[c].M;
}

// f(tile, split by parity) with the tile of the problem's windows.
template <typename F> auto with_tile(const Model& m, F f) {
    const int np = pair_sites(m), ns = layer_sites(m);
    if (np == 1) return f(RsT1{}, std::true_type{});
    if (np > 0 && np <= 4) return f(RsT4{}, std::true_type{});
    if (np > 4) return f(RsT16{}, std::true_type{});
    if (ns <= 1) return f(RsT1{}, std::false_type{});
    if (ns <= 4) return f(RsT4{}, std::false_type{});
    if (ns <= 8) return f(RsT8{}, std::false_type{});
    if (ns <= 12) return f(RsT12{}, std::false_type{});
    return f(RsT16{}, std::false_type{});
}

// Shape of a k_stage_rs launch of `count` visits with M nodes each: warps per
// CTA, visits per CTA, dynamic shared memory.
struct RsStagePlan { int nw, vb; size_t bytes; };

// Visits per CTA: enough that its warps share their nodes evenly (a warp takes
// NPW nodes at a time).
// - Small windows: eight warps and 16 visits, or, for chains, the visits that one
//   turn of the warps takes (24 at 10 nodes); fewer leave turns empty or repeat the
//   CTA's start too often.
// - Up to 8 sites per layer: two (1099 us per 2500 visits of 8x8 clusters at 13
//   nodes against 1219 with four; 1160 us at today's 14).
// - One node per warp and one CTA per SM: the count with the fewest idle warps (3.8
//   against 5.4 ms for 8000 visits of 4x4x4 clusters, 11 nodes on 8 warps), the
//   largest where none idles (12 nodes: a 40^3 sweep takes 38.0 ms with four visits,
//   39.7 with two), of those that `room` bytes hold: eight warps' blocks of 13 to 16 sites per layer
//   take 204 KB, each visit of a 16x16 window 5 KB more.
// - Two nodes per warp and one CTA per SM (9 to 12 sites per layer, seven warps): a
//   visit of 15 nodes leaves one of its eight warp loads to a second turn, where it
//   takes a quarter of a full turn; two visits together leave one of fifteen.  12x12
//   clusters, 576 visits: 1576 -> 1267 us; 2500 visits: 6.54 -> 5.58 ms (14 nodes and
//   one visit: 1261 us and 5.32 ms; two visits 1255 us and 5.53 ms).  Not at 16 nodes,
//   where both leave one per visit (6.54 and 6.88 ms).
template <class Tl, bool kPairs>
RsStagePlan rs_stage_plan(int M, int max_sites, bool uniform, int count, int sms, size_t room) {
    RsStagePlan p{std::min((M + Tl::NPW - 1) / Tl::NPW, Tl::MAXT / 32), 1, 0};
    if (Tl::NS <= 4) {
        p.nw = Tl::MAXT / 32;
        p.vb = Tl::NS == 1 ? std::min(24, 8 * Tl::NPW / M) : 16;
    } else if (Tl::NS <= 8) {
        p.vb = 2;
    } else if (Tl::NPW == 1 && uniform) {
        double best = 0.0;
        for (int v = 1; v <= 5 && (v == 1 || count >= 4 * v * sms); ++v) {
            if (v > 1 && rs_layout<Tl>(v, max_sites, p.nw, uniform, kPairs).total > room) break;
            const double share = (double)v * M / (((v * M + p.nw - 1) / p.nw) * p.nw);
            if (share >= best + (share < 1.0 ? 0.01 : 0.0)) { best = share; p.vb = v; }
        }
    } else if (uniform) {
        // turns of the SM's CTAs one after another, four loads of a part-filled turn as a full one
        auto turns = [&](int v) {
            const int loads = (v * M + Tl::NPW - 1) / Tl::NPW, ctas = (count + v - 1) / v;
            return (ctas + sms - 1) / sms * (loads / p.nw + std::min(1.0, 0.25 * (loads % p.nw)));
        };
        if (turns(2) < turns(1) && rs_layout<Tl>(2, max_sites, p.nw, uniform, kPairs).total <= room) p.vb = 2;
    }
    p.bytes = rs_layout<Tl>(p.vb, max_sites, p.nw, uniform, kPairs).total;
    return p;
}

// Stages of few visits: the tile, and CTAs per visit, threads and dynamic shared
// memory of a k_stage_rs_few launch.
template <typename F> auto with_latency_tile(const Model& m, F f) {
    const int np = pair_sites(m), ns = layer_sites(m);
    if (np > 0 && np <= 4) return f(RsL4{}, std::true_type{});
    if (np > 4) return f(RsT16{}, std::true_type{});
    if (ns <= 4) return f(RsL4{}, std::false_type{});
    if (ns <= 8) return f(RsL8{}, std::false_type{});
    return f(RsT16{}, std::false_type{});
}
struct RsFewPlan { int parts, threads; size_t bytes; };
template <class Tl, bool kPairs> RsFewPlan rs_few_plan(int M, int max_sites, int max_layer, int count, int sms) {
    // a visit's warps over as many CTAs as give four per SM
    const int warps = (M + Tl::NPW - 1) / Tl::NPW;
    RsFewPlan p;
    p.parts = std::max(1, std::min(warps, 4 * sms / count));
    p.threads = std::min(32 * ((warps + p.parts - 1) / p.parts) + 32, Tl::MAXT);
    p.bytes = rs_part_layout<RsWarps<Tl, kPairs>>(max_sites, max_layer, p.threads).total;
    return p;
}

// The re-solve: threads per node, and dynamic shared memory.
template <typename F> auto with_group(const Model& m, F f) {
    const int np = pair_sites(m), ns = layer_sites(m);
    if (np > 0 && np <= 4) return f(RsG8{}, std::true_type{});
    if (np > 4) return f(RsG32{}, std::true_type{});
    if (ns <= 4) return f(RsG8{}, std::false_type{});
    if (ns <= 8) return f(RsG16{}, std::false_type{});
    if (ns <= 12) return f(RsG24{}, std::false_type{});
    return f(RsG32{}, std::false_type{});
}
template <class Gp, bool kPairs> size_t rs_resolve_bytes(int max_sites, int max_layer) {
    const auto lay = rs_part_layout<RsGroups<Gp, kPairs>>(max_sites, max_layer, Gp::TPN * Gp::DFG + 32);
    return std::max(lay.total, lay.site + rs_exact_bytes(2 * max_sites));
}

// What the device's opt-in limit leaves for dynamic shared memory beside the
// kernels' own few words.
constexpr size_t kRsStatic = 256;

// Allow a kernel all the dynamic shared memory of the device.
template <class K> cudaError_t allow_smem(K kernel, size_t smem_limit) {
    cudaFuncAttributes attr;
    cudaError_t e = cudaFuncGetAttributes(&attr, kernel);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(smem_limit - attr.sharedSizeBytes));
    return e;
}

}  // namespace ptca

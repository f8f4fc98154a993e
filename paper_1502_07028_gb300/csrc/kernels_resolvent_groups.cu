// kernels_resolvent_groups.cu -- determinant kernels that spread a visit over
// several CTAs (resolvent.cuh): stages of few visits in FP32, and the
// double-float re-solve.
#include "launch.h"
#include "resolvent_plan.h"

namespace ptca {

// Deferred decisions of a stage, the same elimination in double-float.  A stage
// defers a handful to some tens of visits and the next stage waits for
// them, so the CTAs share each visit's nodes while there are fewer visits than
// CTAs, and take whole visits in turn beyond that.  scratch: node results, one
// set per CTA of the grid.
template <class Gp, bool kPairs>
__global__ void __launch_bounds__(Gp::TPN * Gp::DFG + 32, 1) k_resolve_rs(const __grid_constant__ StageArgs a, int max_sites,
                                                                         int max_layer, RsOut<dfl>* scratch, int max_parts) {
    extern __shared__ __align__(16) unsigned char smem[];
    // No launch_next(): the next stage's blocks, resident while these still hold
    // their shared memory, crowd onto few SMs (32x32, 16 visits a stage: 4.9 ms a
    // sweep instead of 3.1).  The stage does call it: 3.4 ms without chaining.
    wait_previous();
    const int nflag = (int)*(volatile unsigned int*)a.flag_count;
    if (a.flag_next && blockIdx.x == 0 && threadIdx.x == 0) *a.flag_next = 0;
    if (nflag == 0) return;
    int parts = (int)gridDim.x / nflag;
    parts = parts < 1 ? 1 : parts > max_parts ? max_parts : parts;
    const StageVar v = stage_var(a);
    if (parts > 1) {
        const int i = blockIdx.x % nflag, part = blockIdx.x / nflag;
        if (part >= parts) return;
        rs_visit_part<RsGroups<Gp, kPairs>, kPairs>(RS_RESOLVE, a, v, a.flag_list[i], part, parts, scratch + (size_t)i * kFermiMaxNodes,
                                       max_sites, max_layer, smem);
        return;
    }
    for (int i = blockIdx.x; i < nflag; i += gridDim.x)
        rs_visit_part<RsGroups<Gp, kPairs>, kPairs>(RS_RESOLVE, a, v, a.flag_list[i], 0, 1, scratch + (size_t)blockIdx.x * kFermiMaxNodes,
                                       max_sites, max_layer, smem);
}

// A stage of few visits, `parts` CTAs each, FP32 nodes.  scratch: node results by
// stage index.
template <class Tl, bool kPairs>
__global__ void __launch_bounds__(Tl::MAXT, Tl::MINB) k_stage_rs_few(const __grid_constant__ StageArgs a, int max_sites,
                                                                           int max_layer, RsOut<float>* scratch, int parts,
                                                                           RsMode mode, int c0) {
    extern __shared__ __align__(16) unsigned char smem[];
    launch_next();
    wait_previous();
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < a.prev_count + a.prev2_count; k += gridDim.x * blockDim.x) {
        const int s = k < a.prev_count ? a.prev_sites[k] : a.prev2_sites[k - a.prev_count];
        a.S_out[3 * s] = a.S_in[3 * s];
        a.S_out[3 * s + 1] = a.S_in[3 * s + 1];
        a.S_out[3 * s + 2] = a.S_in[3 * s + 2];
    }
    const int count = a.count_dev ? (int)*a.count_dev : a.count;
    const int i = blockIdx.x / parts;
    if (i >= count) return;
    const int c = a.perm ? a.perm[i] : c0 + i;
    rs_visit_part<RsWarps<Tl, kPairs>, kPairs>(mode, a, stage_var(a), c, blockIdx.x % parts, parts, scratch + (size_t)c * kFermiMaxNodes,
                                     max_sites, max_layer, smem);
}

cudaError_t configure_resolvent_groups(size_t smem_limit) {
    cudaError_t e = cudaSuccess;
    auto group = [&](auto g, auto pairs) {
        if (e == cudaSuccess) e = allow_smem(k_resolve_rs<decltype(g), decltype(pairs)::value>, smem_limit);
    };
    auto tile = [&](auto t, auto pairs) {
        if (e == cudaSuccess) e = allow_smem(k_stage_rs_few<decltype(t), decltype(pairs)::value>, smem_limit);
    };
    tile(RsL4{}, std::true_type{});
    tile(RsT16{}, std::true_type{});
    tile(RsL4{}, std::false_type{});
    tile(RsL8{}, std::false_type{});
    tile(RsT16{}, std::false_type{});
    group(RsG8{}, std::true_type{});
    group(RsG32{}, std::true_type{});
    group(RsG8{}, std::false_type{});
    group(RsG16{}, std::false_type{});
    group(RsG24{}, std::false_type{});
    group(RsG32{}, std::false_type{});
    return e;
}

size_t resolvent_scratch_bytes(int sms) {
    return (size_t)2 * sms * kFermiMaxNodes * sizeof(RsOut<dfl>) + 2 * (size_t)kFewVisits * kFermiMaxNodes * sizeof(RsOut<float>);
}

cudaError_t launch_groups(RsMode mode, const StageArgs& a, int c0, int sms, cudaStream_t st) {
    static const FermiNodes tab[kFermiClasses] = {PTCA_FERMI_NODES};
    const int M = class_nodes(tab, unit_bound(a.m)), ms = window_sites(a.m), ml = layer_sites(a.m);
    // node results by stage index: one set per stage parity (a.rs_half), as the
    // other per-visit scratch
    unsigned char* base = static_cast<unsigned char*>(a.rs_scratch) + (size_t)2 * sms * kFermiMaxNodes * sizeof(RsOut<dfl>);
    RsOut<float>* scratch = reinterpret_cast<RsOut<float>*>(base) + (size_t)a.rs_half * kFewVisits * kFermiMaxNodes;
    return with_latency_tile(a.m, [&](auto tile, auto pairs) {
        using Tl = decltype(tile);
        constexpr bool kPairs = decltype(pairs)::value;
        const RsFewPlan p = rs_few_plan<Tl, kPairs>(M, ms, ml, a.count, sms);
        return launch_chained(k_stage_rs_few<Tl, kPairs>, a.count * p.parts, p.threads, p.bytes, st, a, ms, ml, scratch,
                              p.parts, mode, c0);
    });
}

cudaError_t launch_resolve_resolvent(const StageArgs& a, int sms, cudaStream_t st) {
    static const FermiNodes tab[kFermiClasses] = {PTCA_FERMI_NODES_DF};
    const int M = class_nodes(tab, unit_bound(a.m)), ms = window_sites(a.m), ml = layer_sites(a.m);
    return with_group(a.m, [&](auto group, auto pairs) {
        using Gp = decltype(group);
        const size_t smem = rs_resolve_bytes<Gp, decltype(pairs)::value>(ms, ml);
        const int grid = (Gp::TPN == 32 ? 2 : 1) * sms;   // one warp per node: two CTAs fit on an SM
        return launch_chained(k_resolve_rs<Gp, decltype(pairs)::value>, grid, Gp::TPN * Gp::DFG + 32, smem, st, a, ms, ml,
                              static_cast<RsOut<dfl>*>(a.rs_scratch), M);
    });
}

}  // namespace ptca

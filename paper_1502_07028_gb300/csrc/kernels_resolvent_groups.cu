// kernels_resolvent_groups.cu -- determinant kernels with a group of threads per
// node (resolvent.cuh): stages of few visits in FP32, and the double-float
// re-solve.
#include <algorithm>
#include <type_traits>

#include "launch.h"
#include "resolvent_plan.h"

namespace ptca {

// Deferred decisions of a stage, the same elimination in double-float: one
// thread-block cluster per visit, a group of threads per node (a stage defers
// some tens of visits, and the next stage waits for them).
template <class Gp, bool kPairs>
__global__ void __launch_bounds__(Gp::TPN * Gp::DFG, 1) k_resolve_rs(const __grid_constant__ StageArgs a, int max_sites,
                                                                    int max_layer) {
    extern __shared__ __align__(16) unsigned char smem[];
    namespace cg = cooperative_groups;
    const cg::cluster_group cl = cg::this_cluster();
    const int size = (int)cl.num_blocks();
    const int nflag = (int)*(volatile unsigned int*)a.flag_count;
    if (nflag == 0) return;
    cl.sync();       // every CTA of the cluster runs before its shared memory is written
    for (int i = blockIdx.x / size; i < nflag; i += gridDim.x / size) {
        rs_visit_groups<dfl, Gp, kPairs>(RS_RESOLVE, a, stage_var(a), a.flag_list[i], max_sites, max_layer, smem);
        cl.sync();   // the first CTA's results are read before the next visit overwrites them
    }
}

// A stage of few visits: one cluster per visit, a group of threads per FP32 node.
template <class Gp, bool kPairs>
__global__ void __launch_bounds__(Gp::TPN * Gp::SPG, 1) k_stage_rs_few(const __grid_constant__ StageArgs a, int max_sites,
                                                                      int max_layer, RsMode mode, int c0) {
    extern __shared__ __align__(16) unsigned char smem[];
    namespace cg = cooperative_groups;
    const cg::cluster_group cl = cg::this_cluster();
    const int size = (int)cl.num_blocks();
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < a.prev_count + a.prev2_count; k += gridDim.x * blockDim.x) {
        const int s = k < a.prev_count ? a.prev_sites[k] : a.prev2_sites[k - a.prev_count];
        a.S_out[3 * s] = a.S_in[3 * s];
        a.S_out[3 * s + 1] = a.S_in[3 * s + 1];
        a.S_out[3 * s + 2] = a.S_in[3 * s + 2];
    }
    const int count = a.count_dev ? (int)*a.count_dev : a.count;
    const int i = blockIdx.x / size;
    if (i >= count) return;
    if (size > 1) cl.sync();
    rs_visit_groups<float, Gp, kPairs>(mode, a, stage_var(a), a.perm ? a.perm[i] : c0 + i, max_sites, max_layer, smem);
}

template <typename F> static auto with_group(const Model& m, F f) {
    const int np = pair_sites(m), ns = layer_sites(m);
    if (np > 0 && np <= 4) return f(RsG8{}, std::true_type{});
    if (np > 4) return f(RsG32{}, std::true_type{});
    if (ns <= 4) return f(RsG8{}, std::false_type{});
    if (ns <= 8) return f(RsG16{}, std::false_type{});
    if (ns <= 12) return f(RsG24{}, std::false_type{});
    return f(RsG32{}, std::false_type{});
}

cudaError_t configure_resolvent_groups(size_t smem_limit) {
    cudaError_t e = cudaSuccess;
    auto group = [&](auto g, auto pairs) {
        if (e == cudaSuccess) e = allow_smem(k_resolve_rs<decltype(g), decltype(pairs)::value>, smem_limit);
        if (e == cudaSuccess) e = allow_smem(k_stage_rs_few<decltype(g), decltype(pairs)::value>, smem_limit);
    };
    group(RsG8{}, std::true_type{});
    group(RsG32{}, std::true_type{});
    group(RsG8{}, std::false_type{});
    group(RsG16{}, std::false_type{});
    group(RsG24{}, std::false_type{});
    group(RsG32{}, std::false_type{});
    return e;
}

template <typename K, typename... A>
static cudaError_t launch_clusters(K kernel, int grid, int threads, size_t smem, int size, cudaStream_t st, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = size;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = size > 1 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// The smallest cluster of up to 8 CTAs that holds a group for every node.
static int cluster_for(int nodes, int groups) {
    int size = 1;
    while (size < 8 && size * groups < nodes) size *= 2;
    return size;
}

cudaError_t launch_groups(RsMode mode, const StageArgs& a, int c0, cudaStream_t st) {
    static const FermiNodes tab[kFermiClasses] = {PTCA_FERMI_NODES};
    const int M = class_nodes(tab, unit_bound(a.m)), ms = window_sites(a.m), ml = layer_sites(a.m);
    return with_group(a.m, [&](auto group, auto pairs) {
        using Gp = decltype(group);
        const int size = cluster_for(M, Gp::SPG), groups = std::min((M + size - 1) / size, Gp::SPG);
        return launch_clusters(k_stage_rs_few<Gp, decltype(pairs)::value>, a.count * size, Gp::TPN * groups,
                               rs_group_layout<float, Gp>(ms, ml, groups).total, size, st, a, ms, ml, mode, c0);
    });
}

cudaError_t launch_resolve_resolvent(const StageArgs& a, int sms, cudaStream_t st) {
    static const FermiNodes tab[kFermiClasses] = {PTCA_FERMI_NODES_DF};
    const int M = class_nodes(tab, unit_bound(a.m)), ms = window_sites(a.m), ml = layer_sites(a.m);
    return with_group(a.m, [&](auto group, auto pairs) {
        using Gp = decltype(group);
        const int size = cluster_for(M, Gp::DFG);
        const int per_sm = Gp::TPN == 32 ? 2 : 1;   // CTAs that fit on an SM beside each other
        const auto lay = rs_group_layout<dfl, Gp>(ms, ml, Gp::DFG);
        const size_t smem = std::max(lay.total, lay.out + rs_exact_bytes(2 * ms));
        return launch_clusters(k_resolve_rs<Gp, decltype(pairs)::value>, per_sm * sms / size * size, Gp::TPN * Gp::DFG, smem,
                               size, st, a, ms, ml);
    });
}

}  // namespace ptca

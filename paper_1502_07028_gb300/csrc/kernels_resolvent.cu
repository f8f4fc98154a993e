// kernels_resolvent.cu -- stage kernels of PTCA_MIXED sweeps whose free
// energies come from determinants (resolvent.cuh), and their launch rules.
#include <algorithm>

#include "launch.h"
#include "resolvent.cuh"

namespace ptca {

// One PTCA stage (Sec. III.a) on FP32 nodes: CTA b takes visits [b vb, b vb + vb).
template <class Tl>
__global__ void __launch_bounds__(Tl::MAXT, Tl::MINB) k_stage_rs(const __grid_constant__ StageArgs a, int vb, int max_sites,
                                                                    bool uniform) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_task;
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < a.prev_count + a.prev2_count; k += gridDim.x * blockDim.x) {
        const int s = k < a.prev_count ? a.prev_sites[k] : a.prev2_sites[k - a.prev_count];
        a.S_out[3 * s] = a.S_in[3 * s];
        a.S_out[3 * s + 1] = a.S_in[3 * s + 1];
        a.S_out[3 * s + 2] = a.S_in[3 * s + 2];
    }
    const int count = a.count_dev ? (int)*a.count_dev : a.count;
    const int first = blockIdx.x * vb;
    if (first >= count) return;
    rs_visits<Tl, RS_STAGE>(a, stage_var(a), a.perm, first, count - first < vb ? count - first : vb, vb, max_sites, uniform,
                            smem, &s_task);
}

// Deferred decisions of a stage, the same elimination in double-float: one
// thread-block cluster per visit, a group of threads per node (a stage defers
// some tens of visits, and the next stage waits for them).
template <class Gp>
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
        rs_visit_groups<dfl, Gp, RS_RESOLVE>(a, stage_var(a), a.flag_list[i], max_sites, max_layer, smem);
        cl.sync();   // the first CTA's results are read before the next visit overwrites them
    }
}

// A stage of few visits: one cluster per visit, a group of threads per FP32 node.
template <class Gp>
__global__ void __launch_bounds__(Gp::TPN * Gp::SPG, 1) k_stage_rs_few(const __grid_constant__ StageArgs a, int max_sites,
                                                                      int max_layer) {
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
    cl.sync();
    rs_visit_groups<float, Gp, RS_STAGE>(a, stage_var(a), a.perm ? a.perm[i] : i, max_sites, max_layer, smem);
}
template <class Gp>
__global__ void __launch_bounds__(Gp::TPN * Gp::SPG, 1) k_check_rs_few(const __grid_constant__ StageArgs a, int c0, int max_sites,
                                                                      int max_layer) {
    extern __shared__ __align__(16) unsigned char smem[];
    rs_visit_groups<float, Gp, RS_CHECK>(a, stage_var(a), c0 + blockIdx.x, max_sites, max_layer, smem);
}

// Free energies of visits c0 .. c0 + count - 1 for the precision checker.
template <class Tl>
__global__ void __launch_bounds__(Tl::MAXT, Tl::MINB) k_check_rs(const __grid_constant__ StageArgs a, int c0, int max_sites) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_task;
    rs_visits<Tl, RS_CHECK>(a, stage_var(a), nullptr, c0 + blockIdx.x, 1, 1, max_sites, true, smem, &s_task);
}

// Sites per layer of the largest window (layers along its longest axis).
static int layer_sites(const Model& m) {
    const int d = (m.Lx > 1) + (m.Ly > 1) + (m.Lz > 1);
    return d <= 1 ? 1 : d == 2 ? m.Lc : m.Lc * m.Lc;
}
static int window_sites(const Model& m) {
    const int d = (m.Lx > 1) + (m.Ly > 1) + (m.Lz > 1);
    return d <= 1 ? m.Lc : layer_sites(m) * m.Lc;
}

bool resolvent_supported(const Model& m) {
    if (layer_sites(m) > 16) return false;
    // |x| of a window of unit vectors: half the last class leaves room for
    // longer mean fields and distortions (windows beyond it are re-solved).
    const int d = (m.Lx > 1) + (m.Ly > 1) + (m.Lz > 1);
    const double bound = fabs(m.mu - m.e0) + fabs(m.lam) + fabs(m.JH) + 2.0 * d * fabs(m.t);
    return bound / m.T <= 0.5 * kFermiMaxX;
}

// Nodes of a window of unit vectors.
static int nominal_nodes(const Model& m) {
    static const FermiNodes tab[kFermiClasses] = {PTCA_FERMI_NODES};
    const int d = (m.Lx > 1) + (m.Ly > 1) + (m.Lz > 1);
    const double X = (fabs(m.mu - m.e0) + fabs(m.lam) + fabs(m.JH) + 2.0 * d * fabs(m.t)) / m.T;
    int c = 0;
    while (c + 1 < kFermiClasses && X > tab[c].X) ++c;
    return tab[c].M;
}

// f(tile) with the tile of the problem's layers.
template <typename F> static auto with_tile(const Model& m, F f) {
    const int ns = layer_sites(m);
    if (ns <= 1) return f(RsT1{});
    if (ns <= 4) return f(RsT4{});
    if (ns <= 8) return f(RsT8{});
    if (ns <= 12) return f(RsT12{});
    return f(RsT16{});
}

template <typename F> static auto with_group(const Model& m, F f) {
    const int ns = layer_sites(m);
    if (ns <= 4) return f(RsG8{});
    if (ns <= 8) return f(RsG16{});
    if (ns <= 12) return f(RsG24{});
    return f(RsG32{});
}

template <class K> static cudaError_t allow_smem(K kernel, size_t smem_limit) {
    cudaFuncAttributes attr;
    cudaError_t e = cudaFuncGetAttributes(&attr, kernel);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(smem_limit - attr.sharedSizeBytes));
    return e;
}
template <class Tl> static cudaError_t configure(size_t smem_limit) {
    cudaError_t e = allow_smem(k_stage_rs<Tl>, smem_limit);
    if (e == cudaSuccess) e = allow_smem(k_check_rs<Tl>, smem_limit);
    return e;
}
template <class Gp> static cudaError_t configure_groups(size_t smem_limit) {
    cudaError_t e = allow_smem(k_resolve_rs<Gp>, smem_limit);
    if (e == cudaSuccess) e = allow_smem(k_stage_rs_few<Gp>, smem_limit);
    if (e == cudaSuccess) e = allow_smem(k_check_rs_few<Gp>, smem_limit);
    return e;
}
cudaError_t configure_resolvent_kernels(size_t smem_limit) {
    cudaError_t e = configure<RsT1>(smem_limit);
    if (e == cudaSuccess) e = configure<RsT4>(smem_limit);
    if (e == cudaSuccess) e = configure<RsT8>(smem_limit);
    if (e == cudaSuccess) e = configure<RsT12>(smem_limit);
    if (e == cudaSuccess) e = configure<RsT16>(smem_limit);
    if (e == cudaSuccess) e = configure_groups<RsG8>(smem_limit);
    if (e == cudaSuccess) e = configure_groups<RsG16>(smem_limit);
    if (e == cudaSuccess) e = configure_groups<RsG24>(smem_limit);
    if (e == cudaSuccess) e = configure_groups<RsG32>(smem_limit);
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

cudaError_t launch_stage_resolvent(const StageArgs& a, bool few, int sms, cudaStream_t st) {
    if (a.count <= 0) return cudaSuccess;
    const int M = nominal_nodes(a.m), ms = window_sites(a.m), ml = layer_sites(a.m);
    if (few)
        return with_group(a.m, [&](auto group) {
            using Gp = decltype(group);
            // the smallest cluster that holds a group for every node
            int size = 1;
            while (size < 8 && size * Gp::SPG < M) size *= 2;
            const int groups = std::min((M + size - 1) / size, Gp::SPG);
            return launch_clusters(k_stage_rs_few<Gp>, a.count * size, Gp::TPN * groups,
                                   rs_group_layout<float, Gp>(ms, ml, groups).total, size, st, a, ms, ml);
        });
    return with_tile(a.m, [&](auto tile) {
        using Tl = decltype(tile);
        const int tasks = (M + Tl::NPW - 1) / Tl::NPW;
        const bool uniform = a.m.lattice_periodic;
        int vb = 1, nw = std::min(tasks, Tl::MAXT / 32);
        if (Tl::NS <= 4) {
            vb = Tl::NS == 1 ? 24 : 16;
            nw = 8;
        } else if (Tl::NS <= 8) {
            vb = 2;
        }
        k_stage_rs<Tl><<<(a.count + vb - 1) / vb, 32 * nw, rs_layout<Tl>(vb, ms, nw, uniform).total, st>>>(a, vb, ms, uniform);
        return cudaGetLastError();
    });
}

cudaError_t launch_check_resolvent(const StageArgs& a, bool few, int c0, int count, double* F, cudaStream_t st) {
    if (count <= 0) return cudaSuccess;
    StageArgs b = a;
    b.Fbuf = F - 2 * (int64_t)c0;
    const int M = nominal_nodes(a.m), ms = window_sites(a.m), ml = layer_sites(a.m);
    if (few)
        return with_group(a.m, [&](auto group) {
            using Gp = decltype(group);
            k_check_rs_few<Gp><<<count, Gp::TPN * Gp::SPG, rs_group_layout<float, Gp>(ms, ml, Gp::SPG).total, st>>>(b, c0, ms, ml);
            return cudaGetLastError();
        });
    return with_tile(a.m, [&](auto tile) {
        using Tl = decltype(tile);
        const int nw = std::min((M + Tl::NPW - 1) / Tl::NPW, Tl::MAXT / 32);
        k_check_rs<Tl><<<count, 32 * nw, rs_layout<Tl>(1, ms, nw, true).total, st>>>(b, c0, ms);
        return cudaGetLastError();
    });
}

cudaError_t launch_resolve_resolvent(const StageArgs& a, int sms, cudaStream_t st) {
    const int ms = window_sites(a.m);
    return with_group(a.m, [&](auto group) {
        using Gp = decltype(group);
        const int size = 8;
        const auto lay = rs_group_layout<dfl, Gp>(ms, layer_sites(a.m), Gp::DFG);
        const size_t smem = std::max(lay.total, lay.out + rs_exact_bytes(2 * ms));
        return launch_clusters(k_resolve_rs<Gp>, sms / size * size, Gp::TPN * Gp::DFG, smem, size, st, a, ms, layer_sites(a.m));
    });
}

}  // namespace ptca

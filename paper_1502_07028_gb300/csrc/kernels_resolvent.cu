// kernels_resolvent.cu -- stage kernel of PTCA_MIXED sweeps whose free energies
// come from determinants (resolvent.cuh), nodes packed into warps.
#include "launch.h"
#include "resolvent_plan.h"

namespace ptca {

// One PTCA stage (Sec. III.a) on FP32 nodes: CTA b takes visits [b vb, b vb + vb)
// of the work list; of c0, c0 + 1, ... for the precision checker.
template <class Tl, bool kPairs>
__global__ void __launch_bounds__(Tl::MAXT, Tl::MINB) k_stage_rs(const __grid_constant__ StageArgs a, int vb, int max_sites,
                                                                 bool uniform, RsMode mode, int c0) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_task;
    launch_next();
    wait_previous();
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < a.prev_count + a.prev2_count; k += gridDim.x * blockDim.x) {
        const int s = k < a.prev_count ? a.prev_sites[k] : a.prev2_sites[k - a.prev_count];
        a.S_out[3 * s] = a.S_in[3 * s];
        a.S_out[3 * s + 1] = a.S_in[3 * s + 1];
        a.S_out[3 * s + 2] = a.S_in[3 * s + 2];
    }
    const int count = a.count_dev ? (int)*a.count_dev : a.count;
    const int first = blockIdx.x * vb;
    if (first >= count) return;
    rs_visits<Tl, kPairs>(mode, a, stage_var(a), a.perm, c0 + first, count - first < vb ? count - first : vb, vb, max_sites,
                          uniform, smem, &s_task);
}

// Proposals and ln u of a whole sweep, one thread per site.  A site's variable
// changes in its own stage alone, so that its value at the sweep's start is the one
// its visit finds.
__global__ void k_proposals(Model m, const double* __restrict__ S, int N, uint64_t sweep, const unsigned long long* sweep_dev,
                            double4* __restrict__ out) {
    const int site = blockIdx.x * blockDim.x + threadIdx.x;
    if (site >= N) return;
    const uint64_t sw = sweep + (sweep_dev ? *sweep_dev : 0);
    double sn[3], u0, u1;
    propose(m, sw, (uint32_t)site, S + 3 * (int64_t)site, sn);
    uniform2(m.seed, sw, (uint32_t)site, RNG_ACCEPT, u0, u1);
    out[site] = make_double4(sn[0], sn[1], sn[2], log(u0));
}

cudaError_t launch_proposals(const StageArgs& a, const double* S, int N, double4* out, cudaStream_t st) {
    k_proposals<<<(N + 63) / 64, 64, 0, st>>>(a.m, S, N, a.sweep, a.sweep_dev, out);
    return cudaGetLastError();
}

cudaError_t configure_resolvent_kernels(size_t smem_limit) {
    cudaError_t e = configure_resolvent_groups(smem_limit);
    auto tile = [&](auto t, auto pairs) {
        if (e == cudaSuccess) e = allow_smem(k_stage_rs<decltype(t), decltype(pairs)::value>, smem_limit);
    };
    tile(RsT1{}, std::true_type{});
    tile(RsT4{}, std::true_type{});
    tile(RsT16{}, std::true_type{});
    tile(RsT1{}, std::false_type{});
    tile(RsT4{}, std::false_type{});
    tile(RsT8{}, std::false_type{});
    tile(RsT12{}, std::false_type{});
    tile(RsT16{}, std::false_type{});
    return e;
}

bool resolvent_supported(const Model& m) {
    // Blocks of up to 32 rows; |x| of a window of unit vectors up to half the
    // last class leaves room for longer mean fields and distortions (windows
    // beyond the last class are solved in FP64, one by one).
    return layer_sites(m) <= 16 && unit_bound(m) <= 0.5 * kFermiMaxX;
}

static cudaError_t launch(RsMode mode, const StageArgs& a, int c0, const RsDevice& dev, cudaStream_t st) {
    static const FermiNodes tab[kFermiClasses] = {PTCA_FERMI_NODES};
    const int M = class_nodes(tab, unit_bound(a.m)), ms = window_sites(a.m);
    const bool uniform = a.m.lattice_periodic;
    return with_tile(a.m, [&](auto tile, auto pairs) {
        using Tl = decltype(tile);
        constexpr bool kPairs = decltype(pairs)::value;
        const RsStagePlan p = rs_stage_plan<Tl, kPairs>(M, ms, uniform, a.count, dev.sms, dev.smem - kRsStatic);
        return launch_chained(k_stage_rs<Tl, kPairs>, (a.count + p.vb - 1) / p.vb, 32 * p.nw, p.bytes, st, a, p.vb, ms,
                              uniform, mode, c0);
    });
}

cudaError_t launch_stage_resolvent(const StageArgs& a, bool few, const RsDevice& dev, cudaStream_t st) {
    if (a.count <= 0) return cudaSuccess;
    return few ? launch_groups(RS_STAGE, a, 0, dev.sms, st) : launch(RS_STAGE, a, 0, dev, st);
}

cudaError_t launch_check_resolvent(const StageArgs& a, bool few, int c0, int count, double* F,
                                   const RsDevice& dev, cudaStream_t st) {
    if (count <= 0) return cudaSuccess;
    StageArgs b = a;
    b.Fbuf = F - 2 * (int64_t)c0;
    b.count = count;
    b.perm = nullptr;
    b.count_dev = nullptr;
    b.prev_count = b.prev2_count = 0;
    return few ? launch_groups(RS_CHECK, b, c0, dev.sms, st) : launch(RS_CHECK, b, c0, dev, st);
}

}  // namespace ptca

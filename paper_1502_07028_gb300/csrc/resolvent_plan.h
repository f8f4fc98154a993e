// resolvent_plan.h -- host rules of the determinant sweeps (resolvent.cuh):
// which problems they serve and how a window is laid out.
#pragma once

#include <cmath>

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

// Allow a kernel all the dynamic shared memory of the device.
template <class K> cudaError_t allow_smem(K kernel, size_t smem_limit) {
    cudaFuncAttributes attr;
    cudaError_t e = cudaFuncGetAttributes(&attr, kernel);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(smem_limit - attr.sharedSizeBytes));
    return e;
}

}  // namespace ptca

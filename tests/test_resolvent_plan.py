"""Launch shapes of the determinant kernels (csrc/resolvent_plan.h), evaluated on
the host: the shared memory that a stage, a stage of few visits and a re-solve
ask for fits a CTA (232448 bytes may be opted into on sm_103a) for every window
that these kernels serve, every node class and any number of visits; and visits
still share a CTA where that fits."""
import os
import subprocess

import pytest

from paper_1502_07028_gb300 import _build

SOURCE = r"""
#include <cstdio>
#include <cstring>
#include "launch.h"
#include "resolvent_plan.h"
using namespace ptca;
int main() {
    static const FermiNodes tab[2][kFermiClasses] = {{PTCA_FERMI_NODES}, {PTCA_FERMI_NODES_DF}};
    const size_t limit = 232448, room = limit - kRsStatic;
    const int sms = 152;
    long plans = 0, over = 0, shared = 0;
    auto check = [&](const char* what, const Model& m, int M, int count, size_t bytes) {
        ++plans;
        if (bytes <= room) return;
        if (++over <= 20) printf("%s: %d dims L_c=%d M=%d count=%d: %zu bytes\n", what, lattice_dims(m), m.Lc, M, count, bytes);
    };
    for (int dims = 1; dims <= 3; ++dims)
        for (int Lc = 2; Lc <= 16; ++Lc)
            for (int per = 0; per < 4; ++per) {
                Model m;
                std::memset(&m, 0, sizeof m);
                m.Lx = 1 << 10; m.Ly = dims > 1 ? 1 << 10 : 1; m.Lz = dims > 2 ? 1 << 6 : 1;
                m.Lc = Lc; m.lattice_periodic = per & 1; m.cluster_periodic = per >> 1;
                m.T = m.t = 1.0;
                if (layer_sites(m) > 16) continue;
                const int ms = window_sites(m), ml = layer_sites(m);
                for (int c = 0; c < kFermiClasses; ++c) {
                    const int M = tab[0][c].M;
                    for (int count : {1, 65, 607, 608, 1215, 1216, 1824, 2432, 3040, 3136, 10000, 1 << 20})
                        with_tile(m, [&](auto tile, auto pairs) {
                            const auto p = rs_stage_plan<decltype(tile), decltype(pairs)::value>(M, ms, m.lattice_periodic, count, sms, room);
                            check("stage", m, M, count, p.bytes);
                            if (decltype(tile)::NS == 16 && p.vb > 1) ++shared;
                            return 0;
                        });
                    for (int count = 1; count <= kFewVisits; ++count)
                        with_latency_tile(m, [&](auto tile, auto pairs) {
                            check("few", m, M, count, rs_few_plan<decltype(tile), decltype(pairs)::value>(M, ms, ml, count, sms).bytes);
                            return 0;
                        });
                }
                with_group(m, [&](auto group, auto pairs) {
                    check("re-solve", m, 0, 0, rs_resolve_bytes<decltype(group), decltype(pairs)::value>(ms, ml));
                    return 0;
                });
            }
    printf("%ld plans, %ld over, %ld share a CTA\n", plans, over, shared);
    return over || !shared;
}
"""


def test_every_launch_fits_the_shared_memory_of_a_cta(tmp_path):
    try:
        nvcc = _build.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    src, exe = tmp_path / "plan.cu", tmp_path / "plan"
    src.write_text(SOURCE)
    subprocess.run([nvcc, *_build.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-O1", "-I", os.path.join(_build.CSRC),
                    str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout

"""What the FP32 screening's error bound of a scene depends on (host code of
the kernels' header, compiled by itself): the extents that a packet can meet,
and not the radius of a source that has none."""
import os
import subprocess

import pytest

import paper_2112_08035_gb300 as smc

CSRC = os.path.join(os.path.dirname(smc.__file__), "csrc")
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "smcrt_internal.h"
int main(int argc, char **argv)
{
    if (argc != 4) return 2;
    smcrt_prim prim{};
    prim.kind = std::atoi(argv[3]);
    prim.p[3] = 1.0;
    prim.p[4] = 0.5;
    smcrt_csg_node node{};
    node.op = SMCRT_OP_PRIM;
    smcrt_region region{};
    region.node_count = 1;
    region.mu_s = region.n = 1.0;
    smcrt_scene sc{};
    sc.prims = &prim; sc.nprims = 1;
    sc.nodes = &node; sc.nnodes = 1;
    sc.regions = &region; sc.nregions = 1;
    sc.ambient_n = 1.0; sc.delta = 1e-6; sc.max_steps = 100;
    smcrt_grid g{};
    for (int a = 0; a < 3; ++a) { sc.bbox_lo[a] = g.lo[a] = -2.0; sc.bbox_hi[a] = g.hi[a] = 2.0; g.n[a] = 8; }
    smcrt_source src{};
    src.kind = std::atoi(argv[1]);
    src.radius = std::atof(argv[2]);
    src.dir[2] = -1.0;
    const smcrt::Instr ins{};
    const int2 rr = make_int2(0, 1);
    smcrt::DevScene H{};
    smcrt::fill_screen(H, &sc, &src, &g, &ins, &rr);
    std::printf("%.9g %d %d\n", H.feps, H.tfix, smcrt::walk_bits(smcrt::screen_range(&sc, &src)));
}
"""


@pytest.fixture(scope="module")
def bound(tmp_path_factory):
    d = tmp_path_factory.mktemp("screen")
    src, exe = str(d / "screen.cpp"), str(d / "screen")
    with open(src, "w") as f:
        f.write(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", f"-I{CSRC}", f"-I{CUDA}/include", src, "-o", exe])

    def run(kind, radius, prim=SPHERE):
        feps, tfix, walk = subprocess.check_output([exe, str(kind), repr(radius), str(prim)], text=True).split()
        assert tfix == walk                      # the image has the planes where the kernel walks with them
        return float(feps), int(tfix)

    return run


PENCIL, DISC, SQUARE, ISO_POINT = range(4)
SPHERE, TORUS = 0, 3


@pytest.mark.parametrize("kind", [PENCIL, ISO_POINT])
@pytest.mark.parametrize("radius", [-1e3, 1e3, 1e13, float("inf"), float("nan")])
def test_a_source_without_a_radius_leaves_the_bound_alone(bound, kind, radius):
    assert bound(kind, radius) == bound(kind, 0.0)


@pytest.mark.parametrize("kind", [DISC, SQUARE])
def test_a_source_with_a_radius_counts(bound, kind):
    narrow, wide, off = bound(kind, 0.5), bound(kind, 32.0), bound(kind, 1e13)
    assert narrow == bound(kind, 1.0)            # inside the volume of interest
    assert 15.9 < wide[0] / narrow[0] < 16.1     # 32 against the box's 2
    assert off == (0.0, 0)                       # beyond the screening's range


def test_general_shapes_have_no_screening_and_no_planes(bound):
    assert bound(PENCIL, 0.0, TORUS) == (0.0, 0)


def test_the_fixed_point_walk_ends_before_the_screening(bound):
    """The walk's unit is 2^-58 of the range and no coarser than 2^-40."""
    assert bound(SQUARE, 2.0 ** 18 - 1.0)[1] == 40
    assert bound(SQUARE, 2.0 ** 19)[1] == 0 and bound(SQUARE, 2.0 ** 19)[0] > 0.0

"""How the search counts a tiling's rows, finds its blocks' least words and bounds its keys, compiled for the CPU, against the same
by blocks and classes of levels, which test_host_math.py checks against the oracle's rows."""
import ctypes as C
import os
import subprocess

import pytest

import mmee_inputs as mi
import paper_2604_03446_b200.binding as mm
from paper_2604_03446_b200 import build as lib_build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("host_tiling") / "host_tiling.so")
    flags = [f for f in lib_build.NVCC_FLAGS if f not in ("-lineinfo", "-O3")]
    subprocess.check_call([lib_build._nvcc()] + flags + ["-O1", "-o", out, os.path.join(HERE, "host_tiling.cu")] +
                          [os.path.join(lib_build.CSRC, f) for f in ("mmee_plan.cu", "mmee_prune.cu")])
    return C.CDLL(out)


# (I, K, L, J), tilings from one to the next: bounds of one, equal operands, sizes that saturate at 2^30 - 1 words
@pytest.mark.parametrize("dims,stride", [((12, 4, 20, 6), 1), ((7, 5, 1, 3), 1), ((16, 16, 16, 16), 1), ((1, 1, 1, 1), 1),
                                         ((30, 12, 8, 18), 7), ((65536, 128, 65536, 128), 101), ((32768, 16384, 4096, 4096), 211)])
@pytest.mark.parametrize("order_set", [mi.ORD_ALL6, mi.ORD_NORECOMP2])
@pytest.mark.parametrize("fuse_mask", [mi.FUSE_ALL, mi.FUSE_FUSED, mi.FUSE_SEPARATE, mi.FUSE_SOFTMAX_IN_OP1 | mi.FUSE_SEPARATE])
def test_tilings_against_blocks_and_classes(host, dims, stride, order_set, fuse_mask):
    w = mi.workload(1, 1, 1, dims[0], dims[2], dims[1], dims[3], 1)
    o = mi.objective(mi.OBJ_ENERGY, 1, order_set=order_set, fuse_mask=fuse_mask, row_pruning=1)
    whole = sum(dims[i] * dims[j] for i, j in ((0, 1), (1, 2), (0, 2), (2, 3), (0, 3)))
    # from a capacity at which nothing fits to one at which every row does (or the largest that is accepted)
    caps = sorted({min(2 ** 30 - 2, max(1, int(whole * f))) for f in (0, 1e-4, 1e-2, 0.05, 0.1, 0.2, 0.3, 0.45, 0.6, 0.8, 1.0)})
    for cap in caps:
        a = mi.arch(2, 3, 1, cap, 0, 1, 1.0, 0.0, 0.0, 0.0)
        at = C.c_uint64()
        args = [C.byref(mm._fill(s(), d)) for s, d in ((mm.Workload, w), (mm.Arch, a), (mm.Objective, o))]
        assert host.host_tilings(*args, C.c_uint32(stride), C.byref(at)) == mm.OK, (cap, at.value)

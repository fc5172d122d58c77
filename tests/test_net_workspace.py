"""Host-only facts of the warm-start network's C ABI: the group limit is one number in the header and the binding,
and the workspace query names what the gradients' partial sums take (no GPU needed)."""
import ctypes as C
import os
import re
import shutil

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    if shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"):
        pytest.skip("nvcc not available")
    from paper_2011_06842_gb300 import build
    build.build()
    from paper_2011_06842_gb300 import fewha
    fewha.load_library()
    return fewha


def net(fewha, groups, channels=(4, 32, 5)):
    N = fewha.NET()
    N.C0, N.C, N.C3 = channels
    N.ngroups = len(groups)
    for i, (count, side) in enumerate(groups):
        N.count[i], N.side[i] = count, side
    return N


def test_one_group_limit(lib):
    text = open(os.path.join(ROOT, "include", "fewha.h")).read()
    assert int(re.search(r"#define FEWHA_NET_GROUPS (\d+)", text).group(1)) == lib.NET_GROUPS == len(lib.NET().count)


@pytest.mark.parametrize("groups,channels", [([(1, 8)], (4, 32, 5)), ([(5, 128), (4, 64)], (4, 32, 5)),
                                             ([(2, 17), (1, 1)], (40, 3, 50)), ([(16, 128)] * 8, (1, 1, 1))])
def test_workspace_holds_the_partials(lib, groups, channels):
    """One partial per 16 x 16 tile, at most one per CTA of the launch (152), of the largest of the three gradients;
    no less than a single convolution's own query asks for below that number."""
    L, (c0, c, c3) = lib.load_library(), channels
    got = L.fewha_convnet_workspace(C.byref(net(lib, groups, channels)))
    tiles = sum(n * ((s + 15) // 16) ** 2 for n, s in groups)
    for ci, co in ((c0, c), (c, c), (c, c3)):
        assert got >= min(152, tiles) * (9 * ci * co + co)
    if tiles <= 152 and len(groups) == 1:
        (n, s), = groups
        assert got >= max(L.fewha_conv3x3_wgrad_workspace(ci, co, n, s, s) for ci, co in ((c0, c), (c, c), (c, c3)))


def test_invalid_networks_have_no_workspace(lib):
    L = lib.load_library()
    assert L.fewha_convnet_workspace(None) == 0
    assert L.fewha_convnet_workspace(C.byref(net(lib, [(0, 8)]))) == 0
    assert L.fewha_convnet_workspace(C.byref(net(lib, [(1, 8)], (4, 0, 5)))) == 0
    N = net(lib, [(1, 8)])
    N.ngroups = lib.NET_GROUPS + 1
    assert L.fewha_convnet_workspace(C.byref(N)) == 0

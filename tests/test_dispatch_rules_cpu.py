"""The rules on sizes that choose how a call is launched, asked on the host (dispatch_rules_host.cpp): at sizes where both ways
were measured, they have to name the faster one."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SMS = 148


@pytest.fixture(scope="module")
def ask(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    exe = str(tmp_path_factory.mktemp("rules") / "rules")
    subprocess.run([gxx, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2609_19242_b200", "csrc"),
                    os.path.join(ROOT, "tests", "dispatch_rules_host.cpp"), "-o", exe], check=True)
    return lambda rule, *sizes: [int(x) for x in subprocess.run([exe, rule, *map(str, sizes)], check=True, capture_output=True,
                                                                 text=True, timeout=60).stdout.split()]


@pytest.mark.parametrize("batch,L,H_kv,window,fused,dkdv", [
    (1, 8192, 8, 0, 1, 1),        # few stacks of tiles: the heavy tiles of all heads first
    (2, 8192, 4, 0, 1, 1),
    (1, 11264, 8, 0, 1, 1),
    (1, 12288, 8, 0, 1, 1),
    (2, 7168, 8, 0, 0, 1),        # dQ accumulators stay in L2 only while neighbouring tiles of one head run together
    (3, 10240, 4, 0, 0, 1),
    (1, 16384, 8, 0, 0, 0),
    (3, 6144, 8, 0, 0, 0),
    (2, 10240, 8, 0, 0, 0),
    (1, 32768, 8, 0, 0, 0),
    (1, 8192, 8, 7500, 1, 1),     # a window: no tile is much heavier than the others
    (1, 8192, 8, 5200, 0, 1),
    (1, 12288, 8, 4096, 0, 0),
    (2, 12000, 4, 3500, 0, 0),
    (1, 8192, 8, 8192, 1, 1),     # one that cuts nothing off
])
def test_start_order_of_pairs(ask, batch, L, H_kv, window, fused, dkdv):
    units = (-(-L // 256), H_kv, 2 * batch, window, SMS)
    assert ask("order_pairs", *units, 1) == [fused]
    assert ask("order_pairs", *units, 0) == [dkdv]


@pytest.mark.parametrize("nx,stacks,want", [(64, 16, 1), (91, 16, 1), (92, 16, 0), (256, 16, 0)])
def test_start_order_of_one_cta_per_tile(ask, nx, stacks, want):
    """Exactly 10 SMs > stacks (nx + 1)."""
    assert (10 * SMS > stacks * (nx + 1)) == bool(want)
    assert ask("order", nx, stacks, 1, SMS) == [want]

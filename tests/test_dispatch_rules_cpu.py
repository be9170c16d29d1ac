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
    assert ask("order_pairs", batch, L, L, 0, L, H_kv, 4, window, 0, SMS) == [fused, dkdv]


@pytest.mark.parametrize("L,H_kv,G,Lq,Ln,fused,dkdv", [
    (9984, 8, 3, 0, 19712, 1, 1), (10240, 8, 2, 8000, 19200, 1, 1),   # more noisy rows than clean keys
    (12288, 8, 4, 0, 32768, 0, 1), (8192, 8, 8, 0, 20480, 0, 1), (16384, 8, 4, 0, 32768, 0, 0),
    (20480, 8, 4, 0, 9600, 0, 0),
])
def test_start_order_of_pairs_in_the_packed_form(ask, L, H_kv, G, Lq, Ln, fused, dkdv):
    assert ask("order_pairs", 1, L, Lq, 2000 if Lq else 0, Ln, H_kv, G, 0, 0, SMS) == [fused, dkdv]


@pytest.mark.parametrize("nx,stacks,want", [(64, 16, 1), (91, 16, 1), (92, 16, 0), (256, 16, 0)])
def test_start_order_of_one_cta_per_tile(ask, nx, stacks, want):
    """Exactly 10 SMs > stacks (nx + 1)."""
    assert (10 * SMS > stacks * (nx + 1)) == bool(want)
    assert ask("order", nx, stacks, 1, SMS) == [want]


@pytest.mark.parametrize("L,H,H_kv,window,want", [
    (32768, 32, 8, 0, 1), (6144, 32, 8, 0, 1), (16384, 8, 8, 0, 1), (32768, 32, 8, 4096, 1),
    (4096, 32, 8, 0, 0), (8192, 16, 16, 0, 0), (32768, 32, 8, 2048, 0), (32768, 32, 8, 1024, 0),
])
def test_calls_that_pairs_take(ask, L, H, H_kv, window, want):
    assert ask("pairs", 1, L, L, 0, L, H_kv, H // H_kv, window, 0, SMS) == [1, want]


@pytest.mark.parametrize("L,chunk_tiles,rank_of,blocks,want", [
    (32768, 1, None, True, 0), (16128, 3, None, True, 0), (32640, 3, None, True, 0), (16000, 5, None, True, 0),
    (16128, 7, None, True, 1), (32256, 9, None, True, 1),
    (32768, 16, None, True, 1),                              # an even number of tiles: a pair stays within a chunk
    (11264, 11, (3, 4), True, 0), (26624, 13, (4, 8), True, 1), (65536, 32, (3, 8), True, 1),
    (22528, 11, (7, 8), False, 1), (10240, 5, (7, 8), False, 0),
])
def test_pairs_whose_tiles_stand_far_apart(ask, L, chunk_tiles, rank_of, blocks, want):
    """Gathered K/V: whole-sequence calls (rank_of None), and one rank's first run of clean queries with its blocks or its second
    run by itself."""
    if rank_of is None:
        pos0, Lq, Ln = 0, L, L
    else:
        r, P = rank_of
        pos0, Lq, Ln = ((r if blocks else 2 * P - 1 - r) * L // (2 * P), L // (2 * P), L // P if blocks else 0)
    assert ask("pairs", 1, L, Lq, pos0, Ln, 8, 4, 0, 128 * chunk_tiles, SMS) == [1, want]


@pytest.mark.parametrize("T,D,V,n_run,pair", [
    (8192, 4096, 128256, 1, 1), (12288, 4096, 64000, 1, 1), (8192, 1024, 50304, 1, 1), (1531, 1544, 32008, 1, 1),
    (300, 2048, 100000, 1, 0),           # three tiles of 128 rows, two of 256
    (123, 1048, 49664, 2, 0), (137, 4000, 20272, 2, 1),   # few rounds of items: as even as they get
    (8192, 512, 50304, 8, 1), (2048, 384, 128256, 8, 1),
])
def test_forward_items_of_the_loss_head(ask, T, D, V, n_run, pair):
    assert ask("lce_forward", T, D, V, 1, SMS) == [256, n_run, pair]


@pytest.mark.parametrize("D", [256, 1024, 4096])
def test_forward_items_hold_whole_vocabulary_runs(ask, D):
    """With the smallest workspace a vocabulary run is eight tiles, and an item never less."""
    assert ask("lce_forward", 8192, D, 128256, 8, SMS)[1] == 8


@pytest.mark.parametrize("T,D,V,bn,pair", [
    (2609, 224, 4488, 256, 0), (2146, 240, 8992, 256, 0), (4096, 144, 8000, 256, 0),   # one round of narrow matrices
    (3000, 176, 30000, 256, 1), (4096, 256, 8000, 256, 1), (4096, 248, 8000, 256, 1), (4096, 128, 16000, 128, 1), (4000, 72, 9000, 128, 1),
    (4096, 2048, 50304, 256, 1), (300, 2048, 50304, 256, 0),
])
def test_weight_gradient_of_the_loss_head(ask, T, D, V, bn, pair):
    assert ask("lce_dw", T, D, V, SMS) == [bn, pair]

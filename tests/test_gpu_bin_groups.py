"""The list sorts of the binning at the edges of their sizes (bit-exact against the oracle).

A warp takes four consecutive tiles: all four lists at once up to 8 entries, two up to
16, else one by one with 1, 2, 4 or 8 entries per lane, and leaves longer ones to its block.
"""
import numpy as np
import pytest

from paper_2412_03451_gb300 import scenes as S

from gpu_cases import gpu_run, oracle_bins

pytestmark = pytest.mark.gpu

EDGES = {
    "eights": [8, 7, 0, 1, 8, 8, 8, 8, 0, 0, 0, 0, 3],
    "sixteens": [9, 3, 0, 16, 16, 16, 15, 1, 8, 8, 8, 9, 16, 2, 0],
    "mixed": [17, 2, 8, 8, 0, 16, 33, 0, 32, 31, 1, 1],
    "registers": [64, 65, 0, 5, 128, 129, 2, 256],
    "block": [257, 0, 300, 16, 4, 511, 513],
}


@pytest.mark.parametrize("case", sorted(EDGES))
def test_lists_at_sort_edges(case):
    pytest.importorskip("torch")
    counts = EDGES[case]
    rng = np.random.default_rng(len(counts))
    f, depth, c = 100.0, [], []
    for t, n in enumerate(counts):
        z = rng.uniform(1.0, 4.0, n)
        z[1::3] = z[: len(z[1::3])]                        # equal keys: the record id decides
        u = 8 * t + 4 + rng.uniform(-0.4, 0.4, n)
        v = 4 + rng.uniform(-0.4, 0.4, n)
        c.append(np.stack([(u - 4 * len(counts)) / f * z, (v - 4) / f * z, z], 1))
    c = np.concatenate(c)
    order = rng.permutation(len(c))
    p = S.Planes(c[order].astype(np.float32), np.tile(np.float32([1, 0, 0, 0]), (len(c), 1)),
                 np.full((len(c), 4), 0.002, np.float32))
    cams = S.identity_cameras(1, 8, 8 * len(counts), f)
    g = gpu_run(p, cams, 300.0, tile=(8, 8))
    rect, key32, ptr, ent, ekey = oracle_bins(p, cams, g["delta"], (8, 8))
    assert list(np.diff(ptr)) == counts
    assert g["status"] == 0 and g["required"] == len(ent)
    assert np.array_equal(g["tile_ptr"], ptr)
    assert np.array_equal(g["tile_ent"], ent)
    assert np.array_equal(g["tile_key"].view(np.uint32), ekey.view(np.uint32))

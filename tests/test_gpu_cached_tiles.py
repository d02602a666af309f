"""Every tile budget that the autotuner's cache file may hold gives the same K to rounding.

The file is text that a user can edit: budgets from one double up to the largest candidate are taken.
A budget below one staged block is raised to it; the heavy species have blocks of 39 x 39 functions.
"""
import dataclasses

import numpy as np
import pytest

import rix_inputs as ri

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2403_10343_gb300.rix import Exchange  # noqa: E402


def _system(kind):
    if kind == "waters":
        return ri.water_cluster(2, 6, cutoff=False)
    return dataclasses.replace(ri.perovskite(1, 1, 1, 31), cutoff=ri.ang2bohr(3.0))


@pytest.mark.parametrize("kind", ["waters", "heavy"])
def test_budgets_of_the_cache_file(tmp_path, kind):
    s = _system(kind)
    pk = ri.generate(s)
    ex = Exchange.from_system(s)
    D = torch.from_numpy(pk.D).cuda()
    ex.set_CV(torch.from_numpy(pk.C).cuda(), torch.from_numpy(pk.V).cuda())
    K0 = ex.build_K(D).cpu().numpy()
    cache = tmp_path / "tiles.txt"
    ex.autotune(D, str(cache))
    key = cache.read_text().split()[0]
    for tiles in ((1, 1, 1), (300, 700, 300), (4096, 1521, 4096), (16384, 16384, 16384)):
        cache.write_text(f"{key} {tiles[0]} {tiles[1]} {tiles[2]}\n")
        assert tuple(ex.autotune(D, str(cache))) == tiles
        K = ex.build_K(D).cpu().numpy()
        # sums of the same products in another order: 1e3 terms, far inside the FP64 path's 1e-12
        assert np.linalg.norm(K - K0) <= 1e-13 * np.linalg.norm(K0)
    ex.close()

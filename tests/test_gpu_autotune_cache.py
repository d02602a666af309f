"""Tile choices in the autotuner's cache file belong to the kernels that they were timed with."""
import pytest

import rix_inputs as ri


@pytest.mark.gpu
def test_choices_of_earlier_kernels_are_not_taken(tmp_path):
    torch = pytest.importorskip("torch")
    from paper_2403_10343_gb300.rix import Exchange
    s = ri.water_cluster(2, 5, cutoff=False)
    pk = ri.generate(s)
    cache = tmp_path / "tiles.txt"
    ex = Exchange.from_system(s)
    D = torch.from_numpy(pk.D).cuda()
    ex.set_CV(torch.from_numpy(pk.C).cuda(), torch.from_numpy(pk.V).cuda())
    ex.autotune(D, str(cache))
    key = cache.read_text().split()[0]
    assert "|k2|" in key
    old = key.replace("|k2|", "|") + " 12288 16000 12288\n"
    cache.write_text(old)
    chosen = ex.autotune(D, str(cache))
    assert all(c in (4096, 8192, 12288, 16384) for c in chosen)
    lines = cache.read_text().splitlines()
    assert len(lines) == 2 and lines[0] + "\n" == old and lines[1].split()[0] == key
    ex.close()

"""rix_fit_C over the metric sizes and column counts of its launch classes.

The fit keeps a pair's triangle in shared memory up to 158 aux functions and in a workspace above,
solves eight rows at a time with a remainder, and launches by the number of (i, j) columns.  Heavy
pairs (280 aux functions, 1,521 columns), odd sizes around the eight-row blocks and the shared-memory
limit, and single functions are compared with the oracle's fit; the tolerance is the metric's
condition number times rounding, as for any backward-stable solve.
"""
import dataclasses

import numpy as np
import pytest

import rix_inputs as ri
import rix_inputs.systems as S
from oracle.rifit import fit_C, metric

from rifit_systems import eri_from

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2403_10343_gb300 import rix  # noqa: E402

LAM = 1e-3


def _waters(nbas, naux):
    xyz, spc = S._waters(np.array([[0.0, 0.0, 0.0], [2.8, 0.2, -0.1]]), 3)
    rng = np.random.default_rng(4)
    return S.System(name="sizes", seed=3, xyz=ri.ang2bohr(xyz), species=spc, species_names=["O", "H"],
                    nbas=np.array(nbas, np.int32), naux=np.array(naux, np.int32),
                    sigma=[np.sort(0.3 * 10.0 ** rng.random(n)) for n in naux], cell=None, cutoff=0.0, tau=0.0,
                    orbital_centres=np.zeros(5, np.int32))


def _system(kind):
    if kind == "heavy":
        s = S.perovskite(1, 1, 1, 31)
        return dataclasses.replace(s, cutoff=ri.ang2bohr(4.0))
    return _waters(*kind)


@pytest.mark.parametrize("kind", ["heavy", ((1, 1), (1, 1)), ((3, 2), (7, 9)), ((14, 5), (79, 80)),
                                  ((6, 17), (158, 8)), ((16, 1), (159, 3))], ids=str)
def test_fit_sizes(kind):
    s = _system(kind)
    pk = ri.generate(s)
    eri = eri_from(s, pk, pk.C)
    ex = rix.Exchange.from_system(s)
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()  # noqa: E731
    V = dev(pk.V)
    C = rix.fit_C(ex.ctx, V, dev(eri), LAM)
    got, ref = C.cpu().numpy(), fit_C(s, pk, eri, LAM)
    cond = max(np.linalg.cond(metric(s, pk, p, LAM)) for p in range(pk.n_pairs))
    assert np.abs(got - ref).max() <= 100 * cond * 2.0 ** -52 * np.abs(ref).max()
    ex.set_CV(C, V)  # exactly pair-symmetric
    ex.close()

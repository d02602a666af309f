"""Term 4 halved over the pairs {B, G'} of Z or over the K blocks, against the oracle.

The build evaluates half of the symmetric term 4 in one of two ways, chosen at setup from the
estimated cost: clusters and mixed builds take Z over unordered pairs, small periodic cells in
FP64 (many K blocks per pair) take the K blocks in one orientation.  Atoms are put in an order
that mixes the species, so the representative pairs run from light to heavy atoms and back,
and the periodic cells have on-site pairs, self-images and molecules cut by the cell faces.
Row blocks split Z by its row atoms.
"""
import dataclasses

import numpy as np
import pytest

import rix_inputs as ri
import rix_inputs.systems as S
from oracle.oracle import exchange

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2403_10343_gb300.rix import Exchange  # noqa: E402


def _reordered(s, order):
    """The same system with its atoms in another order."""
    order = np.asarray(order)
    back = np.argsort(order)
    return dataclasses.replace(s, xyz=s.xyz[order], species=s.species[order],
                               orbital_centres=back[s.orbital_centres].astype(np.int32))


def _system(kind):
    if kind == "cluster":
        s = ri.water_cluster(2, 6, cutoff=False)
        s = dataclasses.replace(s, xyz=s.xyz[:9], species=s.species[:9], orbital_centres=s.orbital_centres[:15])
        return _reordered(s, [1, 3, 0, 8, 4, 6, 2, 5, 7])
    o = np.array([[1.0, 1.2, 0.8], [3.9, 3.1, 3.3]])[:1 if kind == "periodic1" else 2]
    side, cut = (4.6, 4.8) if kind == "periodic1" else (6.0, 4.0)
    xyz, spc = S._waters(o, 11)
    names = ["O", "H"]
    nb, na = S._species_arrays(names)
    s = S.System(name=kind, seed=11, xyz=ri.ang2bohr(xyz), species=spc, species_names=names, nbas=nb, naux=na,
                 sigma=S._aux_widths(11, names), cell=ri.ang2bohr(np.eye(3) * side), cutoff=ri.ang2bohr(cut), tau=0.0,
                 orbital_centres=np.repeat(np.arange(0, len(spc), 3), 5).astype(np.int32))
    return _reordered(s, [1, 0, 2] if kind == "periodic1" else [4, 1, 0, 3, 5, 2])


@pytest.mark.parametrize("opts", [dict(precision="fp64"), dict(precision="mixed"),
                                  dict(precision="mixed", deterministic=1),
                                  dict(precision="fp64", block_atoms=2), dict(precision="mixed", block_atoms=2)],
                         ids=lambda o: "-".join(f"{k}={v}" for k, v in o.items()))
@pytest.mark.parametrize("kind", ["cluster", "periodic1", "periodic2"])
def test_term4_halves_match_the_oracle(kind, opts):
    s = _system(kind)
    pk = ri.generate(s)
    keys, K_ref, E_ref, _ = exchange(s, pk)
    ex = Exchange.from_system(s, **opts)
    assert np.array_equal(ex.k_keys(), keys)
    ex.set_CV(torch.from_numpy(pk.C).cuda(), torch.from_numpy(pk.V).cuda())
    D = torch.from_numpy(pk.D).cuda()
    K = ex.build_K(D)
    E = ex.energy(D, K).item()
    rel = np.linalg.norm(K.cpu().numpy() - K_ref) / np.linalg.norm(K_ref)
    # the bars of the FP64 and the mixed path
    if opts["precision"] == "fp64":
        assert rel < 1e-12 and abs(E - E_ref) < 1e-12 * abs(E_ref)
    else:
        assert rel < 1e-8 and abs(E - E_ref) < 1e-6
    ex.close()

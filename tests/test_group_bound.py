"""How long the sliced GEMM may accumulate: the bound on a diagonal's partial sums.

With a_s, b_u the digits of a row and a column, every partial sum of a diagonal over any part of K is
at most sum_k sum_{s+u=d} |a_s||b_u| <= sqrt(W_a W_b), W the sum of the squares of all digits
(Cauchy-Schwarz).  A tile whose largest W_a W_b is below 2^48 keeps every sum below 2^24, exact in FP32,
and is accumulated in one group; the kernel keeps the fixed groups of 576 K values otherwise.
The GPU test runs builds on both sides of the rule.
"""
import dataclasses

import numpy as np
import pytest

import rix_inputs as ri


def digits(rng, kind, S, K):
    if kind == "extreme":       # the largest digits a number can have
        return np.stack([np.full(K, 128)] + [np.full(K, -64)] * (S - 1))
    if kind == "dense":
        return np.concatenate([rng.integers(0, 128, (1, K)), rng.integers(-64, 64, (S - 1, K))])
    d = np.concatenate([rng.integers(0, 128, (1, K)), rng.integers(-64, 64, (S - 1, K))])
    return d * (rng.random(K) < 0.3)  # sparse rows


@pytest.mark.parametrize("S", [1, 3, 5, 6])
@pytest.mark.parametrize("kinds", [("extreme", "extreme"), ("dense", "extreme"), ("dense", "dense"),
                                   ("sparse", "dense")])
def test_rule_keeps_every_partial_sum_exact(S, kinds):
    rng = np.random.default_rng(S)
    taken = 0
    for K in (64, 500, 1024, 1100, 2000, 4000):
        a, b = (digits(rng, k, S, K).astype(np.int64) for k in kinds)
        if (a * a).sum() * (b * b).sum() >= 2 ** 48:
            continue
        taken += 1
        for d in range(S):
            terms = sum(np.abs(a[s] * b[d - s]) for s in range(d + 1))
            assert terms.sum() < 2 ** 24
    assert taken > 0


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["generated", "extreme"])
def test_builds_on_both_sides_of_the_rule(kind):
    """36 waters, K of 864 to 944 per problem: the generated data stay below the bound; blocks of equal
    entries 63 sum_t 2^-7t make every digit 63 and exceed it.  Mixed bar: 1e-8 of the FP64 build."""
    torch = pytest.importorskip("torch")
    from paper_2403_10343_gb300.rix import Exchange
    s = ri.water_cluster(4, 5, cutoff=False)
    s = dataclasses.replace(s, xyz=s.xyz[:108], species=s.species[:108], orbital_centres=s.orbital_centres[:180])
    pk = ri.generate(s)
    C, D = pk.C, pk.D
    if kind == "extreme":
        v = sum(63.0 * 2.0 ** (-7 * t) for t in range(1, 7))
        C = np.where(pk.C < 0, -v, v)
        D = np.where(pk.D < 0, -v, v)
    K = []
    for prec in ("fp64", "mixed"):
        ex = Exchange.from_system(s, precision=prec)
        ex.set_CV(torch.from_numpy(C).cuda(), torch.from_numpy(pk.V).cuda())
        K.append(ex.build_K(torch.from_numpy(D).cuda()).cpu().numpy())
        ex.close()
    assert np.linalg.norm(K[1] - K[0]) < 1e-8 * np.linalg.norm(K[0])

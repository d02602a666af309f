"""Both sides of the accumulation rule of the tensor-core plans, counted and exact.

A tile is accumulated in one group where the sums of squares of its operands' digits keep every
partial sum below 2^24, and in groups of 512 K values otherwise.  32 atoms with one aux and 64 basis
functions each, D the identity, V the identity and C zero except in the row and column of atom 0, make

    K(0, 0)[i][l] = sum_{G, k} C(0, G)[i][k] C(0, G)[l][k]   (K = 2,048 in the term-1 plan)

with one product per value in every other plan.  C holds 42-bit numbers given by their six digits; one
entry of 3/4 per row fixes the row's exponent, so the digits are the given ones.  Atoms 16 to 30 repeat
atoms 1 to 15 with the opposite sign for half of the functions, so that the leading parts cancel between
the two halves of the functions and the result is an exact integer of the last kept diagonal's units, in
which a single unit lost by too long a group shows.  With digits near 60 the sums of one group would
pass 2^24; with digits up to 20 they stay below it.
"""
import numpy as np
import pytest

import rix_inputs as ri

NAT, NB, S = 32, 64, 6
HALF = 15 * NB


def digits(kind):
    """Digits [S, NB, 31 NB] of the entries C(0, G)[i][k], G = 1 .. 31, and their signs [NB, 31 NB]."""
    rng = np.random.default_rng(5)
    lo, hi = (58, 64) if kind == "large" else (-20, 21)
    d = np.zeros((S, NB, (NAT - 1) * NB), np.int64)
    d[:, :, :HALF] = rng.integers(lo, hi, (S, NB, HALF))
    d[0, :, :HALF] = np.abs(d[0, :, :HALF])  # the leading digit carries no sign
    d[:, :, HALF:2 * HALF] = d[:, :, :HALF]
    d[2:, :, HALF:HALF + 100] = rng.integers(lo, hi, (S - 2, NB, 100))
    d[0, :, 2 * HALF] = 96
    sign = np.ones((NB, (NAT - 1) * NB), np.int64)
    sign[NB // 2:, HALF:2 * HALF] = -1
    return d, sign


def kept(d, sign, n):
    """The six diagonals over the first n values, exact integers [S, NB, NB]."""
    x = d[:, :, :n] * sign[:, :n]
    return np.stack([sum(x[s] @ x[a - s].T for s in range(a + 1)) for a in range(S)])


def test_operands_lie_on_both_sides():
    """The sums of squares decide as the kernel's bound does, and the large digits need the short groups."""
    for kind in ("large", "small"):
        d, sign = digits(kind)
        W = (d ** 2).sum(axis=(0, 2))
        part = np.abs(kept(d, sign, HALF)).max(axis=(1, 2))
        if kind == "large":
            assert W.min() ** 2 > 2 ** 48 and part[5] > 2 ** 24
        else:
            assert W.max() ** 2 < 2 ** 48 and part.max() < 2 ** 24


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["large", "small"])
def test_group_count_and_exact_result(kind):
    torch = pytest.importorskip("torch")
    from paper_2403_10343_gb300 import rix
    xyz = 6.0 * np.stack(np.meshgrid(*[np.arange(4.0)] * 3, indexing="ij"), -1).reshape(-1, 3)[:NAT]
    ex = rix.Exchange(xyz, np.zeros(NAT, np.int32), [NB], [1], precision="mixed", profile=2)
    keys, offC = rix.layout(ex.ctx, rix.RIX_LIST_C)
    offV, offD = (rix.layout(ex.ctx, w)[1] for w in (rix.RIX_LIST_V, rix.RIX_LIST_D))
    A, B, _ = ri.unpack_key(keys)
    d, sign = digits(kind)
    a = np.tensordot(2.0 ** (-7.0 * np.arange(1, S + 1)), d.astype(float), 1) * sign
    C, V, D = np.zeros(ex.c_elems), np.zeros(ex.v_elems), np.zeros(ex.d_elems)
    for p in range(len(keys)):
        if A[p] == B[p]:
            V[offV[p]] = 1.0
            D[offD[p]:offD[p + 1]] = np.eye(NB).ravel()
        elif A[p] == 0:  # aux of atom 0 first
            C[offC[p]:offC[p] + NB * NB] = a[:, (B[p] - 1) * NB:B[p] * NB].ravel()
        elif B[p] == 0:  # aux of atom A first, then atom 0's
            C[offC[p] + NB * NB:offC[p + 1]] = a[:, (A[p] - 1) * NB:A[p] * NB].T.ravel()
    ex.set_CV(C, V)
    K = ex.build_K(torch.from_numpy(D).cuda())
    tiles, groups = rix.gemm_groups(ex.ctx)
    kkeys, offK = rix.layout(ex.ctx, rix.RIX_LIST_K)
    x = int(np.searchsorted(kkeys, ri.pack_key(0, 0, np.zeros(3, np.int64))))
    K00 = K[offK[x]:offK[x + 1]].cpu().numpy().reshape(NB, NB)
    assert ex.stats()["flops_term1_tc"] > 0 and tiles > 0
    # one tile, of term 1 for atom 0, has 128 stages of products: four groups of 32 stages, or one
    assert groups - tiles == (3 if kind == "large" else 0)
    units = sum(q * 128 ** (S - 1 - n) for n, q in enumerate(kept(d, sign, d.shape[2])))  # of 2^-49
    i, l = slice(0, NB // 2), slice(NB // 2, NB)
    assert np.abs(units[i, l]).max() < 2 ** 53
    assert np.array_equal(K00[i, l], units[i, l] * 2.0 ** -49)
    assert np.array_equal(K00[l, i], units[l, i] * 2.0 ** -49)
    ex.close()

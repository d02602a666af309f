"""The fixed accumulation group of the sliced GEMM: every diagonal of six slices stays exact.

The kernel adds digit products of up to GROUP stages of KC K values in FP32 before it folds them into
64-bit integers.  With six slices each accumulator holds one diagonal; the sixth has the largest bound,
2 * 128 * 64 + 4 * 64 * 64 = 2^15 per K value, so 512 K values stay within 2^24, where FP32 is exact.
The constants are read from the kernel's source, so that this file cannot check another group than the
one that runs.  The GPU test has digits near their extremes, whose sums over more than 527 K values
pass 2^24, and a second half that cancels the leading diagonals: the result is an exact integer far
below 2^53 units of the last kept diagonal, and a single lost unit shows.
"""
import os
import re

import numpy as np
import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2403_10343_gb300", "csrc",
                   "rix_tc.cu")
S = 6


def _constant(name):
    return int(re.search(rf"^constexpr int {name} = (\d+);", open(SRC).read(), re.M).group(1))


def _group():
    return _constant("KC") * _constant("GROUP")  # K values


def diagonals(dA, dB):
    """The S kept diagonals of digits dA [S, M, K], dB [S, K, N], exact integers [S, M, N]."""
    return np.stack([sum(dA[s] @ dB[d - s] for s in range(d + 1)) for d in range(S)])


def test_group_keeps_all_six_diagonals_exact():
    bound = [128 * 128 if d == 0 else 2 * 128 * 64 + (d - 1) * 64 * 64 for d in range(S)]
    assert max(bound) * _group() <= 2 ** 24


def operands(K=1152, M=130, N=90):
    """Digits [S, M, K], [S, K, N] and signs [K]: lead 126 or 127, the others 62 or 63; the second half is
    a permutation of the first with the opposite sign, a few of its low digits changed."""
    rng = np.random.default_rng(11)
    h = K // 2
    dA = np.concatenate([rng.integers(126, 128, (1, M, h)), rng.integers(62, 64, (S - 1, M, h))])
    dB = np.concatenate([rng.integers(126, 128, (1, h, N)), rng.integers(62, 64, (S - 1, h, N))])
    p = rng.permutation(h)
    eA, eB = dA[:, :, p].copy(), dB[:, p, :].copy()
    eA[3:, :, :40] = rng.integers(30, 64, (S - 3, M, 40))
    return np.concatenate([dA, eA], 2), np.concatenate([dB, eB], 1), np.repeat([1, -1], h)


def test_operands_see_a_longer_group():
    dA, dB, _ = operands()
    # the sixth diagonal passes 2^24 within the first half, with odd sums, and 512 values do not
    part = [diagonals(dA[:, :, :k], dB[:, :k])[5] for k in (512, 576)]
    assert part[0].max() <= 2 ** 24 < part[1].min() and (part[1] % 2 == 1).any()


@pytest.mark.gpu
def test_every_unit_of_the_sixth_diagonal_is_kept():
    torch = pytest.importorskip("torch")
    from paper_2403_10343_gb300 import rix
    dA, dB, sign = operands()
    scale = 2.0 ** (-7.0 * np.arange(1, S + 1))
    A = np.tensordot(scale, dA.astype(float), 1) * sign  # 42-bit numbers, exact
    B = np.tensordot(scale, dB.astype(float), 1)
    d = diagonals(dA * sign, dB)
    units = sum(d[a] * 128 ** (S - 1 - a) for a in range(S))  # of 2^-49
    assert np.abs(units).max() < 2 ** 53
    C = rix.gemm_sliced(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), S).cpu().numpy()
    assert np.array_equal(C, units * 2.0 ** -49)

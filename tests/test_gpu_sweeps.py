"""The solve's sweeps at the edges of their layouts: one-warp windows of one and two registers a lane
full and one row beyond, CTA-wide windows at whole numbers of warps and around them, the widest band they
take and the next one, orders that end inside a block of 32 steps and inside a window, zeros, infinities,
NaN (the bits that mark an empty hand-over slot among them).  Bit for bit against the oracle."""
import numpy as np
import pytest

import oracle
from test_gpu_backslash import triangle, trsv_gpu
from test_gpu_parity import assert_same_solution, banded, gbtrs_gpu

pytestmark = pytest.mark.gpu

EMPTY = np.array([0xfff8badc0ffee123], dtype=np.uint64).view(np.float64)[0]


def right_hand_sides(n, nrhs, seed):
    B = np.random.default_rng(seed).standard_normal((nrhs, n))
    if nrhs > 1:
        B[1, ::3] = 0.0
        B[1, n // 2:] = -0.0
    if nrhs > 2:
        B[2, n // 2] = EMPTY
        B[2, n // 3] = np.inf
    return B


# (kl, ku): forward windows of kl+1 rows, backward of kl+ku+1
BANDS = [(1, 0), (31, 0), (31, 1), (32, 0), (63, 0), (64, 0), (20, 43), (20, 44), (95, 0), (96, 1), (127, 0), (128, 32),
         (1, 63), (1, 64), (300, 244), (511, 0), (512, 1), (700, 292), (700, 293), (960, 3), (961, 2), (980, 5)]


@pytest.mark.parametrize("kl,ku", BANDS)
@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 64, 97, 1100])
def test_gbtrs_window_edges(n, kl, ku):
    kl, ku = min(kl, n - 1), min(ku, n - 1)
    A = banded(n, kl, ku, seed=n + kl, dist="normal").numpy()
    ABf, ipiv, _, _ = oracle.gbtrf(oracle.dense_to_band(A, kl, ku), kl, ku)
    B = right_hand_sides(n, 3, n)
    assert_same_solution(gbtrs_gpu(ABf, ipiv, kl, ku, B), oracle.gbtrs(ABf, ipiv, kl, ku, B))


@pytest.mark.parametrize("lower", [True, False])
@pytest.mark.parametrize("k", [1, 30, 31, 32, 33, 63, 64, 65, 480, 481, 992, 993])
@pytest.mark.parametrize("n", [2, 33, 64, 200, 1100])
def test_trsv_window_edges(n, k, lower):
    k = min(k, n - 1)
    A = triangle(n, k, lower, seed=n + k, boost=2.0 + 0.2 * k)
    B = right_hand_sides(n, 3, k)
    ref, info = oracle.tbsv_dense(A, lower, k, B)
    got, ginfo = trsv_gpu(A, lower, k, B)
    assert ginfo == info == 0
    assert_same_solution(got, ref)


@pytest.mark.parametrize("what,lost", [(0, -1), (0, 40), (1, 5), (1, 199), (2, 70)])
def test_a_value_that_never_arrives_shows_in_the_result(what, lost):
    """A CTA-wide sweep in which a copied column (0: forward) or the value of a step (1: forward, 2:
    backward) is lost: the waits give up after about a second, every entry formed from it is NaN and the
    status says why."""
    import torch

    from gpu_helpers import DEV
    from paper_2608_22099_gb300 import bandlu
    n, kl, ku = 240, 90, 40
    A = banded(n, kl, ku, seed=3, dist="normal").numpy() + 100.0 * np.eye(n)  # (no interchanges)
    ABf, ipiv, _, _ = oracle.gbtrf(oracle.dense_to_band(A, kl, ku), kl, ku)
    AB, ip = torch.from_numpy(ABf).to(DEV), torch.from_numpy(ipiv).to(DEV)
    b = torch.ones(n, dtype=torch.float64, device=DEV)
    info = torch.zeros(1, dtype=torch.int32, device=DEV)
    assert bandlu.bandlu_selftest_sweep_lost(what, lost, n, kl, ku, AB, ABf.shape[1], ip, b, info) == 0
    torch.cuda.synchronize()
    if lost < 0:
        assert int(info.item()) == 0 and not bool(torch.isnan(b).any())
    else:
        assert int(info.item()) == -bandlu.BANDLU_ERR_TIMEOUT
        # every entry outside the lost step's block takes its multiple; the columns of a block land together
        first = {0: lost // 32 * 32, 1: lost // 32 * 32 + 32, 2: lost // 32 * 32 + 32}[what]
        affected = b[first:] if what < 2 else b.flip(0)[first:]
        assert affected.numel() and bool(torch.isnan(affected).all())


@pytest.mark.parametrize("kl,ku", [(40, 30), (64, 0), (64, 63), (64, 64), (100, 27), (127, 0), (0, 127), (30, 90), (200, 50),
                                   (397, 3)])
@pytest.mark.parametrize("nrhs", [153, 305, 609, 700])
def test_gbtrs_many_right_hand_sides(kl, ku, nrhs):
    """More right-hand sides than SMs, than staged CTAs on the chip, and than sub-partitions."""
    n = 450
    A = banded(n, kl, ku, seed=kl, dist="normal").numpy()
    ABf, ipiv, _, _ = oracle.gbtrf(oracle.dense_to_band(A, kl, ku), kl, ku)
    B = right_hand_sides(n, nrhs, kl + ku)
    assert_same_solution(gbtrs_gpu(ABf, ipiv, kl, ku, B), oracle.gbtrs(ABf, ipiv, kl, ku, B))


@pytest.mark.parametrize("lower", [True, False])
@pytest.mark.parametrize("k", [100, 480, 481, 512, 513, 544, 545])
@pytest.mark.parametrize("nrhs", [152, 153, 400])
def test_trsv_many_right_hand_sides(k, lower, nrhs):
    n = 1100
    A = triangle(n, k, lower, seed=k, boost=2.0 + 0.2 * k)
    B = right_hand_sides(n, nrhs, k)
    ref, info = oracle.tbsv_dense(A, lower, k, B)
    got, ginfo = trsv_gpu(A, lower, k, B)
    assert ginfo == info == 0
    assert_same_solution(got, ref)

"""The register windows of one warp (single matrices and batches) at the edges of what they hold: one
plane of 16 and of 32 lanes full and not, two to nine planes, the first bands beyond them, orders that
end inside a window, ties, zero pivots and NaN.  Bit for bit against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import DEV, gbtrf_gpu
from paper_2608_22099_gb300 import bandlu
from paper_2608_22099_gb300.workloads import make_dense
from test_gpu_parity import assert_parity_with_nan, run_batched

pytestmark = pytest.mark.gpu


def matrices(batch, n, kl, ku, values, lda):
    A = make_dense(n, kl, ku, dist="uniform", seed=17 * n + kl, batch=batch, lda=lda)
    if values == "small integers":  # equal moduli in most columns, and exact zeros among the pivots
        A = torch.sign(A) * torch.floor(2.5 * A.abs())
        A[1, :, min(3, n - 1)] = 0.0
    elif values == "nan and inf":
        A[0, n // 2, n // 2] = float("nan")
        if kl:
            A[1, min(n - 1, n // 2 + 1), n // 2] = float("nan")
            A[2, min(n - 1, n // 2 + 1), n // 2] = float("inf")
    return A


@pytest.mark.parametrize("values", ["uniform", "small integers", "nan and inf"])
@pytest.mark.parametrize("kl,ku", [(0, 0), (1, 1), (2, 2), (3, 0), (1, 6), (0, 15), (3, 4),  # 16 lanes, the first beyond
                                   (3, 3), (1, 14), (0, 31), (5, 5), (3, 12), (4, 4), (4, 20), (7, 1), (8, 8),
                                   (8, 23), (8, 24), (9, 9), (9, 5)])
@pytest.mark.parametrize("n", [61, 128])
def test_batched_register_windows(n, kl, ku, values):
    batch, ldab = 7, 2 * kl + ku + 1
    A = matrices(batch, n, kl, ku, values, n + (kl & 1))
    got = run_batched(A, ldab)
    ref = oracle.dispatch_lu_batched(A[:, :, :n].contiguous().numpy(), ldab)
    for key in ("kl", "ku", "status", "info"):
        assert np.array_equal(got[key], ref[key]), key
    for b in np.nonzero(ref["status"] == 0)[0]:
        assert_parity_with_nan(got["AB"][b], got["ipiv"][b], int(got["info"][b]), ref["AB"][b], ref["ipiv"][b],
                               int(ref["info"][b]))


@pytest.mark.parametrize("values", ["uniform", "small integers", "nan and inf"])
@pytest.mark.parametrize("n", [3, 4, 5, 8, 9, 33, 100])
@pytest.mark.parametrize("kl,ku", [(0, 0), (1, 1), (2, 2), (3, 3), (3, 4), (1, 14), (0, 31), (4, 1)])
def test_single_register_window(n, kl, ku, values):
    kl, ku = min(kl, n - 1), min(ku, n - 1)
    A = matrices(3, n, kl, ku, values, n)
    for b in range(3):
        AB = oracle.dense_to_band(A[b].numpy(), kl, ku, 2 * kl + ku + 3)
        assert_parity_with_nan(*gbtrf_gpu(AB, kl, ku), *oracle.gbtrf(AB, kl, ku)[:3])


@pytest.mark.parametrize("batch", [600, 1300, 1900, 2500, 5000])
@pytest.mark.parametrize("kl,ku", [(2, 2), (2, 3), (4, 4), (6, 6), (7, 7), (4, 27), (8, 8), (8, 23), (9, 9)])
def test_batched_windows_by_the_batch(batch, kl, ku):
    """The same bands in a window or column by column, as the number of warps on the chip has it: one to
    four to a sub-partition with up to nine planes, beyond with one."""
    n, ldab = 35, 2 * kl + ku + 1
    A = make_dense(n, kl, ku, dist="uniform", seed=batch + kl, batch=batch)
    got = run_batched(A, ldab)
    ref = oracle.dispatch_lu_batched(A.numpy(), ldab)
    for key in ("kl", "ku", "status", "info", "ipiv"):
        assert np.array_equal(got[key], ref[key]), key
    assert np.array_equal(got["AB"], ref["AB"])


@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("n,pad", [(31, 0), (31, 1), (40, 1), (64, 2), (65, 3), (129, 1), (256, 1)])
def test_batched_padding_is_not_part_of_the_matrix(n, pad, off):
    """Rows with little padding are scanned as one run, padding and all: NaN there, and an odd base
    address, change nothing."""
    batch, lda, kl, ku = 5, n + pad, 2, 3
    ldab = 2 * kl + ku + 1
    A = make_dense(n, kl, ku, dist="uniform", seed=n, batch=batch)
    A[2, n - 1, 0] = 1.0                      # the last row, far from the diagonal
    A[3, 0, n - 1] = 1.0
    P = torch.full((batch * n * lda + off,), float("nan"), dtype=torch.float64)
    P[off:].view(batch, n, lda)[:, :, :n] = A
    Pd = P.to(DEV)
    AB = torch.full((batch, n, ldab), -3.0, dtype=torch.float64, device=DEV)
    ip = torch.full((batch, n), -1, dtype=torch.int32, device=DEV)
    out = torch.full((4, batch), -1, dtype=torch.int32, device=DEV)
    rc = bandlu.dispatch_lu_batched(Pd.data_ptr() + 8 * off, n, lda, n * lda, batch, AB, ldab, n * ldab, ip, n,
                                    out[0], out[1], out[2], out[3])
    torch.cuda.synchronize()
    ref = oracle.dispatch_lu_batched(A.numpy(), ldab)
    assert rc == 0
    for row, key in zip(out.cpu().numpy(), ("kl", "ku", "info", "status")):
        assert np.array_equal(row, ref[key]), key
    for b in np.nonzero(ref["status"] == 0)[0]:
        assert np.array_equal(AB[b].cpu().numpy(), ref["AB"][b]) and np.array_equal(ip[b].cpu().numpy(), ref["ipiv"][b])


@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("n,pad", [(2, 0), (3, 0), (3, 1), (33, 0), (100, 3), (1001, 0), (1000, 1), (2047, 0), (2048, 7), (2048, 40)])
def test_detect_reads_one_run_of_any_alignment(n, pad, off):
    lda = n + pad
    for (i, j) in ((n - 1, 0), (0, n - 1), (n - 1, n - 1), (n // 2, n // 3), (0, 0)):
        P = torch.full((n * lda + off,), float("nan"), dtype=torch.float64, device=DEV)
        M = P[off:].view(n, lda)[:, :n]
        M.zero_()
        M[i, j] = -1.0
        out = torch.full((2,), -7, dtype=torch.int32, device=DEV)
        assert bandlu.detect_bandwidth(P.data_ptr() + 8 * off, n, lda, out, out.data_ptr() + 4) == 0
        torch.cuda.synchronize()
        assert out.tolist() == [max(0, i - j), max(0, j - i)], (i, j)


@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("n,pad", [(2, 0), (5, 1), (33, 0), (100, 3), (513, 0), (1001, 0), (1500, 9), (4501, 1), (4600, 2)])
def test_detect_of_matrices_full_of_nonzeros(n, pad, off):
    """Every row and column that a thread carries along is one of a nonzero: a dense matrix, its triangles,
    and bands whose edge runs through every vector."""
    lda = n + pad
    P = torch.full((n * lda + off,), float("nan"), dtype=torch.float64, device=DEV)
    M = P[off:].view(n, lda)[:, :n]
    ones = torch.ones((n, n), dtype=torch.float64, device=DEV)
    for kl, ku in ((n - 1, n - 1), (0, n - 1), (n - 1, 0), (n // 3, n // 2), (n // 2, 1), (0, 0)):
        M.copy_(torch.triu(torch.tril(ones, ku), -kl))
        out = torch.full((2,), -7, dtype=torch.int32, device=DEV)
        assert bandlu.detect_bandwidth(P.data_ptr() + 8 * off, n, lda, out, out.data_ptr() + 4) == 0
        torch.cuda.synchronize()
        assert out.tolist() == [kl, ku]

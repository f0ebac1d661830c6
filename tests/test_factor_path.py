"""Which kernel factors a band, around the largest storage that 32-bit offsets reach: the shared-memory
window never gets a band with fewer columns than its panel warp keeps slots for."""
import numpy as np
import pytest

from paper_2608_22099_gb300 import bandlu

REGISTER, SHARED, WIDE = 0, 1, 2
INT_MAX = 2 ** 31 - 1


@pytest.mark.parametrize("n,ldab", [(1, 1), (512, 10), (1 << 20, 2047), (1 << 20, 2048), (1 << 21, 1024),
                                    (1 << 30, 2), (1 << 30, 3), (INT_MAX - 64, 1), (INT_MAX - 63, 1), (INT_MAX, 64),
                                    (256, 1 << 23), (255, (1 << 23) + 7)])
def test_narrow_bands_take_the_register_window_in_any_storage(n, ldab):
    for kl in range(0, 34):
        for ku in range(0, 34):
            path = bandlu.bandlu_selftest_gbtrf_path(n, kl, ku, ldab)
            if n > INT_MAX - 64:  # the windows count rows past the last one in 32 bits
                assert path == WIDE
            elif (kl + 1) * (kl + ku + 1) <= 32:
                assert path == REGISTER, (kl, ku)
            elif path == SHARED:
                assert kl <= 27 and kl + ku + 1 >= 3, (kl, ku)
    assert bandlu.bandlu_selftest_gbtrf_path(n, 28, 28, ldab) == WIDE


@pytest.mark.gpu
@pytest.mark.parametrize("kl,ku", [(0, 0), (1, 0), (0, 1), (2, 3)])
def test_register_window_beyond_32_bit_offsets(kl, ku):
    """2^31 stored elements and more (17 GB of band storage): the last columns' offsets need 64 bits."""
    import torch

    import oracle
    from gpu_helpers import DEV
    n, ldab, w = (1 << 20) + 3, 2048, 2 * kl + ku + 1
    if torch.cuda.mem_get_info()[0] < 3 * 8 * n * ldab:
        pytest.skip("needs 52 GB of free device memory")
    g = torch.Generator().manual_seed(5)
    band = torch.rand((n, w), generator=g, dtype=torch.float64) * 2 - 1
    ref, ipiv_ref, info_ref = oracle.gbtrf(band.numpy(), kl, ku)[:3]
    AB = torch.full((n, ldab), 7.0, dtype=torch.float64, device=DEV)
    AB[:, :w] = band.to(DEV)
    ipiv = torch.full((n,), -1, dtype=torch.int32, device=DEV)
    info = torch.full((1,), -5, dtype=torch.int32, device=DEV)
    assert bandlu.gbtrf(n, kl, ku, AB, ldab, ipiv, info) == 0
    torch.cuda.synchronize()
    assert int(info.item()) == info_ref and np.array_equal(ipiv.cpu().numpy(), ipiv_ref)
    assert np.array_equal(AB[:, :w].cpu().numpy().view(np.int64), ref.view(np.int64))
    assert bool((AB[:, w:w + 8] == 7.0).all()) and bool((AB[-1, w:] == 7.0).all())

"""The dispatches that read the bandwidths back to the host leave nothing of their scratch for the
caller's next synchronisation: memory that is free in the stream-ordered pool there goes back to the
system, which is part of the call's own cost and not to fall after its return.  (A wide band's flags are
taken and given back after it, in stream order.)"""
import ctypes

import pytest
import torch

from gpu_helpers import DEV
from paper_2608_22099_gb300 import bandlu
from paper_2608_22099_gb300.workloads import make_dense
from test_zz_no_alloc import _loaded_cudart

pytestmark = pytest.mark.gpu


def reserved(rt, pool) -> int:
    v = ctypes.c_uint64(0)
    assert rt.cudaMemPoolGetAttribute(pool, 0x5, ctypes.byref(v)) == 0  # cudaMemPoolAttrReservedMemCurrent
    return v.value


@pytest.mark.parametrize("ldab", [11, 56, 57, 200])  # from 57 rows on the storage may hold a wide band
@pytest.mark.parametrize("entry", ["dispatch_lu", "dispatch_lu_cm", "declined", "dispatch_solve", "dispatch_backslash"])
def test_no_pool_memory_is_left_behind(entry, ldab):
    n, kl, ku = 600, 0 if entry == "dispatch_backslash" else 4, 2
    A = make_dense(n, kl, ku, dist="uniform", diag_boost=9.0, seed=4)
    if entry == "declined":
        A[n - 1, 0] = 1e-3
    Ad = A.to(DEV)
    AB = torch.zeros((n, ldab), dtype=torch.float64, device=DEV)
    ipiv = torch.zeros(n, dtype=torch.int32, device=DEV)
    info = torch.zeros(1, dtype=torch.int32, device=DEV)
    B = torch.ones((1, n), dtype=torch.float64, device=DEV)
    rt = _loaded_cudart()
    pool = ctypes.c_void_p()
    assert rt.cudaDeviceGetDefaultMemPool(ctypes.byref(pool), 0) == 0
    torch.cuda.synchronize()
    before = reserved(rt, pool)
    if entry in ("dispatch_lu", "declined"):
        rc = bandlu.dispatch_lu(Ad, n, n, AB, ldab, ipiv, info)[0]
    elif entry == "dispatch_lu_cm":
        rc = bandlu.dispatch_lu_cm(Ad, n, n, AB, ldab, ipiv, info)[0]
    elif entry == "dispatch_solve":
        rc = bandlu.dispatch_solve(Ad, n, n, B, n, 1, AB, ldab, ipiv, info)[0]
    else:
        rc = bandlu.dispatch_backslash(Ad, n, n, B, n, 1, AB, ldab, ipiv, info)[0]
    assert rc == (bandlu.BANDLU_NOT_BANDED if entry == "declined" else bandlu.BANDLU_OK)
    assert reserved(rt, pool) <= before  # asked before any synchronisation of the caller
    torch.cuda.synchronize()

"""The bytes a server counts for a problem (rtg::context_bytes) hold every array
of its context, each on a 512-byte boundary of the one allocation."""
import ctypes

import pytest

import paper_1403_6126_gb300 as rt
from paper_1403_6126_gb300 import build as rtbuild


@pytest.mark.parametrize("N,M", [(1, 1), (7, 5), (64, 8), (1000, 24), (12345, 79)])
@pytest.mark.parametrize("fp64", [False, True])
def test_context_bytes_count_the_rounding(N, M, fp64):
    rtbuild.build()
    f = rt.lib()["_ZN3rtg13context_bytesExib"]
    f.restype, f.argtypes = ctypes.c_size_t, [ctypes.c_longlong, ctypes.c_int, ctypes.c_bool]
    rs = 8 if fp64 else 4
    stored = M if fp64 else 4 * ((M + 3) // 4)
    # intensities, moments, T and its source, momentum source; rho, sigma_a,
    # sigma_s, v; angles, inflow, flags; cell centers; staging (seven fields or
    # the inflow table) with alpha for three cell sides
    arrays = 2 * [rs * stored * N] + 2 * [80 * N] + 2 * [8 * N] + [24 * N] + 3 * [rs * N] + [3 * rs * N]
    arrays += [4 * rs * M, 6 * rs * M, 8] + ([] if fp64 else 2 * [4 * N])
    arrays += [8 * max(7 * N, 6 * M) + 3 * rs * N]
    assert f(N, M, fp64) >= sum((b + 511) // 512 * 512 for b in arrays)

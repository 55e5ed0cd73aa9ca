"""pmpm_power_spectrum_noalloc on stores as callers have them: the counts are a
pointer of the caller's, aligned for an int32 and no further (include/pmpm.h)."""

import ctypes

import numpy as np
import pytest

from paper_2003_03931_gb300 import synth
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def _noalloc(nc, m, counts, nmesh, nbins):
    import torch

    from paper_2003_03931_gb300 import _lib
    lib = _lib.load()
    k, pk, nm = np.zeros(nbins), np.zeros(nbins), np.zeros(nbins, np.int64)
    rc = lib.pmpm_power_spectrum_noalloc(nc, m[0].numel(), m[0].data_ptr(), m[1].data_ptr(), m[2].data_ptr(),
                                         counts.data_ptr(), nmesh, nbins, k.ctypes.data, pk.ctypes.data,
                                         nm.ctypes.data, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    return rc, lib.pmpm_noalloc_last_error(), k, pk, nm


@pytest.mark.parametrize("nc", [8, 16, 32, 64])
@pytest.mark.parametrize("skip", [1, 2, 3])
def test_counts_at_any_int(nc, skip):
    # every block of the scan but the first adds up the counts before its own
    need_gpu()
    import torch
    rng = np.random.default_rng(nc)
    Q = synth.uniform_codes(rng, 4096, nc)
    cell = (Q[0] >> 8) + nc * ((Q[1] >> 8) + nc * (Q[2] >> 8).astype(np.int64))
    Q = Q[:, np.argsort(cell, kind="stable")]
    m = [torch.from_numpy((Q[d] & 255).astype(np.uint8)).cuda() for d in range(3)]
    counts = torch.from_numpy(np.bincount(cell, minlength=nc ** 3).astype(np.int32)).cuda()
    slice_ = torch.zeros(skip + nc ** 3, dtype=torch.int32, device="cuda")[skip:]
    slice_.copy_(counts)
    assert counts.data_ptr() % 16 == 0 and slice_.data_ptr() % 16 == 4 * skip
    nmesh = min(64, 2 * nc)
    want, got = _noalloc(nc, m, counts, nmesh, nmesh // 2), _noalloc(nc, m, slice_, nmesh, nmesh // 2)
    assert want[0] == 0 and got[0] == 0, got[1]
    np.testing.assert_array_equal(got[4], want[4])
    np.testing.assert_array_equal(got[2], want[2])
    np.testing.assert_allclose(got[3], want[3], rtol=1e-13)   # blocks' doubles add up in any order

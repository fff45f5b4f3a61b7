"""Uploads that fail leave nothing behind."""
import contextlib
import ctypes

import numpy as np
import pytest

from test_zz_no_alloc import _DefaultPool

pytestmark = pytest.mark.gpu

MB = 1 << 20
CKKS_ENOMEM = 2


@contextlib.contextmanager
def left(nbytes):
    """The device with about this much memory left."""
    import torch

    def trim():
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        pool = _DefaultPool(torch.cuda.current_device())
        if pool.cu:
            pool.cu.cuMemPoolTrimTo(pool.pool, ctypes.c_size_t(0))

    trim()
    hog = torch.empty(torch.cuda.mem_get_info()[0] - nbytes, dtype=torch.uint8, device="cuda")
    try:
        yield
    finally:
        del hog
        trim()


def test_a_key_whose_upload_failed_stays_unknown():
    """An N = 2^16 key is 122 MB as stored and 352 MB on its way there: with 222 MB left, its place can be
    had and the staging buffer not."""
    from paper_2605_17222_gb300 import binding, synth
    g = binding.Context.from_params(synth.param_set("n16"))
    key = np.zeros((g.beta_max, 2, g.L + g.k, g.N), dtype=np.uint64)
    try:
        used = g.bytes_in_use()
        with left(222 * MB):
            with pytest.raises(binding.CkksError) as e:
                g.upload_rotation_key(5, key)
            assert e.value.status == CKKS_ENOMEM
            assert not g.has_key(5)
            assert g.bytes_in_use() == used
        g.upload_rotation_key(5, key)
        assert g.has_key(5)
        g.device_status()
    finally:
        g.close()

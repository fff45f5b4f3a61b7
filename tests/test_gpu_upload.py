"""Uploads from any memory, beside a recording, and at the limits of memory; the ones that fail leave nothing behind."""
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


def diagonals(ps, D):
    from paper_2605_17222_gb300 import synth
    return np.ascontiguousarray(synth.uniform_mod(5, "f", ps.moduli, ps.n * D).reshape(len(ps.moduli), D, ps.n)
                                .transpose(1, 0, 2))


def lt_of(g, ps, f, ct=None):
    """The LT of one fixed ciphertext, without rotations' keys but the ones of a window of four."""
    from paper_2605_17222_gb300 import synth
    for r in (1, 2, 3):
        if not g.has_key(r):
            k = np.broadcast_to(synth.uniform_mod(r, "k", ps.moduli, ps.n), (g.beta_max, 2, len(ps.moduli), ps.n))
            g.upload_rotation_key(r, np.ascontiguousarray(k))
    c = np.stack([synth.uniform_mod(7 + c, "ct", ps.q, ps.n) for c in range(2)])
    return g.lt_eval(g.ct_from_host(c), f, "th", (1, 2, 2))[0].numpy()


@pytest.mark.parametrize("where", ["pinned", "pageable", "half a word off"])
def test_device_upload_from_other_memory(where):
    """A pointer that is not this device's memory, or not at a word, goes to the copy engine and never to a
    kernel: it is copied or refused.  Host memory stands for another GPU's."""
    import torch

    from paper_2605_17222_gb300 import binding, synth
    ps = synth.param_set("toy")
    g = binding.Context.from_params(ps)
    f = diagonals(ps, 4)
    try:
        want = lt_of(g, ps, g.upload_diagonals(f))
        src = torch.from_numpy(f.view(np.int64))
        if where == "pinned":
            src = src.pin_memory()
        elif where != "pageable":
            src = torch.cat([torch.zeros(1, dtype=torch.int32), src.view(torch.int32).flatten()]).cuda()[1:]
            assert src.data_ptr() % 8 == 4
        part = g.diags_create(4)
        st = binding.lib().ckks_diags_write_device(part.handle, 0, 4, ctypes.c_void_p(src.data_ptr()), f.size,
                                                   binding._stream(None))
        torch.cuda.synchronize()
        if st != 0:  # nothing of a refused call is left
            assert where == "pageable"
            g.diags_write(part, 0, binding.to_device(f))
        assert np.array_equal(lt_of(g, ps, part), want)
        g.device_status()
    finally:
        g.close()


def test_uploads_beside_a_recording():
    """While one thread records a stream, another uploads to a context of its own from the host."""
    import threading

    import torch

    from paper_2605_17222_gb300 import binding, synth
    ps = synth.param_set("toy")
    g, other = binding.Context.from_params(ps), binding.Context.from_params(ps)
    f = diagonals(ps, 4)
    try:
        fh = g.upload_diagonals(f)
        want = lt_of(g, ps, fh)
        ct = g.ct_from_host(np.stack([synth.uniform_mod(7 + c, "ct", ps.q, ps.n) for c in range(2)]))
        out, stream = g.ct_empty(ps.L - 1), torch.cuda.Stream()
        torch.cuda.synchronize()
        recording, uploaded, got = threading.Event(), threading.Event(), []

        def record():
            try:
                g.graph_begin(stream)
                g.lt_eval(ct, fh, "th", (1, 2, 2), out=out, stream=stream)
                recording.set()
                uploaded.wait(60)
                got.append(g.graph_end(stream, keep=(ct, fh, out)))
            except Exception as e:
                got.append(e)
                recording.set()

        t = threading.Thread(target=record)
        t.start()
        recording.wait(60)
        try:
            theirs = other.upload_diagonals(f)
            other.upload_rotation_key(1, np.broadcast_to(synth.uniform_mod(1, "k", ps.moduli, ps.n),
                                                         (g.beta_max, 2, len(ps.moduli), ps.n)))
        finally:
            uploaded.set()
            t.join()
        assert not isinstance(got[0], Exception), got[0]
        got[0].launch(stream)
        torch.cuda.synchronize()
        assert np.array_equal(out.numpy(), want)
        assert np.array_equal(lt_of(other, ps, theirs), want)
        got[0].close()
        g.device_status()
    finally:
        g.close()
        other.close()


def test_host_upload_of_diagonals_in_little_memory():
    """128 diagonals at N = 2^14 are 118 MB as stored and 168 MB on their way there: with room for half of
    those, they are staged in smaller parts."""
    from paper_2605_17222_gb300 import binding, synth
    ps = synth.param_set("n14")
    g = binding.Context.from_params(ps)
    f, split = diagonals(ps, 128), (4, 8, 4)
    key = np.ascontiguousarray(np.broadcast_to(synth.uniform_mod(1, "k", ps.moduli, ps.n),
                                               (g.beta_max, 2, len(ps.moduli), ps.n)))
    ct = np.stack([synth.uniform_mod(7 + c, "ct", ps.q, ps.n) for c in range(2)])
    try:
        with left((118 + 80) * MB):
            staged = g.upload_diagonals(f)
        for r in g.required_rotations("th", split, 128):
            g.upload_rotation_key(r, key)
        whole = g.upload_diagonals_device(binding.to_device(f))
        ct = g.ct_from_host(ct)
        got, want = (g.lt_eval(ct, x, "th", split)[0].numpy() for x in (staged, whole))
        assert np.array_equal(got, want)
        g.device_status()
    finally:
        g.close()

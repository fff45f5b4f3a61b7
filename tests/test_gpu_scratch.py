"""Device memory at its limits: BSGS's scratch stays within its stated bound
and shrinks to what the device has left, with the oracle's residues either way."""
import ctypes

import numpy as np
import pytest

from gpu_common import assert_same
from test_zz_no_alloc import CU_MEMPOOL_ATTR_USED_MEM_CURRENT, CU_MEMPOOL_ATTR_USED_MEM_HIGH, _DefaultPool

pytestmark = pytest.mark.gpu

MB = 1 << 20


def bsgs_problem(split):
    """N = 2^14, level 8: enough rotations (63) that one chunk's scratch is past 512 MB."""
    import oracle.ckks as ock
    from oracle import lt as olt
    from paper_2605_17222_gb300 import binding, synth

    ps = synth.param_set("n14")
    octx, g, D = ock.Ctx(ps), binding.Context.from_params(ps), split[0] * split[1]
    key = np.stack([synth.uniform_mod(b, "key", ps.moduli, ps.n) for b in range(2 * octx.beta_max)]).reshape(
        octx.beta_max, 2, len(ps.moduli), ps.n)
    keys = {r: key for r in olt.rotation_set("bsgs", D, split, 1, ps.n // 2)}
    dev = binding.to_device(key)
    for r in keys:
        g.upload_rotation_key_device(r, dev)
    f = np.ascontiguousarray(synth.uniform_mod(5, "f", ps.moduli, ps.n * D).reshape(len(ps.moduli), D, ps.n)
                             .transpose(1, 0, 2))
    ct = np.stack([synth.uniform_mod(7 + c, "ct", ps.q, ps.n) for c in range(2)])
    want = np.stack(olt.run(octx, "bsgs", (ct[0], ct[1]), f, keys, split)[0])
    # the polynomials that outlive a chunk: rotated pairs of the baby steps, sums of the giant ones
    kept = 8 * ps.n * 2 * ps.L * (split[0] - 1 + split[1])
    return g, g.upload_diagonals(f), g.ct_from_host(ct), want, kept


@pytest.mark.parametrize("split", [(64, 2), (2, 64)])
def test_bsgs_scratch_bound(split):
    import torch
    g, f, ct, want, kept = bsgs_problem(split)
    try:
        out, _ = g.lt_eval(ct, f, "bsgs", split)
        assert_same(out.numpy(), want, f"{split}")
        pool = _DefaultPool(torch.cuda.current_device())
        if not pool.cu:
            pytest.skip("no driver library")
        torch.cuda.synchronize()
        pool.reset_high()
        used = pool.get(CU_MEMPOOL_ATTR_USED_MEM_CURRENT)
        g.lt_eval(ct, f, "bsgs", split, out=out)
        torch.cuda.synchronize()
        peak = pool.get(CU_MEMPOOL_ATTR_USED_MEM_HIGH) - used
        assert peak <= kept + 512 * MB + 4 * MB, f"{split}: {peak / MB:.0f} MB, {kept / MB:.0f} MB of them kept"
        g.device_status()
    finally:
        g.close()


def test_bsgs_in_little_memory():
    """With room for a third of a chunk, the chunks get smaller instead of the call failing."""
    import torch
    split = (64, 2)
    g, f, ct, want, kept = bsgs_problem(split)
    pool = _DefaultPool(torch.cuda.current_device())
    if not pool.cu:
        pytest.skip("no driver library")
    hog = None
    try:
        out, _ = g.lt_eval(ct, f, "bsgs", split)  # the level's tables
        torch.cuda.synchronize()
        out.tensor.zero_()
        torch.cuda.empty_cache()
        assert pool.cu.cuMemPoolTrimTo(pool.pool, ctypes.c_size_t(0)) == 0
        free, _ = torch.cuda.mem_get_info()
        hog = torch.empty(free - kept - 200 * MB, dtype=torch.uint8, device="cuda")
        g.lt_eval(ct, f, "bsgs", split, out=out)
        torch.cuda.synchronize()
        del hog
        assert_same(out.numpy(), want, "chunks of fewer rotations")
        g.device_status()
    finally:
        hog = None
        torch.cuda.empty_cache()
        pool.cu.cuMemPoolTrimTo(pool.pool, ctypes.c_size_t(0))
        g.close()


@pytest.mark.parametrize("params,level,split,offset0", [
    ("n14", 8, (1, 16, 4), 0), ("n14", 8, (1, 16, 4), 5), ("n14", 3, (4, 1, 16), 1), ("n14", 8, (16, 2, 2), 0),
    ("setA", 2, (8, 1, 8), 0), ("setA", 5, (1, 1, 16), 3), ("n16", 24, (1, 16, 4), 1),
])
def test_serving_estimate_is_an_upper_one(params, level, split, offset0):
    """The serving loop's scratch_bytes covers what an LT, and each of a batch, takes from the pool."""
    import torch

    from paper_2605_17222_gb300 import binding, synth
    from paper_2605_17222_gb300.serving import scratch_bytes
    ps = synth.param_set(params)
    g, D = binding.Context.from_params(ps), int(np.prod(split))
    pool = _DefaultPool(torch.cuda.current_device())
    if not pool.cu:
        pytest.skip("no driver library")
    try:
        key = synth.uniform_mod_device(1, "k", ps.moduli, ps.n, 2 * g.beta_max)
        for r in g.required_rotations("th", split, D, offset0=offset0):
            g.upload_rotation_key_device(r, key)
        f = g.diags_create(D, offset0=offset0)
        g.diags_write(f, 0, synth.uniform_mod_device(2, "f", ps.moduli, ps.n, D))
        cts = [g.ct_wrap(synth.uniform_mod_device(3 + i, "c", ps.q[:level], ps.n, 2), level) for i in range(3)]
        outs = [g.ct_empty(level - 1) for _ in cts]
        one = scratch_bytes(g, level, split)
        for count, run in ((1, lambda: g.lt_eval(cts[0], f, "th", split, out=outs[0])),
                           (3, lambda: g.lt_eval_batch(cts, [f] * 3, ["th"] * 3, [split] * 3, outs))):
            run()
            torch.cuda.synchronize()
            pool.reset_high()
            used = pool.get(CU_MEMPOOL_ATTR_USED_MEM_CURRENT)
            run()
            torch.cuda.synchronize()
            peak = pool.get(CU_MEMPOOL_ATTR_USED_MEM_HIGH) - used
            assert peak <= count * one, f"{count} LTs: {peak / MB:.1f} MB, estimated {count * one / MB:.1f}"
        g.device_status()
    finally:
        g.close()

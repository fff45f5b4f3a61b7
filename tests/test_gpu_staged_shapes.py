"""Shapes at the edges of the staged diagonal kernel's shared memory, bit for
bit with the oracle: up to eight digits of a key with many more, a long table of
middle indices, and a basis past the kernel's list of limbs."""
import numpy as np
import pytest

from gpu_common import assert_same

pytestmark = pytest.mark.gpu

CKKS_ETIMEOUT = 5


def problem(q_bits, p_bits, dnum, level, split):
    """Like test_gpu_packed.problem at N = 2^12, with two keys for all rotations."""
    import oracle.ckks as ock
    from oracle import lt as olt
    from paper_2605_17222_gb300 import binding, synth

    ps = synth.make_params("shapes", 12, q_bits, p_bits, dnum)
    octx, g, D = ock.Ctx(ps), binding.Context.from_params(ps), int(np.prod(split))
    n = len(ps.moduli)
    some = [np.ascontiguousarray(synth.uniform_mod(11 + i, "key", ps.moduli, ps.n * 2 * octx.beta_max)
                                 .reshape(n, 2 * octx.beta_max, ps.n).transpose(1, 0, 2)).reshape(octx.beta_max, 2, n, ps.n)
            for i in range(2)]
    dev = [binding.to_device(k) for k in some]
    rots = olt.rotation_set("th", D, split, 1, ps.n // 2)
    for r in rots:
        g.upload_rotation_key_device(r, dev[r % 2])
    f = np.ascontiguousarray(synth.uniform_mod(5, "f", ps.moduli, ps.n * D).reshape(n, D, ps.n).transpose(1, 0, 2))
    ct = np.stack([synth.uniform_mod(7 + c, "ct", ps.q[:level], ps.n) for c in range(2)])
    want = np.stack(olt.run(octx, "th", (ct[0], ct[1]), f, {r: some[r % 2] for r in rots}, split)[0])
    return g, g.upload_diagonals(f), g.ct_from_host(ct), want


@pytest.mark.parametrize("q_bits,p_bits,dnum,level,split,staged", [
    ([40] * 36, [40], 36, 8, (1, 2, 4), True),     # eight digits of 36: three CTAs
    ([40] * 64, [40], 64, 8, (1, 2, 8), True),     # of 64, eight outer indices: two CTAs
    ([40] * 160, [40], 160, 8, (1, 2, 4), False),  # of 160: one CTA's share only, the plain kernel
    ([54] * 8, [55], 8, 8, (1, 400, 2), True),     # a j table of 1.6 KB beside the wide limbs' stages
])
def test_up_to_eight_digits_stay_staged(q_bits, p_bits, dnum, level, split, staged):
    from paper_2605_17222_gb300 import binding
    g, f, ct, want = problem(q_bits, p_bits, dnum, level, split)
    try:
        got, _ = g.lt_eval(ct, f, "th", split)
        assert_same(got.numpy(), want, f"{split} level {level}")
        g.device_status()
        g.debug_diag_mac_waits(20_000, 1)  # only the staged kernel has a step to leave out
        g.lt_eval(ct, f, "th", split)
        if staged:
            with pytest.raises(binding.CkksError) as e:
                g.device_status()
            assert e.value.status == CKKS_ETIMEOUT
        g.debug_diag_mac_waits(0, 0xFFFFFFFF)
        g.device_status()
    finally:
        g.close()


def test_more_limbs_than_the_kernels_list():
    """A basis of 258 limbs, past DM_MAX_LIMBS: one launch of the plain kernel over every limb."""
    g, f, ct, want = problem([55] + [40] * 253, [60] * 4, 127, 254, (2, 2, 2))
    try:
        got, _ = g.lt_eval(ct, f, "th", (2, 2, 2))
        assert_same(got.numpy(), want, "258 limbs")
        g.device_status()
    finally:
        g.close()

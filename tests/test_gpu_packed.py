"""The stored layouts of keys and diagonals and the arithmetic class of each
modulus, bit for bit with the oracle on a chain that mixes every class: below
2^32, just above it, packed 40-bit, 41-bit, 55-bit and the 56- to 59-bit wide
forms; digit counts at the edges of the staged diagonal kernel (1, 6, 7, 8 and
9 digits), and more terms than one reduction interval."""
import numpy as np
import pytest

from gpu_common import assert_same

pytestmark = pytest.mark.gpu

Q_BITS = [55, 31, 33, 40, 41, 54, 56, 59, 40]


def problem(dnum, level, D, split, algo, offset0=0):
    import oracle.ckks as ock
    from oracle import lt as olt
    from paper_2605_17222_gb300 import binding, synth

    ps = synth.make_params("mixed", 12, Q_BITS, [60, 50], dnum)
    octx, g = ock.Ctx(ps), binding.Context.from_params(ps)
    rots = olt.rotation_set(algo, D, split, 1, ps.n // 2, offset0)
    keys = {}
    for r in rots:
        k = synth.uniform_mod(11 + r, "key", ps.moduli, ps.n * 2 * octx.beta_max)
        keys[r] = np.ascontiguousarray(k.reshape(len(ps.moduli), 2 * octx.beta_max, ps.n).transpose(1, 0, 2)).reshape(
            octx.beta_max, 2, len(ps.moduli), ps.n)
        g.upload_rotation_key(r, keys[r])
    f = np.ascontiguousarray(synth.uniform_mod(5, "f", ps.moduli, ps.n * D).reshape(len(ps.moduli), D, ps.n)
                             .transpose(1, 0, 2))
    ct = np.stack([synth.uniform_mod(7 + c, "ct", ps.q[:level], ps.n) for c in range(2)])
    want = np.stack(olt.run(octx, algo, (ct[0], ct[1]), f, keys, split, 1, offset0)[0])
    return g, g.upload_diagonals(f, offset0=offset0), ct, want


@pytest.mark.parametrize("dnum,level,D,split,algo,offset0", [
    (9, 9, 12, (2, 3, 2), "th", 0),      # 9 digits: the plain kernel
    (9, 8, 12, (2, 3, 2), "th", -3),     # 8 digits
    (9, 7, 8, (1, 4, 2), "th", 0),       # 7
    (9, 6, 70, (1, 35, 2), "th", 5),     # 6, more than 32 terms, an odd count
    (1, 9, 40, (2, 10, 2), "th", 0),     # 1 digit of every limb
    (3, 5, 66, (33, 2, 1), "dh", 0),     # baby steps materialised or fused
    (3, 9, 9, (3, 3, 1), "bsgs", 1),
    (3, 2, 10, (1, 1, 10), "th", 0),     # outer indices past one block of eight
])
def test_mixed_moduli_lt(dnum, level, D, split, algo, offset0):
    g, f, ct, want = problem(dnum, level, D, split, algo, offset0)
    try:
        got, _ = g.lt_eval(g.ct_from_host(ct), f, algo, split)
        assert_same(got.numpy(), want, f"{algo} {split} dnum {dnum} level {level}")
        outs = g.lt_eval_batch([g.ct_from_host(ct) for _ in range(3)], [f] * 3, [algo] * 3, [split] * 3)
        for o in outs:
            assert_same(o.numpy(), want, f"batch {algo} {split}")
        g.device_status()
    finally:
        g.close()


@pytest.mark.parametrize("copies,level,split", [
    (2, 18, (1, 3, 1)),   # 18 digits: groups of four and a rest of two; one outer index
    (2, 13, (2, 2, 2)),   # a rest of one
    (2, 12, (1, 4, 3)),   # no rest; a tile of four with an idle index
    (2, 10, (1, 2, 9)),   # eight outer indices and one more
    (4, 36, (1, 2, 8)),   # stages too large for the wide limbs: the plain kernel for them
])
def test_more_than_eight_digits(monkeypatch, copies, level, split):
    monkeypatch.setitem(globals(), "Q_BITS", Q_BITS * copies)
    g, f, ct, want = problem(9 * copies, level, int(np.prod(split)), split, "th")
    try:
        got, _ = g.lt_eval(g.ct_from_host(ct), f, "th", split)
        assert_same(got.numpy(), want, f"{split} {level} digits")
        g.device_status()
    finally:
        g.close()


def test_words_beyond_the_modulus_are_taken_as_residues():
    """Diagonals written in pieces, with words in [q, 2q), give the same result as their residues."""
    import torch

    from paper_2605_17222_gb300 import binding, synth
    ps = synth.param_set("toy")
    g = binding.Context.from_params(ps)
    f = np.ascontiguousarray(synth.uniform_mod(5, "f", ps.moduli, ps.n * 4).reshape(len(ps.moduli), 4, ps.n)
                             .transpose(1, 0, 2))
    q = np.array(ps.moduli, dtype=np.uint64)[None, :, None]
    ct = g.ct_from_host(np.stack([synth.uniform_mod(7, "ct", ps.q, ps.n)] * 2))
    for r in (1, 2, 3):
        k = np.broadcast_to(synth.uniform_mod(r, "k", ps.moduli, ps.n), (g.beta_max, 2, len(ps.moduli), ps.n))
        g.upload_rotation_key(r, np.ascontiguousarray(k))
    want, _ = g.lt_eval(ct, g.upload_diagonals(f), "th", (1, 2, 2))
    part = g.diags_create(4)
    t = binding.to_device(f + q)
    g.diags_write(part, 1, t[1:])
    g.diags_write(part, 0, t[:1])
    got, _ = g.lt_eval(ct, part, "th", (1, 2, 2))
    torch.cuda.synchronize()
    assert_same(got.numpy(), want.numpy(), "words above the modulus")
    g.close()


@pytest.mark.parametrize("words", [0, 1])
def test_operands_at_any_word(words):
    """Digits and ciphertexts that start at an odd word (8-byte aligned) give the same results."""
    import torch

    from paper_2605_17222_gb300 import binding, synth
    ps = synth.param_set("toy")
    g = binding.Context.from_params(ps)

    def at(a):
        buf = torch.empty(a.size + 2, dtype=torch.int64, device="cuda")
        t = buf[words:words + a.size].view(a.shape)
        t.copy_(binding.to_device(a))
        return t

    for r in (1, 2, 3):
        k = np.broadcast_to(synth.uniform_mod(r, "k", ps.moduli, ps.n), (g.beta_max, 2, len(ps.moduli), ps.n))
        g.upload_rotation_key(r, np.ascontiguousarray(k))
    d = np.stack([synth.uniform_mod(20 + b, "d", ps.moduli, ps.n) for b in range(g.beta_max)])
    c = np.stack([synth.uniform_mod(30 + b, "c", ps.q, ps.n) for b in range(2)])
    f = np.stack([synth.uniform_mod(40 + b, "f", ps.moduli, ps.n) for b in range(4)])
    fh = g.upload_diagonals(f)
    got = [t.cpu() for t in g.ks_inner(ps.L, at(d), 2, 2)]
    want = [t.cpu() for t in g.ks_inner(ps.L, binding.to_device(d), 2, 2)]
    for algo, split in (("th", (1, 2, 2)), ("bsgs", (2, 2))):
        want.append(g.lt_eval(g.ct_wrap(binding.to_device(c), ps.L), fh, algo, split)[0].tensor.cpu())
        got.append(g.lt_eval(g.ct_wrap(at(c), ps.L), fh, algo, split)[0].tensor.cpu())
    for x, y in zip(got, want):
        assert_same(x.numpy(), y.numpy(), f"offset {words}")
    g.close()


@pytest.mark.parametrize("params,level,split,algo", [
    ("n14", 8, (3, 2, 3), "th"),    # ModDown into Decompose as one step
    ("n14", 5, (9, 2), "bsgs"),     # a partial last digit, rotations in one chunk
    ("setA", 5, (2, 2, 4), "th"),   # five special limbs
])
def test_merged_key_switches_equal_their_steps(params, level, split, algo):
    """LTs whose key switches run merged or batched, bit for bit with the oracle's step by step."""
    import oracle.ckks as ock
    from oracle import lt as olt
    from paper_2605_17222_gb300 import binding, synth

    ps = synth.param_set(params)
    octx, g = ock.Ctx(ps), binding.Context.from_params(ps)
    D = int(np.prod(split))
    keys = {}
    for r in olt.rotation_set(algo, D, split, 1, ps.n // 2, 2):
        keys[r] = np.stack([synth.uniform_mod(11 + r + 1000 * b, "key", ps.moduli, ps.n)
                            for b in range(2 * octx.beta_max)]).reshape(octx.beta_max, 2, len(ps.moduli), ps.n)
        g.upload_rotation_key(r, keys[r])
    f = np.stack([synth.uniform_mod(5 + d, "f", ps.moduli, ps.n) for d in range(D)])
    ct = np.stack([synth.uniform_mod(7 + c, "ct", ps.q[:level], ps.n) for c in range(2)])
    want = np.stack(olt.run(octx, algo, (ct[0], ct[1]), f, keys, split, 1, 2)[0])
    got, _ = g.lt_eval(g.ct_from_host(ct), g.upload_diagonals(f, offset0=2), algo, split)
    assert_same(got.numpy(), want, f"{params} {algo} {split}")
    g.close()

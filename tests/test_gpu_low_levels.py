"""Levels with fewer Q limbs than special primes, bit for bit with the oracle.

A ModDown of n polynomials writes n k limbs of scratch there and a Decompose
of them only n level, so a scratch sized for the Decompose alone is overrun:
these are the shapes that show it, several baby and outer indices at once,
single, batched and chained."""
import numpy as np
import pytest

from gpu_common import assert_same

pytestmark = pytest.mark.gpu


def uniform(seed, tag, moduli, n, *lead):
    """[*lead][len(moduli)][n] residues."""
    from paper_2605_17222_gb300 import synth
    a = synth.uniform_mod(seed, tag, moduli, n * int(np.prod(lead)))
    return np.ascontiguousarray(a.reshape(len(moduli), -1, n).transpose(1, 0, 2)).reshape(*lead, len(moduli), n)


def problem(params, level, algo, split, offset0=0):
    """Context, diagonals, ciphertext and the oracle's result."""
    import oracle.ckks as ock
    from oracle import lt as olt
    from paper_2605_17222_gb300 import binding, synth

    ps = synth.param_set(params) if isinstance(params, str) else params
    octx, g, D = ock.Ctx(ps), binding.Context.from_params(ps), int(np.prod(split))
    keys = {r: uniform(11 + r, "key", ps.moduli, ps.n, octx.beta_max, 2)
            for r in olt.rotation_set(algo, D, split, 1, ps.n // 2, offset0)}
    for r, k in keys.items():
        g.upload_rotation_key(r, k)
    f = uniform(5, "f", ps.moduli, ps.n, D)
    ct = uniform(7, "ct", ps.q[:level], ps.n, 2)
    want = np.stack(olt.run(octx, algo, (ct[0], ct[1]), f, keys, split, 1, offset0)[0])
    return g, g.upload_diagonals(f, offset0=offset0), ct, want


def many_special():
    from paper_2605_17222_gb300 import synth
    return synth.make_params("many special primes", 12, [55, 40, 40, 40], [60] * 8, 2)


# Set-A (k = 5, one digit of every limb): one outer index, and several of both
# kinds; Set-B (k = 8); eight special primes over packed limbs, in the form
# with the ModDown merged into the Decompose and the baby steps materialised.
@pytest.mark.parametrize("params,level,algo,split,offset0", [
    ("setA", 2, "th", (14, 5, 1), 0),
    ("setA", 4, "th", (3, 2, 9), -4),
    ("setB", 2, "th", (7, 4, 5), 0),
    ("setA", 2, "dh", (6, 8), 3),
    ("setA", 3, "bsgs", (7, 6), 0),
    (many_special, 2, "th", (9, 2, 3), 1),
    (many_special, 3, "diag", (1, 13, 1), 2),
])
def test_fewer_q_limbs_than_special_primes(params, level, algo, split, offset0):
    g, f, ct, want = problem(params() if callable(params) else params, level, algo, split, offset0)
    try:
        got, _ = g.lt_eval(g.ct_from_host(ct), f, algo, split)
        assert_same(got.numpy(), want, f"{algo} {split} level {level}")
        for o in g.lt_eval_batch([g.ct_from_host(ct) for _ in range(3)], [f] * 3, [algo] * 3, [split] * 3):
            assert_same(o.numpy(), want, f"batch {algo} {split} level {level}")
        if algo != "bsgs":
            chained, _ = g.lt_eval_chain(g.ct_from_host(ct), [f], algos=[algo], splits=[split])
            assert_same(chained.numpy(), want, f"chain {algo} {split} level {level}")
        g.device_status()
    finally:
        g.close()

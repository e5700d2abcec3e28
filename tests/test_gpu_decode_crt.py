"""Exact CRT of decoding on the device: integers at the ends of the centred range, from one limb to
966 bits (FP64 holds less than the whole chain), against Python integers.  Each of the level + 1 Horner steps rounds its product-sum
and its digit once, so the decoded value lies within 2 (level + 1) 2^-53 of the integer, relatively."""
import random

import numpy as np
import pytest

from tests.pairs import gpu_ctx, oracle_params

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("name,level", [("cfg1", 0), ("cfg1", 3), ("cfg2_small", 1), ("cfg2_small", 9), ("cfg2_small", 20)])
def test_decode_centred_integers(name, level):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_04356_gb300 import build
    from paper_2312_04356_gb300 import ckks as K
    build.build()
    P = oracle_params(name)
    ctx = gpu_ctx(name, 3)
    q = [int(x) for x in P.q[:level + 1]]
    Q = 1
    for x in q:
        Q *= x
    g = random.Random(7)
    vals = [0, 1, -1, 2, -2, Q // 2, -(Q // 2), Q // 2 - 1, 1 - Q // 2, q[0], -q[0], Q // q[-1], -(Q // q[-1])]
    vals = [v for v in vals if abs(v) <= Q // 2]
    vals += [g.randrange(-(Q // 2), Q // 2 + 1) >> g.randrange(0, Q.bit_length()) for _ in range(P.n - len(vals))]
    limbs = np.array([[v % x for v in vals] for x in q], dtype=np.uint64)
    pt = K.ckks_pt_import_rns(ctx, limbs, level, 1.0)
    got = K.ckks_decode(ctx, pt, K.CKKS_COEFF)
    want = np.array([float(v) for v in vals])
    assert (np.abs(got - want) <= 2 * (level + 1) * 2.0 ** -53 * np.abs(want)).all()
    with pytest.raises(K.CkksError):
        K.ckks_decode(ctx, K.ckks_pt_create(ctx))          # nothing to decode

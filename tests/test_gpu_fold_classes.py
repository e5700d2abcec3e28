"""Folded products over the widths of primes that qualify (33 to 60 bits; from 58 on values are folded
every four stages) and over the rings that the general pass transforms: extremes against the oracle, bit
for bit.  Every chain's primes are checked to qualify, so that the folded kernels are the ones that run."""
import gc

import numpy as np
import pytest

import workloads as WL
from tests.test_fold_bounds import consts  # noqa: F401  (fixture: the library's rule)

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


# (log_n, q0, scale, special primes) in bits; the widths between 43 and 59 have no named chain
@pytest.mark.parametrize("log_n,q0,sc,pb", [
    (3, 60, 36, 60), (7, 58, 33, 59), (13, 50, 45, 55), (14, 60, 42, 60), (14, 58, 53, 56), (15, 60, 45, 60), (15, 58, 50, 59),
    (17, 60, 48, 60), (17, 59, 54, 58), (10, 50, 45, 55), (12, 58, 50, 59), (10, 59, 54, 58), (10, 58, 53, 56), (16, 50, 45, 55),
    (16, 58, 50, 59), (16, 60, 54, 58)])
def test_transform_extremes(consts, log_n, q0, sc, pb):  # noqa: F811
    from oracle import _clib as C
    from oracle import params as PP
    from paper_2312_04356_gb300 import ckks as K
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d = dict(log_n=log_n, n_q=3, dnum=1, n_p=1, q0_bits=q0, scale_bits=sc, p_bits=pb, boot_bits=0, n_boot=0, h=0, sigma=3.2)
    ctx = K.ckks_ctx_create(d, 1, torch.cuda.current_stream().cuda_stream)
    P = PP.Params(log_n, 3, 1, q0, sc, pb, h=0, n_p=1)
    q, p, _, _ = K.ckks_ctx_info(ctx)
    mods, n = q + p, 1 << log_n
    assert mods == list(P.q) + list(P.p) and all(consts(m) for m in mods)
    g = np.random.default_rng(13)
    x = np.stack([r for m in mods for r in (
        np.full(n, m - 1, dtype=np.uint64), np.where(np.arange(n) % 2 == 0, 0, m - 1).astype(np.uint64),
        np.where(np.arange(n) < n // 2, m // 2, m // 2 + 1).astype(np.uint64), g.integers(0, m, n, dtype=np.uint64))])
    ids = [i for i in range(len(mods)) for _ in range(4)]
    psi = list(P.psi_q) + list(P.psi_p)
    for call, ref in ((K.ckks_ntt_forward, C.ntt_forward), (K.ckks_ntt_inverse, C.ntt_inverse)):
        dev = torch.from_numpy(x.view(np.int64).copy()).cuda()
        call(ctx, dev.data_ptr(), len(ids), ids)
        torch.cuda.synchronize()
        want = ref(x, [mods[i] for i in ids], [psi[i] for i in ids], log_n)
        assert (dev.cpu().numpy().view(np.uint64) == want).all(), call.__name__


# 128-bit sums, conversions, lifts and tails over the same widths
@pytest.mark.parametrize("log_n,q0,sc,pb,dnum", [(10, 50, 45, 55, 2), (10, 59, 54, 58, 4), (10, 58, 53, 56, 3), (10, 58, 50, 59, 1),
                                                 (13, 50, 45, 55, 2), (10, 60, 36, 60, 2)])
def test_key_switch(consts, log_n, q0, sc, pb, dnum):  # noqa: F811
    from tests.pairs import assert_ct_equal, import_ct, import_plan, make_pair
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    WL.PARAMS["fold_test"] = dict(log_n=log_n, n_q=4, dnum=dnum, n_p=0, q0_bits=q0, scale_bits=sc, p_bits=pb,
                                  boot_bits=0, n_boot=0, h=0, sigma=3.2)
    try:
        m = 1 << (log_n - 1)
        K, o, ctx, keys = make_pair("fold_test", 37, rotations=list(range(1, 9)))
        P, lev = o.P, o.P.L
        assert all(consts(x) for x in list(P.q) + list(P.p))
        ct = o.encrypt(o.encode_pt(WL.slots(1, m, 0.5), lev, P.delta[lev]), 1)
        gct = import_ct(K, ctx, ct)
        for s, g, w in zip([1, 7], K.ckks_rotate_hoisted(ctx, keys, gct, [1, 7]), o.rotate_hoisted(ct, [1, 7])):
            assert_ct_equal(K, ctx, g, w, "HRot %d" % s)
        assert_ct_equal(K, ctx, K.ckks_mul_relin(ctx, keys, gct, gct), o.mul_relin(ct, ct), "HMult")
        assert_ct_equal(K, ctx, K.ckks_rescale(ctx, gct), o.rescale(ct), "rescale")
        assert_ct_equal(K, ctx, K.ckks_level_down(ctx, gct, 1), o.level_down(ct, 1), "level_down")
        c0 = o.mod_drop(ct, 0)
        assert_ct_equal(K, ctx, K.ckks_mod_raise(ctx, import_ct(K, ctx, c0)), o.mod_raise(c0), "ModRaise")
        for B in (4, 1):            # 3 giant steps (fused kernel), 9 (stored babies)
            plan = o.make_plan({i: WL.slots(40 + i, m) for i in range(9)}, 0, 1, 9, lev, P.delta[lev], B=B)
            assert_ct_equal(K, ctx, K.ckks_bsgs(ctx, keys, gct, import_plan(K, ctx, plan)), o.bsgs(ct, plan), "BSGS B=%d" % B)
        K.ckks_sync(ctx)
    finally:
        del WL.PARAMS["fold_test"]
        K = o = ctx = keys = ct = gct = g = w = plan = None
        gc.collect()

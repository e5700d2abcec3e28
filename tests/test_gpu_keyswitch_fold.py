"""Key-switch products in both reductions (folded 128-bit sums, Shoup products) over the digit
counts and both BSGS kernels, and the lifts and tails inside the transforms or beside them:
rotations, HMult, rescales, ModRaise and a BSGS map bit-exact against the oracle."""
import gc

import pytest

import workloads as WL
from tests.pairs import assert_ct_equal, gpu_ctx, import_ct, import_plan, make_pair

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


# every digit count; a 61-bit base prime puts the context on Shoup products; N = 2^13 transforms the
# conversions' lazy outputs in the general shared-memory pass
@pytest.mark.parametrize("log_n,q0,dnum,n_q", [(10, 60, 1, 4), (10, 60, 2, 4), (10, 60, 4, 4), (10, 61, 1, 4),
                                               (10, 61, 3, 5), (10, 61, 4, 4), (13, 60, 2, 4)])
def test_key_switch_bitexact(log_n, q0, dnum, n_q):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_04356_gb300 import build
    build.build()
    WL.PARAMS["fold_test"] = dict(log_n=log_n, n_q=n_q, dnum=dnum, n_p=0, q0_bits=q0, scale_bits=42, p_bits=60,
                                  boot_bits=0, n_boot=0, h=0, sigma=3.2)
    try:
        m = 1 << (log_n - 1)
        K, o, ctx, keys = make_pair("fold_test", 31, rotations=list(range(1, 9)) + [m - 4, m - 8])
        P, lev = o.P, o.P.L
        ct = o.encrypt(o.encode_pt(WL.slots(1, m, 0.5), lev, P.delta[lev]), 1)
        gct = import_ct(K, ctx, ct)
        for s, g, w in zip([1, 7], K.ckks_rotate_hoisted(ctx, keys, gct, [1, 7]), o.rotate_hoisted(ct, [1, 7])):
            assert_ct_equal(K, ctx, g, w, "HRot %d" % s)
        assert_ct_equal(K, ctx, K.ckks_mul_relin(ctx, keys, gct, gct), o.mul_relin(ct, ct), "HMult")
        assert_ct_equal(K, ctx, K.ckks_rescale(ctx, gct), o.rescale(ct), "rescale")
        assert_ct_equal(K, ctx, K.ckks_level_down(ctx, gct, 1), o.level_down(ct, 1), "level_down")
        c0 = o.mod_drop(ct, 0)
        assert_ct_equal(K, ctx, K.ckks_mod_raise(ctx, import_ct(K, ctx, c0)), o.mod_raise(c0), "ModRaise")
        diags = {i: WL.slots(40 + i, m) for i in range(9)}
        for B in (4, 1):            # 3 giant steps (fused kernel), 9 (stored babies)
            plan = o.make_plan(diags, 0, 1, 9, lev, P.delta[lev], B=B)
            assert_ct_equal(K, ctx, K.ckks_bsgs(ctx, keys, gct, import_plan(K, ctx, plan)), o.bsgs(ct, plan), "BSGS B=%d" % B)
        K.ckks_sync(ctx)
    finally:
        del WL.PARAMS["fold_test"]
        K = o = ctx = keys = ct = gct = g = w = plan = None
        gc.collect()        # the device memory goes back here, not in the middle of a later test


# rotations brought down together against each alone: two pass kernels (N = 2^16), one CTA a limb and
# the general transform with separate tails; an identity, a repeated step and more than one group
@pytest.mark.parametrize("log_n,q0", [(16, 60), (10, 60), (13, 60), (10, 61)])
def test_hoisted_rotations_together_match_single(log_n, q0):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_04356_gb300 import build
    build.build()
    WL.PARAMS["fold_test"] = dict(log_n=log_n, n_q=3, dnum=2, n_p=0, q0_bits=q0, scale_bits=42, p_bits=60,
                                  boot_bits=0, n_boot=0, h=0, sigma=3.2)
    try:
        from paper_2312_04356_gb300 import ckks as K
        ctx = gpu_ctx("fold_test", 33)
        keys = K.ckks_keygen(ctx, list(range(1, 9)), False)
        ct = K.ckks_encrypt(ctx, keys, K.ckks_encode(ctx, WL.slots(1, 1 << (log_n - 1), 0.5), 2, 2.0 ** 42), 1)
        steps = [3, 0, 1, 2, 4, 5, 6, 7, 8, 3]
        for s, got in zip(steps, K.ckks_rotate_hoisted(ctx, keys, ct, steps)):
            want = K.ckks_rotate_hoisted(ctx, keys, ct, [s])[0] if s else ct
            assert (K.ckks_ct_export_rns(ctx, got) == K.ckks_ct_export_rns(ctx, want)).all(), s
        K.ckks_sync(ctx)
    finally:
        del WL.PARAMS["fold_test"]
        K = ctx = keys = ct = got = want = None
        gc.collect()


# batches share key words between pairs of ciphertexts; an odd number leaves one over.  Both reductions,
# the block's accumulated key switches and (cin = 16, w0 = 2) the stored babies
@pytest.mark.parametrize("B", [1, 2, 5])
@pytest.mark.parametrize("q0", [60, 61])
@pytest.mark.parametrize("spec", [WL.CONV["cfg2_small"], dict(cin=16, cout=16, w0=2, f=3, weight="gauss")])
def test_batched_pairs_match_single(B, q0, spec):
    from tests.test_gpu_batch import _setup
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_04356_gb300 import build
    build.build()
    WL.PARAMS["fold_test"] = dict(WL.PARAMS["cfg2_small"], q0_bits=q0)
    try:
        d = _setup("fold_test", 57, spec, B, oracle_keys=False)
        K, ctx, keys = d["K"], d["ctx"], d["keys"]
        outs = K.ckks_block_batched(ctx, keys, d["gcts"], d["gplan"], d["bt"])
        for c, out in zip(d["gcts"], outs):
            one = K.ckks_block(ctx, keys, c, d["gplan"], d["bt"])
            assert (K.ckks_ct_export_rns(ctx, out) == K.ckks_ct_export_rns(ctx, one)).all()
    finally:
        del WL.PARAMS["fold_test"]
        d = K = ctx = keys = outs = c = out = one = None
        gc.collect()


# more rotated giant steps than one sum holds (9 at four digits, 13 at three, 16 otherwise) and than are
# raised together, with and without an unrotated one to add to
@pytest.mark.parametrize("log_n,q0,dnum,n_q", [(10, 60, 4, 4), (10, 61, 4, 4), (10, 60, 3, 5), (13, 60, 2, 4)])
@pytest.mark.parametrize("a0", [0, 1])
def test_many_giant_steps_bitexact(log_n, q0, dnum, n_q, a0):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_04356_gb300 import build
    build.build()
    WL.PARAMS["fold_test"] = dict(log_n=log_n, n_q=n_q, dnum=dnum, n_p=0, q0_bits=q0, scale_bits=42, p_bits=60,
                                  boot_bits=0, n_boot=0, h=0, sigma=3.2)
    try:
        m = 1 << (log_n - 1)
        K, o, ctx, keys = make_pair("fold_test", 35, rotations=list(range(1, 22)))
        P, lev = o.P, o.P.L
        ct = o.encrypt(o.encode_pt(WL.slots(1, m, 0.5), lev, P.delta[lev]), 1)
        plan = o.make_plan({a0 + i: WL.slots(60 + i, m) for i in range(20)}, a0, 1, 20, lev, P.delta[lev], B=1)
        got = K.ckks_bsgs(ctx, keys, import_ct(K, ctx, ct), import_plan(K, ctx, plan))
        assert_ct_equal(K, ctx, got, o.bsgs(ct, plan), "20 giant steps from %d" % a0)
        K.ckks_sync(ctx)
    finally:
        del WL.PARAMS["fold_test"]
        K = o = ctx = keys = ct = got = plan = None
        gc.collect()

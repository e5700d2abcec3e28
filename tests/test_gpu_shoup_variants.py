"""Launch variants of the N = 2^16 transforms in a context on Shoup products (a 61-bit base prime): the one
asked for is the one that runs, and operations that use the transforms in every form (in place, out of
place, limb lists, output factors, host memory) give the same words with each."""
import ctypes

import pytest

import workloads as WL

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_variants_run_and_agree():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_04356_gb300 import build
    from paper_2312_04356_gb300 import ckks as K
    build.build()
    d = dict(log_n=16, n_q=9, dnum=2, n_p=0, q0_bits=61, scale_bits=42, p_bits=60, boot_bits=0, n_boot=0, h=0, sigma=3.2)
    ctx = K.ckks_ctx_create(d, 3, torch.cuda.current_stream().cuda_stream)
    keys = K.ckks_keygen(ctx, [1, 5], False)
    lev = 8
    ct = K.ckks_encrypt(ctx, keys, K.ckks_encode(ctx, WL.slots(1, 1 << 15, 0.5), lev, 2.0 ** 42), 1)
    host = torch.empty((2, lev + 1, 1 << 16), dtype=torch.int64, pin_memory=True)
    x = torch.zeros((20, 1 << 16), dtype=torch.int64, device="cuda")
    want = None
    for v in range(-1, 6):
        K.ckks_ctx_set_ntt_variant(ctx, v)
        K.ckks_ctx_reset_counters(ctx)
        K.ckks_ntt_forward(ctx, x.data_ptr(), 20, [i % 9 for i in range(20)])
        K.ckks_ntt_inverse(ctx, x.data_ptr(), 20, [i % 9 for i in range(20)])
        assert K.ckks_ctx_counters(ctx)["launches"] == (2 if v == 5 else 4), v     # the cluster takes one launch
        ctx.check(K.lib().ckks_ct_export_rns(ctx, ct, ctypes.c_void_p(host.data_ptr())))
        back = K.ckks_ct_create(ctx)
        ctx.check(K.lib().ckks_ct_import_rns(ctx, ctypes.c_void_p(host.data_ptr()), lev, 2.0 ** 42, back))
        outs = K.ckks_rotate_hoisted(ctx, keys, back, [1, 5])
        outs += [K.ckks_rescale(ctx, K.ckks_mul_relin(ctx, keys, back, ct)), K.ckks_level_down(ctx, ct, 2)]
        outs.append(K.ckks_mod_raise(ctx, K.ckks_mod_drop(ctx, ct, 0)))
        got = [K.ckks_ct_export_rns(ctx, o) for o in outs + [back]]
        want = want or got
        for i, (a, b) in enumerate(zip(got, want)):
            assert (a == b).all(), (v, i)


def test_conversions_and_shapes_agree():
    """tensor-core conversions (one and two threads a coefficient) leave lazy words below 4 p; every transform
    shape takes them to the words that the integer-pipe conversion leads to"""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_04356_gb300 import build
    from paper_2312_04356_gb300 import ckks as K
    build.build()
    d = dict(log_n=16, n_q=6, dnum=2, n_p=0, q0_bits=61, scale_bits=42, p_bits=61, boot_bits=0, n_boot=0, h=0, sigma=3.2)
    ctx = K.ckks_ctx_create(d, 3, torch.cuda.current_stream().cuda_stream)
    keys = K.ckks_keygen(ctx, [3], False)
    ct = K.ckks_encrypt(ctx, keys, K.ckks_encode(ctx, WL.slots(1, 1 << 15, 0.5), 5, 2.0 ** 42), 1)
    want = None
    for mode in (0, 1, 2):
        for v in (-1, 0, 1, 2, 3, 4, 5):
            K.ckks_ctx_set_tensor_conversion(ctx, mode)
            K.ckks_ctx_set_ntt_variant(ctx, v)
            outs = [K.ckks_rotate_hoisted(ctx, keys, ct, [3])[0], K.ckks_mul_relin(ctx, keys, ct, ct)]
            got = [K.ckks_ct_export_rns(ctx, o) for o in outs]
            want = want or got
            for i, (a, b) in enumerate(zip(got, want)):
                assert (a == b).all(), (mode, v, i)

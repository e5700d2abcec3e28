"""Transforms in both arithmetics (folded products for primes next to a power of two, Shoup products
for others) at the ends of their ranges: every one-CTA ring size, the two-pass ring in every
launch variant, and residues at the extremes (all q - 1, 0 / q - 1 alternating), where the lazy
values are largest.  Integers: compared bit for bit with the oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# (log_n, q0_bits, scale_bits, p_bits): primes 2^k +- small qualify for folding up to 60 bits; one
# 61-bit (or below 33-bit) prime puts the whole context on Shoup products
CASES = [(n, 60, 42, 60) for n in (7, 8, 9, 10, 11, 12, 13, 16)] + \
        [(12, 50, 34, 57), (16, 55, 36, 56), (12, 61, 40, 60), (16, 60, 42, 61), (8, 45, 30, 45)]


@pytest.mark.parametrize("log_n,q0,sc,pb", CASES)
def test_transform_extremes_bitexact(log_n, q0, sc, pb):
    from oracle import _clib as C
    from oracle import params as PP
    from paper_2312_04356_gb300 import build
    from paper_2312_04356_gb300 import ckks as K
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    d = dict(log_n=log_n, n_q=4, dnum=1, n_p=1, q0_bits=q0, scale_bits=sc, p_bits=pb, boot_bits=0, n_boot=0, h=0,
             sigma=3.2)
    P = PP.Params(log_n, 4, 1, q0, sc, pb, h=0, n_p=1)
    ctx = K.ckks_ctx_create(d, 1, torch.cuda.current_stream().cuda_stream)
    q, p, _, _ = K.ckks_ctx_info(ctx)
    mods = q + p
    assert mods == list(P.q) + list(P.p)
    n, ids = 1 << log_n, list(range(len(mods))) * 4
    g = np.random.default_rng(3)
    rows = []
    for fill in ("top", "alternate", "random", "impulse"):
        for m in mods:
            if fill == "top":
                r = np.full(n, m - 1, dtype=np.uint64)
            elif fill == "alternate":
                r = np.where(np.arange(n) % 2 == 0, 0, m - 1).astype(np.uint64)
            elif fill == "random":
                r = g.integers(0, m, n, dtype=np.uint64)
            else:
                r = np.zeros(n, dtype=np.uint64)
                r[-1] = m - 1
            rows.append(r)
    x = np.stack(rows)
    psi = (list(P.psi_q) + list(P.psi_p)) * 4
    fwd = C.ntt_forward(x, mods * 4, psi, log_n)
    inv = C.ntt_inverse(x, mods * 4, psi, log_n)
    for variant in range(-1, 6) if log_n == 16 else [-1]:
        K.ckks_ctx_set_ntt_variant(ctx, variant)
        for call, want in ((K.ckks_ntt_forward, fwd), (K.ckks_ntt_inverse, inv)):
            dev = torch.from_numpy(x.view(np.int64).copy()).cuda()
            call(ctx, dev.data_ptr(), len(ids), ids)
            torch.cuda.synchronize()
            assert (dev.cpu().numpy().view(np.uint64) == want).all(), (variant, call.__name__)


# id lists that are runs of consecutive primes (whole, cut off, not from the first prime, one prime) and
# lists that are not: each against every limb transformed by itself
@pytest.mark.parametrize("log_n", [9, 13, 16])
@pytest.mark.parametrize("ids", [[0, 1, 2, 3, 4, 0, 1, 2], [2, 3, 4, 2, 3, 4, 2], [3, 3, 3], [4], [0, 1, 2, 4], [2, 1, 0],
                                 [0, 1, 0, 2], [1, 2, 1, 2, 3], [0, 0, 1, 1]])
def test_id_lists_match_single_limbs(log_n, ids):
    from paper_2312_04356_gb300 import build
    from paper_2312_04356_gb300 import ckks as K
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    d = dict(log_n=log_n, n_q=4, dnum=1, n_p=1, q0_bits=60, scale_bits=42, p_bits=60, boot_bits=0, n_boot=0, h=0, sigma=3.2)
    ctx = K.ckks_ctx_create(d, 1, torch.cuda.current_stream().cuda_stream)
    q, p, _, _ = K.ckks_ctx_info(ctx)
    g = np.random.default_rng(5)
    x = np.stack([g.integers(0, (q + p)[i], 1 << log_n, dtype=np.uint64) for i in ids]).view(np.int64)
    for call in (K.ckks_ntt_forward, K.ckks_ntt_inverse):
        dev, one = torch.from_numpy(x.copy()).cuda(), torch.from_numpy(x.copy()).cuda()
        call(ctx, dev.data_ptr(), len(ids), ids)
        for k, i in enumerate(ids):
            call(ctx, one[k].data_ptr(), 1, [i])
        torch.cuda.synchronize()
        assert torch.equal(dev, one), call.__name__


# limbs that cross the host boundary in pinned memory (read and written by the transforms) and in pageable
# memory (copied), whole buffers and parts of one: the same words, and back what went in
@pytest.mark.parametrize("log_n,q0", [(9, 60), (12, 61), (13, 60), (16, 60), (16, 61)])
def test_pinned_and_pageable_limbs_agree(log_n, q0):
    import ctypes

    from paper_2312_04356_gb300 import build
    from paper_2312_04356_gb300 import ckks as K
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    d = dict(log_n=log_n, n_q=9, dnum=1, n_p=1, q0_bits=q0, scale_bits=42, p_bits=60, boot_bits=0, n_boot=0, h=0, sigma=3.2)
    ctx = K.ckks_ctx_create(d, 1, torch.cuda.current_stream().cuda_stream)
    q, _, _, _ = K.ckks_ctx_info(ctx)
    g = np.random.default_rng(7)
    pool = torch.zeros((2 * 9 + 2) << log_n, dtype=torch.int64).pin_memory()
    for level in (0, 3, 8):
        x = np.stack([[g.integers(0, q[i], 1 << log_n, dtype=np.uint64) for i in range(level + 1)] for _ in range(2)])
        for variant in (-1, 4) if log_n == 16 else (-1,):
            K.ckks_ctx_set_ntt_variant(ctx, variant)
            for skip in (0, 1, 1 << log_n):           # the buffer's start, an odd word, a whole limb further
                pool.zero_()
                host = pool[skip:skip + x.size]
                host.copy_(torch.from_numpy(x.view(np.int64).ravel()))
                ct, out = K.ckks_ct_create(ctx), pool[skip:skip + x.size]
                ctx.check(K.lib().ckks_ct_import_rns(ctx, ctypes.c_void_p(host.data_ptr()), level, 2.0 ** 42, ct))
                K.ckks_sync(ctx)
                ref = K.ckks_ct_import_rns(ctx, x, level, 2.0 ** 42)
                assert (K.ckks_ct_export_rns(ctx, ct) == x).all() and (K.ckks_ct_export_rns(ctx, ref) == x).all()
                out.zero_()
                ctx.check(K.lib().ckks_ct_export_rns(ctx, ref, ctypes.c_void_p(out.data_ptr())))
                assert (out.numpy().view(np.uint64).reshape(x.shape) == x).all(), (level, variant, skip)
                assert not pool[:skip].any() and not pool[skip + x.size:].any(), "words outside the buffer"
    K.ckks_ctx_set_ntt_variant(ctx, -1)

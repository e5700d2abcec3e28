"""Grouped rotations and giant steps under a fixed memory budget: with room for one at a time the calls
still run, return the same words as with room for all, and hold no more than the budget; without that
room they report CKKS_ENOMEM and the context stays usable."""
import numpy as np
import pytest

import workloads as WL

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


class Budget:
    """a caller allocator that holds at most `limit` bytes"""

    def __init__(self, limit=None):
        self.limit, self.live, self.peak, self.size = limit, 0, 0, {}

    def alloc(self, nbytes, stream):
        if self.limit is not None and self.live + nbytes > self.limit:
            return 0
        p = torch.cuda.caching_allocator_alloc(nbytes, 0, stream)
        self.size[p] = nbytes
        self.live += nbytes
        self.peak = max(self.peak, self.live)
        return p

    def free(self, ptr, nbytes, stream):
        self.live -= self.size.pop(ptr)
        torch.cuda.caching_allocator_delete(ptr)


@pytest.mark.parametrize("q0", [60, 61])
@pytest.mark.parametrize("log_n,n_q,dnum", [(12, 4, 2), (13, 6, 3), (10, 4, 4)])
def test_calls_fit_where_one_at_a_time_fits(log_n, n_q, dnum, q0):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_04356_gb300 import build
    from paper_2312_04356_gb300 import ckks as K
    build.build()
    d = dict(log_n=log_n, n_q=n_q, dnum=dnum, n_p=0, q0_bits=q0, scale_bits=42, p_bits=60, boot_bits=0, n_boot=0, h=0, sigma=3.2)
    ctx = K.ckks_ctx_create(d, 3, torch.cuda.current_stream().cuda_stream)
    q, p, _, delta = K.ckks_ctx_info(ctx)
    n, lev = ctx.n, n_q - 1
    nl, nxt = n_q, n_q + len(p)
    keys = K.ckks_keygen(ctx, list(range(1, 9)) + [12, 16, 20], False)
    ct = K.ckks_encrypt(ctx, keys, K.ckks_encode(ctx, WL.slots(1, n // 2, 0.5), lev, delta[lev]), 1)
    g = np.random.default_rng(5)

    def plan(a0, count, B):
        ps = K.ckks_ptset_create(ctx, a0, 1, count, B, lev, delta[lev])
        for i in range(count):
            K.ckks_ptset_set_rns(ctx, ps, i // B, i % B, np.stack([g.integers(0, m, n, dtype=np.uint64) for m in q + p]))
        return ps

    two, split, rotated = 2 * nxt, plan(0, 16, 4), plan(4, 16, 4)      # two: a sum over Q u P, in limbs
    one = nl + dnum * nxt + nl                                         # c1 brought down, digits, coefficients
    steps = list(range(1, 9))
    calls = [
        # eight rotations: digits, one sum and its ModDown, the results
        (dnum * nxt + two + 2 * nl + 8 * 2 * nl, lambda: K.ckks_rotate_hoisted(ctx, keys, ct, steps)),
        # four giant steps, three of them rotated: the inner sums and one giant at a time
        (4 * two + one, lambda: [K.ckks_bsgs(ctx, keys, ct, split)]),
        # all rotated: their sum as well
        (4 * two + two + one, lambda: [K.ckks_bsgs(ctx, keys, ct, rotated)]),
    ]
    for limbs, call in calls:
        want = [K.ckks_ct_export_rns(ctx, o) for o in call()]
        free = Budget()
        tight = Budget(limbs * n * 8)
        for b in (free, tight):
            K.ckks_ctx_set_allocator(ctx, b.alloc, b.free)
            outs = call()
            K.ckks_ctx_set_allocator(ctx)
            got = [K.ckks_ct_export_rns(ctx, o) for o in outs]
            del outs
            assert all((x == y).all() for x, y in zip(got, want))
        assert tight.peak <= tight.limit < free.peak        # the group did not fit, one did
        short = Budget(limbs * n * 8 // 3)
        K.ckks_ctx_set_allocator(ctx, short.alloc, short.free)
        with pytest.raises(K.CkksError) as e:
            call()
        K.ckks_ctx_set_allocator(ctx)
        assert e.value.code == K.CKKS_ENOMEM and short.live == 0
        assert all((K.ckks_ct_export_rns(ctx, o) == w).all() for o, w in zip(call(), want))

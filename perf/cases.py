"""The work this library is measured on: calls that a program using it makes, through the public
binding, over the range of sizes it is used at.

Two rings: N = 2^12 with a short chain (one conv layer, the smallest useful circuit) and the
N = 2^16, 24-limb chain that bootstraps.  A program keeps one context, its keys, plaintext sets
and bootstrapping configurations for as long as it serves a model, so they are made once per
ring and shared by every state; what changes from call to call is the ciphertexts, images and
residues, which prepare() draws from its seed.  Ciphertexts that come from or go to a client
cross as coefficient-domain limbs in pinned host memory, as a server handles them; raw-array
calls work on device tensors.
"""
import ctypes
import math

import numpy as np
import torch

import paper_2312_04356_gb300.ckks as K

RINGS = {
    # N = 2^12, 4 limbs (60, 3 x 40 bits), 2 special primes
    "small": dict(log_n=12, n_q=4, dnum=2, n_p=0, q0_bits=60, scale_bits=40, p_bits=60, boot_bits=0, n_boot=0, h=0,
                  sigma=3.2),
    # N = 2^16, 24 limbs (60, 9 x 42, 14 x 48 bits), 7 special primes, dnum 3, h = 192
    "boot": dict(log_n=16, n_q=24, dnum=3, n_p=7, q0_bits=60, scale_bits=42, p_bits=60, boot_bits=48, n_boot=14,
                 h=192, sigma=3.2),
}
DELTA0 = 2.0 ** 49          # scale of the level-0 ciphertext that enters ModRaise
SLOTS = 4                   # requests a server keeps in flight


def listed():
    return [
        # one fused conv layer on the small ring: about twenty launches over a few limbs of 32 KB,
        # the smallest request a server answers (launch latency)
        dict(name="conv_small", kind="conv", ring="small", channels=1, width=16, f=3, level=3),
        # a rescale on caller-owned device arrays at a middle level: the shortest device-only call
        dict(name="rescale", kind="rescale", level=9),
        # forward and inverse transforms of a top-level ciphertext's 48 limbs: what importing and
        # exporting it cost
        dict(name="ntt", kind="ntt", limbs=48),
        # HMult + relinearise + rescale in the middle of the chain, the step of any encrypted product
        dict(name="mult", kind="mult", level=15),
        # rotate-and-sum over eight steps at the top circuit level (pooling, inner products)
        dict(name="rotate_sum", kind="rotate", level=9, steps=8),
        # conv2d of 16 channels 32 x 32 fused with StoC2 at level 1, the layer before a bootstrap
        dict(name="conv", kind="conv", ring="boot", channels=16, width=32, f=3, level=1),
        # one conv + bootstrap block, recorded once and replayed per request (16 x 32 x 32): the
        # library's headline use
        dict(name="block", kind="block", channels=16, width=32, graph=True),
        # the same network's middle stage (32 x 16 x 16) with eight requests in lockstep
        dict(name="block_batch", kind="batch", channels=32, width=16, batch=8),
        # a downsampling layer: two ciphertexts of 16 x 32 x 32 into 64 x 16 x 16
        dict(name="downsample", kind="downsample", channels=32, width=32),
        # the composite polynomial ReLU from the top level (18 levels)
        dict(name="relu", kind="relu", level=23, stages="15,15,27"),
        # twelve requests through the serving loop, every third a two-block model
        dict(name="serve", kind="serve", requests=12),
        # the client's two ends: encode + encrypt an image, decrypt + decode a result
        dict(name="client", kind="client", channels=16, width=32, level=5),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["conv_small", "rescale", "ntt", "mult", "rotate", "conv", "block", "batch", "downsample", "relu",
                       "serve", "client"])
    if kind == "conv_small":
        width = rng.randint(5, 30)
        w = _padded(width, 3)
        return dict(kind="conv", ring="small", channels=rng.randint(1, 4096 // (w * w)), width=width,
                    f=rng.choice([1, 3, 5]) if _padded(width, 5) == w else 3, level=rng.randint(1, 3))
    if kind == "rescale":
        return dict(kind="rescale", level=rng.randint(1, 23))
    if kind == "ntt":
        return dict(kind="ntt", limbs=_log_int(rng, 1, 256))
    if kind == "mult":
        return dict(kind="mult", level=rng.randint(1, 23))
    if kind == "rotate":
        return dict(kind="rotate", level=rng.randint(0, 23), steps=rng.randint(1, 12))
    if kind == "conv":
        width = rng.randint(12, 48)
        w = _padded(width, 3)
        return dict(kind="conv", ring="boot", channels=rng.randint(1, 65536 // (w * w)), width=width, f=3,
                    level=rng.randint(1, 9))
    if kind in ("block", "batch"):
        width = rng.randint(8, 40)
        w = _padded(width, 3)
        channels = rng.randint(1, min(64, 65536 // (w * w)))
        if kind == "batch":
            return dict(kind="batch", channels=channels, width=width, batch=rng.randint(2, 8))
        return dict(kind="block", channels=channels, width=width, graph=rng.random() < 0.5)
    if kind == "downsample":
        return dict(kind="downsample", channels=rng.randint(1, 32), width=2 * rng.randint(16, 20))
    if kind == "relu":
        stages = [rng.choice([3, 5, 7, 9, 13, 15, 21, 27]) for _ in range(rng.randint(1, 3))]
        need = _relu_levels(stages)
        return dict(kind="relu", level=rng.randint(need + 1, 23), stages=",".join(str(d) for d in stages))
    if kind == "serve":
        return dict(kind="serve", requests=rng.randint(2, 12))
    return dict(kind="client", channels=rng.randint(1, 16), width=rng.randint(8, 32), level=rng.randint(1, 9))


def _padded(width, f):
    w = 1
    while w < width + f // 2:
        w *= 2
    return w


def _relu_levels(stages):
    """levels of the composite (one more where it crosses between the chain's segments)"""
    return sum(math.ceil(math.log2(d)) + 1 for d in stages) + 2


# --------------------------------------------------------- what a program keeps ---
class _Ring:
    """one context on a stream of its own, its keys (rotation keys added as plans need them) and
    the plans made so far"""

    def __init__(self, name):
        self.name = name
        self.stream = torch.cuda.Stream()
        self.ctx = K.ckks_ctx_create(RINGS[name], 2024, self.stream.cuda_stream)
        self.q, self.p, _, self.delta = K.ckks_ctx_info(self.ctx)
        self.n = self.ctx.n
        self.keys = K.ckks_keygen(self.ctx, [], True)
        self.have = set()
        self.plans = {}

    def need(self, steps):
        new = sorted(set(int(s) % (self.n // 2) for s in steps) - self.have - {0})
        if new:
            K.ckks_keys_add_rotations(self.ctx, self.keys, new)
            self.have |= set(new)

    def plan(self, key, make):
        if key not in self.plans:
            self.plans[key] = make()
            K.ckks_sync(self.ctx)
        return self.plans[key]

    def conv_scale(self, level):
        """plaintext scale after which a rescale lands on the next canonical scale (at level 1: on
        the scale ModRaise takes)"""
        below = DELTA0 if level == 1 and self.name == "boot" else self.delta[level - 1]
        return below * self.q[level] / self.delta[level]

    def conv(self, channels, width, f, level):
        def make():
            w = _padded(width, f)
            W = np.random.default_rng(11).normal(0.0, 0.1, (channels, channels, f, f))
            ps = K.ckks_ptset_conv_fused(self.ctx, W, channels, channels, f, w, level, self.conv_scale(level))
            self.need(K.ckks_ptset_rotations(ps))
            return ps
        return self.plan(("conv", channels, width, f, level), make)

    def boot(self, w, width, channels, stride=1):
        def make():
            bt = K.ckks_boot_create(self.ctx, w, width, channels, stride=stride)
            self.need(K.ckks_boot_rotations(bt))
            return bt
        return self.plan(("boot", w, width, channels, stride), make)

    def graph(self, channels, width):
        """a recorded block, the buffers it reads and writes, and a handle to import requests into"""
        def make():
            conv, bt = self.conv(channels, width, 3, 1), self.boot(_padded(width, 3), width, channels)
            src = self.encrypt_image(np.zeros((channels, width, width)), _padded(width, 3), 1, 1)
            dst = K.ckks_ct_create(self.ctx)
            return dict(src=src, dst=dst, stage=K.ckks_ct_create(self.ctx),
                        graph=K.ckks_block_graph_create(self.ctx, self.keys, src, conv, bt, dst))
        return self.plan(("graph", channels, width), make)

    def server(self):
        def make():
            conv, bt = self.conv(16, 32, 3, 1), self.boot(64, 32, 16)
            srv = K.ckks_server_create(self.ctx, self.keys, SLOTS)
            models = [K.ckks_server_add_model(srv, [conv] * n, [bt] * n) for n in (1, 2)]
            K.ckks_server_start(srv)
            return srv, models
        return self.plan("server", make)

    def encrypt_image(self, img, w, level, nonce):
        return K.ckks_encrypt(self.ctx, self.keys, K.ckks_encode_image(self.ctx, img, w, level, self.delta[level]),
                              nonce)

    def encrypt_slots(self, values, level, nonce, scale=None):
        pt = K.ckks_encode(self.ctx, values, level, scale or self.delta[level])
        return K.ckks_encrypt(self.ctx, self.keys, pt, nonce)

    def pinned(self, level):
        return torch.empty((2, level + 1, self.n), dtype=torch.int64, pin_memory=True)

    def export(self, ct, host):
        """the ciphertext's limbs into a pinned buffer (returns when they are there)"""
        self.ctx.check(K.lib().ckks_ct_export_rns(self.ctx, ct, ctypes.c_void_p(host.data_ptr())))
        return host

    def load(self, host, level, out):
        """a client's limbs from a pinned buffer into a ciphertext handle"""
        self.ctx.check(K.lib().ckks_ct_import_rns(self.ctx, ctypes.c_void_p(host.data_ptr()), level,
                                                  self.delta[level], out))
        return out

    def request(self, ct, level):
        """a ciphertext as a client sends it: limbs in pinned memory"""
        return self.export(ct, self.pinned(level))


_rings = {}


def _ring(name):
    if name not in _rings:
        _rings[name] = _Ring(name)
    return _rings[name]


def _stages(case):
    """odd sign-like fits, the last one (1 + sign) / 2: the coefficients of a composite ReLU"""
    nodes = np.cos(np.pi * (np.arange(4096) + 0.5) / 4096)
    degs = [int(d) for d in case["stages"].split(",")]
    out = []
    for i, d in enumerate(degs):
        last = i == len(degs) - 1
        c = np.polynomial.chebyshev.chebfit(nodes, (1 + np.tanh(8 * nodes)) / 2 if last else np.tanh(5 * nodes), d)
        if not last:
            c[0::2] = 0.0
        out.append(c)
    return out


# ---------------------------------------------------------------------- prepare ---
def prepare(case, seed):
    kind = case["kind"]
    g = np.random.default_rng(seed)
    r = _ring(case.get("ring", "boot"))
    nonce = 1 + seed * 64
    s = dict(kind=kind, r=r)
    with torch.cuda.stream(r.stream):
        if kind in ("rescale", "ntt"):
            gen = torch.Generator(device="cuda")
            gen.manual_seed(seed)
            if kind == "rescale":
                s["level"] = case["level"]
                ids = list(range(case["level"] + 1)) * 2
                shape = (2, case["level"] + 1, r.n)
                s["out"] = torch.empty((2, case["level"], r.n), dtype=torch.int64, device="cuda")
            else:
                ids = [i % len(r.q) for i in range(case["limbs"])]
                shape = (case["limbs"], r.n)
            x = torch.stack([torch.randint(0, r.q[i], (r.n,), generator=gen, device="cuda") for i in ids])
            s["x"], s["ids"] = x.view(shape), ids
            if kind == "ntt":
                s["fwd"], s["inv"] = torch.empty_like(s["x"]), torch.empty_like(s["x"])
        elif kind == "conv":
            w = _padded(case["width"], case["f"])
            s["level"] = case["level"]
            s["conv"] = r.conv(case["channels"], case["width"], case["f"], case["level"])
            ct = r.encrypt_image(g.random((case["channels"], case["width"], case["width"])), w, case["level"], nonce)
            s["host"], s["out"] = r.request(ct, case["level"]), r.pinned(case["level"] - 1)
            s["ct"], s["res"] = K.ckks_ct_create(r.ctx), K.ckks_ct_create(r.ctx)
        elif kind == "mult":
            s["a"], s["b"] = [r.encrypt_slots(g.uniform(-1, 1, r.n // 2), case["level"], nonce + i) for i in (0, 1)]
            s["prod"], s["res"] = K.ckks_ct_create(r.ctx), K.ckks_ct_create(r.ctx)
            s["out"] = r.pinned(case["level"] - 1)
        elif kind == "rotate":
            s["steps"] = [1 << i for i in range(case["steps"])]
            r.need(s["steps"])
            s["ct"] = r.encrypt_slots(g.uniform(-1, 1, r.n // 2), case["level"], nonce)
            s["rot"] = [K.ckks_ct_create(r.ctx) for _ in s["steps"]]
            s["res"], s["out"] = K.ckks_ct_create(r.ctx), r.pinned(case["level"])
        elif kind in ("block", "batch"):
            w = _padded(case["width"], 3)
            s["conv"] = r.conv(case["channels"], case["width"], 3, 1)
            s["bt"] = r.boot(w, case["width"], case["channels"])
            nb = case.get("batch", 1)
            cts = [r.encrypt_image(g.random((case["channels"], case["width"], case["width"])), w, 1, nonce + i)
                   for i in range(nb)]
            lev = int(K.ckks_boot_info(s["bt"])["l_out"])
            s["host"] = [r.request(ct, 1) for ct in cts]
            s["out"] = [r.pinned(lev) for _ in cts]
            s["ct"] = cts
            s["res"] = [K.ckks_ct_create(r.ctx) for _ in cts]
            s["graph"] = r.graph(case["channels"], case["width"]) if case.get("graph") else None
        elif kind == "downsample":
            c, width = case["channels"], case["width"]
            w = _padded(width, 3)
            n_in = -(-c * w * w // r.n)              # N / w^2 channels per ciphertext
            s["bt_in"] = r.boot(w, width, min(c, r.n // (w * w)), stride=2)
            s["bt_out"] = r.boot(w // 2, width // 2, min(2 * c, 4 * r.n // (w * w)))

            def make():
                W = np.random.default_rng(12).normal(0.0, 0.1, (min(2 * c, 4 * r.n // (w * w)), c, 3, 3))
                sets = [K.ckks_ptset_conv_fused_s2(r.ctx, W, c, len(W), 3, w, t, 1, r.conv_scale(1))
                        for t in range(n_in)]
                for ps in sets:
                    r.need(K.ckks_ptset_rotations(ps))
                return sets
            s["convs"] = r.plan(("s2", c, width), make)
            info = K.ckks_boot_info(s["bt_in"])
            lev, sc = int(info["l_em"]), info["s_em"]
            half = [[r.encrypt_slots(1e-3 * g.uniform(-1, 1, r.n // 2), lev, nonce + 2 * t + i, sc) for t in range(n_in)]
                    for i in (0, 1)]
            s["re"], s["im"] = half
            s["res"], s["out"] = K.ckks_ct_create(r.ctx), r.pinned(int(K.ckks_boot_info(s["bt_out"])["l_out"]))
        elif kind == "relu":
            s["stages"] = _stages(case)
            s["ct"] = r.encrypt_slots(g.uniform(-1, 1, r.n // 2), case["level"], nonce)
            s["res"] = K.ckks_ct_create(r.ctx)

            def out_level():
                return K.ckks_ct_info(K.ckks_eval_relu(r.ctx, r.keys, s["ct"], s["stages"]))[0]
            s["out"] = r.pinned(r.plan(("relu", case["level"], case["stages"]), out_level))
        elif kind == "serve":
            s["srv"], s["models"] = r.server()
            s["host"] = [r.request(r.encrypt_image(g.random((16, 32, 32)), 64, 1, nonce + i), 1).numpy().view(np.uint64)
                         for i in range(case["requests"])]
        elif kind == "client":
            w = _padded(case["width"], 3)
            s["w"], s["nonce"], s["level"], s["shape"] = w, nonce + 1, case["level"], (case["channels"], case["width"])
            s["img"] = _client_image(case, seed)
            s["host"], s["back"] = r.pinned(1), r.encrypt_image(s["img"], w, case["level"], nonce)
            s["pt"], s["ct"] = K.ckks_pt_create(r.ctx), K.ckks_ct_create(r.ctx)
            s["dec"] = K.ckks_pt_create(r.ctx)
        K.ckks_sync(r.ctx)
    return s


def _client_image(case, seed):
    return np.random.default_rng(seed + 1).random((case["channels"], case["width"], case["width"]))


# -------------------------------------------------------------------------- run ---
def run(s):
    r, kind = s["r"], s["kind"]
    ctx, keys = r.ctx, r.keys
    if kind == "rescale":
        K.ckks_rescale_noalloc(ctx, s["x"].data_ptr(), s["level"], s["out"].data_ptr())
        return s["out"]
    if kind == "ntt":
        with torch.cuda.stream(r.stream):        # the transforms work in place
            s["fwd"].copy_(s["x"])
            s["inv"].copy_(s["x"])
        K.ckks_ntt_forward(ctx, s["fwd"].data_ptr(), len(s["ids"]), s["ids"])
        K.ckks_ntt_inverse(ctx, s["inv"].data_ptr(), len(s["ids"]), s["ids"])
        return s["fwd"], s["inv"]
    if kind == "conv":
        r.load(s["host"], s["level"], s["ct"])
        K.ckks_conv2d_cins(ctx, keys, s["ct"], s["conv"], s["res"])
        return r.export(s["res"], s["out"])
    if kind == "mult":
        K.ckks_mul_relin(ctx, keys, s["a"], s["b"], s["prod"])
        K.ckks_rescale(ctx, s["prod"], s["res"])
        return r.export(s["res"], s["out"])
    if kind == "rotate":
        acc = s["ct"]
        for t in K.ckks_rotate_hoisted(ctx, keys, s["ct"], s["steps"], s["rot"]):
            acc = K.ckks_add(ctx, acc, t, s["res"])
        return r.export(acc, s["out"])
    if kind == "block" and s["graph"]:
        g = s["graph"]
        r.load(s["host"][0], 1, g["stage"])
        K.ckks_ct_copy_into(ctx, g["stage"], g["src"])
        K.ckks_graph_launch(g["graph"])
        return r.export(g["dst"], s["out"][0])
    if kind in ("block", "batch"):
        for host, ct in zip(s["host"], s["ct"]):
            r.load(host, 1, ct)
        if kind == "block":
            K.ckks_block(ctx, keys, s["ct"][0], s["conv"], s["bt"], s["res"][0])
        else:
            K.ckks_block_batched(ctx, keys, s["ct"], s["conv"], s["bt"], s["res"])
        return [r.export(ct, out) for ct, out in zip(s["res"], s["out"])]
    if kind == "downsample":
        K.ckks_downsample_layer(ctx, keys, s["re"], s["im"], s["bt_in"], s["convs"], s["bt_out"], s["res"])
        return r.export(s["res"], s["out"])
    if kind == "relu":
        K.ckks_eval_relu(ctx, keys, s["ct"], s["stages"], s["res"])
        return r.export(s["res"], s["out"])
    if kind == "serve":
        ids = [K.ckks_server_submit(s["srv"], s["models"][i % 3 == 2], h, 1, r.delta[1])
               for i, h in enumerate(s["host"])]
        for rid in ids:
            K.ckks_server_wait(s["srv"], rid)
        return [K.ckks_server_result(s["srv"], rid, r.n)[0].view(np.int64) for rid in ids]
    # client
    K.ckks_encode_image(ctx, s["img"], s["w"], 1, r.delta[1], s["pt"])
    K.ckks_encrypt(ctx, keys, s["pt"], s["nonce"], s["ct"])
    limbs = r.export(s["ct"], s["host"])
    K.ckks_decrypt(ctx, keys, s["back"], s["dec"])
    return {"limbs": limbs, "image": K.ckks_decode_image(ctx, s["dec"], s["shape"][0], s["shape"][1], s["w"])}


# ------------------------------------------------------------------------- work ---
def _limbs(nq, n=65536):
    return 8.0 * n * nq


def _hmatmul(level, diags, rots, np_=7, alpha=8, n=65536):
    """keys of its rotations and diagonals over Q_level u P, each read once, and the ciphertext in
    and out"""
    ndig = -(-(level + 1) // alpha)
    return _limbs((level + 1 + np_) * (2 * ndig * rots + diags) + 4 * (level + 1), n)


def _conv_bytes(case):
    if case.get("ring") == "small":
        c = 4096 // _padded(case["width"], case["f"]) ** 2
        return _hmatmul(case["level"], c, max(0, 2 * math.sqrt(c) - 2), 2, 2, 4096)
    c = 65536 // _padded(case["width"], case.get("f", 3)) ** 2
    return _hmatmul(case.get("level", 1), c, max(0, 2 * math.sqrt(c) - 2))


def _block_bytes(nb=1):
    """the rotation and relinearisation keys, the bootstrapping diagonals, and per ciphertext its
    limbs in and out"""
    maps = sum(_hmatmul(lev, 63, 18) for lev in (23, 22, 21)) + sum(_hmatmul(lev, 31, 16) for lev in (8, 7, 6))
    return maps + _limbs(2 * 3 * 27) + nb * _limbs(4 + 12)


def work(case):
    kind = case["kind"]
    if kind == "rescale":
        b = _limbs(4 * case["level"] + 2)
    elif kind == "ntt":
        b = _limbs(3 * case["limbs"])
    elif kind == "conv":
        b = _conv_bytes(case)
    elif kind == "mult":
        ndig = -(-(case["level"] + 1) // 8)
        b = _limbs(6 * case["level"] + 4 + 2 * ndig * (case["level"] + 8))
    elif kind == "rotate":
        ndig = -(-(case["level"] + 1) // 8)
        b = _limbs(4 * (case["level"] + 1) + case["steps"] * 2 * ndig * (case["level"] + 8))
    elif kind in ("block", "batch"):
        b = _block_bytes(case.get("batch", 1)) + _conv_bytes(case)
    elif kind == "downsample":
        b = _block_bytes() + -(-case["channels"] // 16) * (_hmatmul(8, 127, 22) + sum(_hmatmul(lev, 31, 12) for lev in (7, 6, 5)))
    elif kind == "relu":
        b = _limbs(2 * (case["level"] + 1) + 12 + 2 * 3 * (case["level"] + 8))      # in, out, the key
    elif kind == "serve":
        b = _block_bytes(case["requests"])
    else:
        b = _limbs(4 + 2 * (case["level"] + 1)) + 16.0 * case["channels"] * case["width"] ** 2
    # the arithmetic is 64-bit modular, no floating point
    return {"bytes": b, "flops": 0}


# ------------------------------------------------------------------------ exact ---
def exact(case, seed):
    """limbs are whole numbers; the client's decoded image is the image it encrypted"""
    if case["kind"] != "client":
        return None
    return {"limbs": None, "image": _client_image(case, seed)}

"""The calls this library is measured on: pixel-level CKKS encryption, image operations on the
ciphertexts and decryption, through the binding's public functions (paper_2409_03568_gb300.ichee).

listed() are the cases, draw() makes more of the same ranges, prepare() builds what a program holds
before the call (context, keys, caches, input images, output buffers), run() is one pass of the
calls. Rings are those of the library's own workloads and tests. Every ciphertext word and every
decoded value is a deterministic function of the seeds, so ciphertexts are compared exactly.
"""
import math

import numpy as np
import torch

from paper_2409_03568_gb300 import ichee, inputs

# Parameter sets: the toy ring, the paper's N = 2^12 / 109-bit set, the encryption ring, the
# image-operation ring with one more prime, the large serving ring.
RINGS = {
    "n1024": dict(log_n=10, prime_bits=[30, 30], log2_scale=25, special_bits=0),
    "n1024l4": dict(log_n=10, prime_bits=[60, 40, 40, 40], log2_scale=40, special_bits=61),
    "n2048": dict(log_n=11, prime_bits=[45, 30, 30], log2_scale=30, special_bits=50),
    "n4096": dict(log_n=12, prime_bits=[45, 32, 32], log2_scale=32, special_bits=50),
    "n8192": dict(log_n=13, prime_bits=[60, 40, 60], log2_scale=40, special_bits=61),
    "n8192l4": dict(log_n=13, prime_bits=[60, 40, 40, 40], log2_scale=40, special_bits=61),
    "n16384": dict(log_n=14, prime_bits=[60, 40, 40, 40, 40], log2_scale=40, special_bits=61),
}


def listed():
    return [
        # the smallest call: an 8x8 image from host memory, encrypted and decrypted back to the
        # host (launch and copy latency)
        dict(name="roundtrip_n1024_8x8", kind="roundtrip", ring="n1024", h=8, w=8, c=1),
        # an odd-sized colour thumbnail on the paper's own ring: encrypt, filter, decrypt
        dict(name="chain_n4096_24x17x3", kind="chain", ring="n4096", h=24, w=17, c=3),
        # fresh encryption of a whole grayscale image (no cache: the baseline of the method, the
        # way caches are filled, and what scanning caches do for values they lack)
        dict(name="fresh_n8192_64x64", kind="encrypt", ring="n8192", h=64, w=64, c=1, cache="fresh"),
        # the same on the large ring, a small odd-sized tile
        dict(name="fresh_n16384_23x37", kind="encrypt", ring="n16384", h=23, w=37, c=1, cache="fresh"),
        # the scanning cache: 32 most frequent values, pool of 64 zeros, misses encrypted fresh
        dict(name="freq32_n8192_64x64", kind="encrypt", ring="n8192", h=64, w=64, c=1, cache="freq32"),
        # the full cache with its pool on the serving ring, a colour image
        dict(name="full_n16384_48x48x3", kind="encrypt", ring="n16384", h=48, w=48, c=3, cache="full"),
        # 3x3 mean filter of a colour image (the largest single operation)
        dict(name="meanfilter_n8192l4_128x128x3", kind="meanfilter", ring="n8192l4", h=128, w=128, c=3),
        # watermark: blend with a one-channel encrypted pattern, odd size
        dict(name="blend_n8192l4_97x61x3", kind="blend", ring="n8192l4", h=97, w=61, c=3),
        # matching of two images (one relinearised sum of squared differences)
        dict(name="match_n8192_64x64", kind="match", ring="n8192", h=64, w=64, c=1),
        # matching of two small tiles on the serving ring: the relinearisation's chain of short
        # kernels counts as much as the sum
        dict(name="match_n16384_9x11x3", kind="match", ring="n16384", h=9, w=11, c=3),
        # decryption of an image into device memory
        dict(name="decrypt_n8192_64x64", kind="decrypt", ring="n8192", h=64, w=64, c=1, limbs=3),
        # the batched pipeline: a ragged batch of grayscale images, radix-16 encryption and mean
        # filter, every filtered image decrypted
        dict(name="batch_n8192_16x16to80", kind="batch", ring="n8192", images=16, lo=16, hi=80, cache="radix16"),
    ]


# Pixels per call of each kind at N = 8192 with three limbs (smallest, largest); other rings in
# proportion to the size of a ciphertext.
_RANGE = {"roundtrip": (1, 1024), "chain": (16, 4096), "encrypt": (1, 4096), "cached": (1, 16384),
          "meanfilter": (9, 24576), "blend": (1, 16384), "brightness": (1, 16384), "match": (1, 4096),
          "sqdiff": (1, 2048), "decrypt": (1, 16384), "batch": (64, 16384)}
_CACHES = ["radix16", "radix10", "radix10plain", "radix2", "freq32", "freq32radix", "full"]


def draw(rng):
    kind = rng.choice(["roundtrip", "chain", "encrypt", "cached", "cached", "meanfilter", "blend", "brightness",
                       "match", "match", "sqdiff", "decrypt", "batch"])
    keyed = [r for r in RINGS if RINGS[r]["special_bits"]]   # matching needs the special prime
    ring = rng.choice(keyed if kind in ("match", "sqdiff") else list(RINGS))
    size = 3 * 8192 / (len(RINGS[ring]["prime_bits"]) << RINGS[ring]["log_n"])
    lo, hi = _RANGE[kind]
    hi = max(lo + 1, min(int(hi * min(size, 4.0)), 65536))
    px = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    case = dict(kind=kind, ring=ring)
    if kind == "batch":
        case["images"] = rng.randint(2, 70)
        side = max(2, int(math.sqrt(px / case["images"])))
        case["lo"], case["hi"] = max(1, side // 2), max(2, side + side // 4)
        case["cache"] = rng.choice(["radix16", "radix10", "full", "freq32"])
        return case
    case["c"] = rng.choice([1, 3])
    case["h"] = max(1, int(math.sqrt(px / case["c"]) * rng.uniform(0.6, 1.6)))
    case["w"] = max(1, int(px / case["c"] / case["h"]))
    if kind == "encrypt":
        case["cache"] = "fresh"
    if kind == "cached":
        case["kind"], case["cache"] = "encrypt", rng.choice(_CACHES)
    if kind == "decrypt":
        # the toy ring's first prime alone does not hold a pixel at its scale
        case["limbs"] = rng.randint(2 if ring == "n1024" else 1, len(RINGS[ring]["prime_bits"]))
    return case


# ------------------------------------------------------------------------------ preparation
def _image(h, w, c, seed):
    return np.ascontiguousarray(inputs.random_field_image(h, w, seed=seed, channels=c)).reshape(-1)


def _cache(ctx, name, seed, scan=None):
    if name == "fresh":
        return None
    if name.startswith("radix"):
        return ctx.build_cache(ichee.CACHE_RADIX, seed, radix_base={"radix16": 16, "radix2": 2}.get(name, 10),
                               randomize=0 if name.endswith("plain") else 1)
    if name.startswith("freq32"):
        return ctx.build_cache(ichee.CACHE_FREQ, seed, radix_base=10, top_k=32, pool_size=64,
                               miss_policy=1 if name.endswith("radix") else 0, scan=scan)
    return ctx.build_cache(ichee.CACHE_FULL, seed, pool_size=64)


def _sides(case):
    """Sides of a ragged batch's images: the same for every seed, which changes their contents."""
    rng = np.random.default_rng([case["images"], case["lo"], case["hi"], 7])
    return [int(x) for x in rng.integers(case["lo"], case["hi"] + 1, size=case["images"])]


def prepare(case, seed):
    kind = case["kind"]
    ctx = ichee.Context(**RINGS[case["ring"]])
    s = dict(case=case, ctx=ctx, seed=seed * 1000 + 17)
    if kind == "decrypt":
        return _prepare_decrypt(case, seed, s)
    ctx.keygen(seed + 11, with_evk=kind in ("match", "sqdiff"))
    top = ctx.L - 1
    if kind == "batch":
        sides = _sides(case)
        s["shapes"] = [(d, d, 1) for d in sides]
        img = [inputs.random_field_image(d, d, seed=seed * 100 + i).reshape(-1) for i, d in enumerate(sides)]
        counts = [d * d for d in sides]
        s["px_flat"] = torch.from_numpy(np.concatenate(img)).cuda()
        s["cache"] = _cache(ctx, case["cache"], seed + 23, scan=s["px_flat"])
        s["seeds"] = [seed + 500 + i for i in range(len(sides))]
        s["enc"], s["flt"] = ctx.empty_cts(sum(counts), top), ctx.empty_cts(sum(counts), top - 1)
        s["dec"] = torch.empty(sum(counts), dtype=torch.float64, device="cuda")
        s["px"] = list(torch.split(s["px_flat"], counts))
        s["enc_l"] = list(torch.split(s["enc"], [n * ctx.ct_words(top) for n in counts]))
        s["flt_l"] = list(torch.split(s["flt"], [n * ctx.ct_words(top - 1) for n in counts]))
        s["dec_l"] = list(torch.split(s["dec"], counts))
        torch.cuda.synchronize()
        return s
    h, w, c = case["h"], case["w"], case["c"]
    n = h * w * c
    px = _image(h, w, c, seed)
    if kind == "roundtrip":   # host buffers on both sides
        s["px"], s["out"] = px, ctx.empty_cts(n, top)
        s["dec"] = np.zeros(n, dtype=np.float64)
        return s
    s["px"] = torch.from_numpy(px).cuda()
    if kind == "encrypt":
        s["cache"], s["out"] = _cache(ctx, case["cache"], seed + 23, scan=s["px"]), ctx.empty_cts(n, top)
    elif kind == "chain":
        s["ct"], s["out"] = ctx.empty_cts(n, top), ctx.empty_cts(n, top - 1)
        s["dec"] = torch.empty(n, dtype=torch.float64, device="cuda")
    else:   # operations on ciphertexts: the inputs are encryptions with a radix-16 cache
        radix = _cache(ctx, "radix16", seed + 23)
        s["a"], s["ma"] = ctx.encrypt(s["px"], h, w, c, seed + 1, cache=radix)
        if kind == "blend":
            w8 = inputs.binary_pattern(h, w, seed + 5).reshape(-1)
            s["b"], s["mb"] = ctx.encrypt(torch.from_numpy(w8).cuda(), h, w, 1, seed + 2, cache=radix)
        elif kind in ("match", "sqdiff"):
            noisy = torch.from_numpy(inputs.noisy_copy(px, seed + 6)).cuda()
            s["b"], s["mb"] = ctx.encrypt(noisy, h, w, c, seed + 2, cache=radix)
        drop = kind != "brightness"
        s["out"] = ctx.empty_cts(1 if kind == "match" else n, top - 1 if drop else top)
        s["beta"] = inputs.brightness_beta(seed + 4)
    torch.cuda.synchronize()
    return s


def _decrypt_values(case, seed):
    """Pixels and small errors of the synthetic ciphertexts of a decryption case."""
    n = case["h"] * case["w"] * case["c"]
    px = _image(case["h"], case["w"], case["c"], seed).astype(np.int64)
    err = np.random.default_rng([seed, 3]).integers(-4096, 4097, size=n)
    return px, err


def _prepare_decrypt(case, seed, s):
    """Ciphertexts as an encryption leaves them, made without the library's encryption: c1 uniform,
    coefficient 0 of c0 = Delta p + e - (c1 s)_0, the other coefficients of c0 uniform."""
    ctx, limbs = s["ctx"], case["limbs"]
    n, dev = ctx.n, "cuda"
    px, err = _decrypt_values(case, seed)
    sk = np.random.default_rng([seed, 1]).integers(-1, 2, size=n).astype(np.int8)
    ichee.ichee_import_key(ctx.handle, 0, sk)
    rev = torch.from_numpy(np.concatenate([sk[:1], -sk[:0:-1]]).astype(np.int64)).to(dev)
    x = torch.from_numpy((px << RINGS[case["ring"]]["log2_scale"]) + err).to(dev)
    g = torch.Generator(device=dev).manual_seed(seed)
    ct = torch.empty(len(px), 2, limbs, n, dtype=torch.int64, device=dev)
    for l in range(limbs):
        q = ctx.q[l]
        for b in range(2):
            ct[:, b, l].random_(0, q, generator=g)
        v = torch.empty(len(px), dtype=torch.int64, device=dev)
        for i in range(0, len(px), 1024):   # (c1 s)_0 mod q in two 30-bit halves
            part = ct[i:i + 1024, 1, l]
            hi, lo = ((part >> 30) * rev).sum(1) % q, ((part & (2 ** 30 - 1)) * rev).sum(1) % q
            for _ in range(30):
                hi = hi * 2 % q
            v[i:i + 1024] = (hi + lo) % q
        ct[:, 0, l, 0] = (x - v) % q
    s["ct"] = ct
    s["meta"] = ichee.CtImgMeta(case["h"], case["w"], case["c"], limbs - 1, float(2 ** RINGS[case["ring"]]["log2_scale"]))
    s["dec"] = torch.empty(len(px), dtype=torch.float64, device=dev)
    torch.cuda.synchronize()
    return s


# ------------------------------------------------------------------------------------ a pass
def run(s):
    case, ctx = s["case"], s["ctx"]
    kind = case["kind"]
    if kind == "encrypt":
        return ctx.encrypt(s["px"], case["h"], case["w"], case["c"], s["seed"], cache=s["cache"], out=s["out"])[0]
    if kind == "roundtrip":
        ct, m = ctx.encrypt(s["px"], case["h"], case["w"], case["c"], s["seed"], out=s["out"])
        return [ct, ctx.decrypt(ct, m, out=s["dec"])]
    if kind == "chain":
        ct, m = ctx.encrypt(s["px"], case["h"], case["w"], case["c"], s["seed"], out=s["ct"])
        flt, mf = ctx.eval(ichee.OP_MEANFILTER3, ct, m, out=s["out"])
        return [ct, flt, ctx.decrypt(flt, mf, out=s["dec"])]
    if kind == "decrypt":
        return ctx.decrypt(s["ct"], s["meta"], out=s["dec"])
    if kind == "batch":
        st = ctx.stream()
        if case["cache"].startswith("radix"):
            _, mf = ichee.ichee_encrypt_meanfilter_batch(ctx.handle, s["cache"], s["px"], s["shapes"], s["seeds"],
                                                         s["enc_l"], s["flt_l"], st)
        else:
            mc = ichee.ichee_encrypt_batch(ctx.handle, s["cache"], s["px"], s["shapes"], s["seeds"], s["enc_l"], st)
            mf = ichee.ichee_eval_batch(ctx.handle, ichee.OP_MEANFILTER3, s["enc_l"], mc, outs=s["flt_l"], stream=st)
        ichee.ichee_decrypt_batch(ctx.handle, s["flt_l"], mf, s["dec_l"], st)
        return [s["enc"], s["flt"], s["dec"]]
    if kind == "meanfilter":
        return ctx.eval(ichee.OP_MEANFILTER3, s["a"], s["ma"], out=s["out"])[0]
    if kind == "brightness":
        return ctx.eval(ichee.OP_BRIGHTNESS, s["a"], s["ma"], args=(s["beta"],), out=s["out"])[0]
    if kind == "blend":
        return ctx.eval(ichee.OP_BLEND, s["a"], s["ma"], s["b"], s["mb"], args=(0.9,), out=s["out"])[0]
    op = ichee.OP_SQDIFF_SUM if kind == "match" else ichee.OP_SQDIFF
    return ctx.eval(op, s["a"], s["ma"], s["b"], s["mb"], out=s["out"])[0]


# ------------------------------------------------------------------------- work and tolerance
def work(case):
    """Bytes: every input ciphertext or pixel read once (decryption: c1 and one coefficient of
    c0), every output written once. flops: two per modular product (fresh encryption: three
    transforms of (N/2) log2 N products and two products by the key per limb; matching: two
    transforms and three products per limb and pair; the per-pixel form its L^2 + 5L + 2
    transforms; rescaled operations one product per kept limb and operand)."""
    r = RINGS[case["ring"]]
    n, ln, L = 1 << r["log_n"], r["log_n"], len(r["prime_bits"])
    kind, word = case["kind"], 8.0
    if kind == "batch":
        px = float(sum(d * d for d in _sides(case)))
    else:
        px = float(case["h"] * case["w"] * case["c"])
    ct, low = 2 * L * n * word, 2 * (L - 1) * n * word
    ntt = n / 2 * ln
    fresh = L * (3 * ntt + 2 * n)
    dec = px * ((L - 1) * n * word + 8 * L)
    if kind == "encrypt":
        misses = {"fresh": 1.0, "freq32": 0.7}.get(case["cache"], 0.0)
        return {"bytes": px * (1 + ct), "flops": 2 * px * misses * fresh}
    if kind == "roundtrip":
        return {"bytes": px * (1 + ct + L * n * word + 8), "flops": 2 * px * fresh}
    if kind == "chain":
        return {"bytes": px * (1 + 2 * ct + low) + dec, "flops": 2 * px * (fresh + 2 * (L - 1) * n)}
    if kind == "decrypt":
        return {"bytes": px * (case["limbs"] * (n + 1) * word + 8), "flops": px * case["limbs"] * n}
    if kind == "batch":
        return {"bytes": px * (1 + 2 * ct + low) + dec, "flops": 2 * px * 2 * (L - 1) * n}
    if kind == "meanfilter":
        return {"bytes": px * (ct + low), "flops": 2 * px * 2 * (L - 1) * n}
    if kind == "brightness":
        return {"bytes": 2 * px * ct, "flops": px * L}
    if kind == "blend":
        return {"bytes": px * (ct + low) + px / case["c"] * ct, "flops": 2 * px * 2 * 2 * (L - 1) * n}
    if kind == "match":
        return {"bytes": 2 * px * ct + low, "flops": 2 * px * L * (2 * ntt + 3 * n)}
    return {"bytes": px * (2 * ct + low), "flops": 2 * px * ((L * L + 5 * L + 2) * ntt + (2 * L * L + 12 * L) * n)}


def tolerance(case):
    """Ciphertext words are exact. Decoded values are an exact integer converted to float64 and
    divided once; a few roundings of 2^-53 apart at most."""
    if case["kind"] in ("roundtrip", "chain", "decrypt", "batch"):
        return {"rel": 1e-15, "max": 4e-15, "differ": 0.0}
    return "exact"


def exact(case, seed):
    """Decryption: the value the synthetic ciphertexts were built around. Elsewhere the outputs
    are ciphertext words (compared exactly) or values decoded from them."""
    if case["kind"] != "decrypt":
        return None
    px, err = _decrypt_values(case, seed)
    return px.astype(np.float64) + err.astype(np.float64) / float(2 ** RINGS[case["ring"]]["log2_scale"])

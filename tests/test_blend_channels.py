"""Blend of a several-channel image with a one-channel pattern (the form that takes a coefficient of all
channels in one thread, four limbs up), against the oracle: every limb count, one pixel to more
pixels than a share, two to five channels, and primes too small for the shared-constant form."""
import numpy as np
import pytest

from oracle import Oracle, Params

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits,log_n", [([50] + [40] * k, 10) for k in range(2, 8)] + [([30, 29, 28, 27], 10),
                                        ([60, 40, 40, 60, 50], 11)], ids=lambda v: str(v))
def test_blend_channels(bits, log_n):
    from paper_2409_03568_gb300 import ichee
    scale = 40 if min(bits) >= 40 else 26
    ctx = ichee.Context(log_n, bits, scale)
    ctx.keygen(12)
    o = Oracle(Params(log_n, bits, scale)).keygen(12)
    L = len(bits)
    rng = np.random.default_rng(L)
    for h, w, c, alpha in [(1, 1, 2, 0.9), (2, 3, 3, 0.9), (1, 5, 5, 0.25)]:
        pi = rng.integers(0, 256, size=h * w * c, dtype=np.uint8)
        pw = (rng.integers(0, 2, size=h * w) * 255).astype(np.uint8)
        a, ma = ctx.encrypt(torch.from_numpy(pi).cuda(), h, w, c, 21)
        b, mb = ctx.encrypt(torch.from_numpy(pw).cuda(), h, w, 1, 22)
        ref = o.blend(o.encrypt_pixels(pi, 21), o.encrypt_pixels(pw, 22), o.delta, alpha, c, 1)[0]
        out, _ = ctx.eval(ichee.OP_BLEND, a, ma, b, mb, args=(alpha,), out_level=L - 2)
        assert np.array_equal(out.cpu().numpy().view(np.uint64).reshape(ref.shape), ref), (h, w, c)
    ctx.close()

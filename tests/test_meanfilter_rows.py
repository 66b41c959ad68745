"""The mean filter's row groups: every limb count (each has its own group height), image heights that
leave remainders, one- and two-column images, and bands that start and end inside a group, against
the oracle."""
import numpy as np
import pytest

from oracle import Oracle, Params

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("limbs", range(2, 9))
def test_row_groups(limbs):
    from paper_2409_03568_gb300 import ichee
    bits = [50] + [40] * (limbs - 1)
    ctx = ichee.Context(10, bits, 40)
    ctx.keygen(8)
    o = Oracle(Params(10, bits, 40)).keygen(8)
    n = ctx.n
    rng = np.random.default_rng(limbs)
    for h, w, c in [(1, 1, 1), (2, 3, 1), (3, 2, 1), (4, 1, 3), (5, 4, 1), (9, 2, 1)]:
        px = rng.integers(0, 256, size=h * w * c, dtype=np.uint8)
        ct, m = ctx.encrypt(torch.from_numpy(px).cuda(), h, w, c, 40 + h)
        ref, _ = o.meanfilter3(o.encrypt_pixels(px, 40 + h), o.delta, h, w, c)
        out, _ = ctx.eval(ichee.OP_MEANFILTER3, ct, m, out_level=limbs - 2)
        assert np.array_equal(out.cpu().numpy().view(np.uint64).reshape(ref.shape), ref), (h, w, c)
        # bands: input rows only as far as the outputs need them, in a buffer that ends there
        words = ctx.ct_words(limbs - 1)
        for y0, y1 in [(0, 1), (h // 2, h), (1, max(2, h - 1))]:
            if not (0 <= y0 < y1 <= h):
                continue
            r0, r1 = max(0, y0 - 1), min(h, y1 + 1)
            rows = ct[r0 * w * c * words:r1 * w * c * words].clone()
            band = ctx.empty_cts((y1 - y0) * w * c, limbs - 2)
            ichee.ichee_meanfilter_rows(ctx.handle, rows, m, r0, r1 - r0, y0, y1, band, ctx.stream())
            got = band.cpu().numpy().view(np.uint64).reshape((y1 - y0) * w * c, 2, limbs - 1, n)
            assert np.array_equal(got, ref[y0 * w * c:y1 * w * c]), (h, w, c, y0, y1)
    ctx.close()

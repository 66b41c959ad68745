"""The mean filter's row groups: every limb count, every group height that the launch can choose (by the
blocks there are: the tall images have just as many as fit the GPU with 1, 2, 3 and 4 rows a group),
image heights that leave remainders, one- and two-column images, bands that start and end inside a
group, and ragged batches, against the oracle."""
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
    groups = torch.cuda.get_device_properties(0).multi_processor_count * 4 // 16   # of 2 polynomials x 8 chunks at N = 2^10
    tall = [(r * groups - 1, 1, 1) for r in (2, 3, 4)] + [(5 * groups, 2, 1)]
    tall = [s for s in tall if s[0] * limbs < 600]   # a few limbs: the others take fewer rows
    cts, metas, refs = [], [], []
    for h, w, c in [(1, 1, 1), (2, 3, 1), (3, 2, 1), (4, 1, 3), (5, 4, 1), (9, 2, 1)] + tall:
        px = rng.integers(0, 256, size=h * w * c, dtype=np.uint8)
        ct, m = ctx.encrypt(torch.from_numpy(px).cuda(), h, w, c, 40 + h)
        ref, _ = o.meanfilter3(o.encrypt_pixels(px, 40 + h), o.delta, h, w, c)
        out, _ = ctx.eval(ichee.OP_MEANFILTER3, ct, m, out_level=limbs - 2)
        assert np.array_equal(out.cpu().numpy().view(np.uint64).reshape(ref.shape), ref), (h, w, c)
        cts.append(ct), metas.append(m), refs.append(ref)
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
    # batches: the small images, then each tall one with the first, then all
    small = len(cts) - len(tall)
    for pick in [range(small)] + [[0, i] for i in range(small, len(cts))] + [range(len(cts))]:
        outs = [ctx.empty_cts(metas[i].n_ct, limbs - 2) for i in pick]
        ichee.ichee_eval_batch(ctx.handle, ichee.OP_MEANFILTER3, [cts[i] for i in pick], [metas[i] for i in pick],
                               outs=outs, stream=ctx.stream())
        for i, out in zip(pick, outs):
            assert np.array_equal(out.cpu().numpy().view(np.uint64).reshape(refs[i].shape), refs[i]), i
    ctx.close()

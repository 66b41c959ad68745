"""Decryption's block shapes: both sides of every line of the rule (ciphertexts per SM, by ring size), the
single-image and the batched kernel, against the plain pixels and one warp per ciphertext."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("log_n,bits,scale", [(10, [30, 30], 25), (11, [60, 40, 40], 40), (12, [45, 32, 32], 32),
                                              (13, [60, 40], 40), (14, [60, 40, 40, 40, 40], 40)],
                         ids=lambda v: str(v))
def test_decrypt_shapes(log_n, bits, scale):
    from paper_2409_03568_gb300 import ichee
    ctx = ichee.Context(log_n, bits, scale)
    ctx.keygen(5)
    warp = ichee.Context(log_n, bits, scale)   # one warp sums a whole ciphertext; the other context's shape is never set
    warp.keygen(5)
    ichee.ichee_set_tuned_shape(warp.handle, ichee.TUNE_DECRYPT, 32)
    cache = ctx.build_cache(ichee.CACHE_RADIX, seed=3, radix_base=16)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    lines = {10: [1, 3], 11: [1, 3], 12: [1, 6], 13: [1, 2], 14: [1, 4]}[log_n]
    for n in sorted({1, 63, 64} | {sms * k + d for k in lines for d in (0, 1)}):
        px = torch.randint(0, 256, (n,), dtype=torch.uint8, device="cuda")
        ct, m = ctx.encrypt(px, 1, n, 1, 9, cache=cache)
        one = ctx.decrypt(ct, m, out=torch.empty(n, dtype=torch.float64, device="cuda"))
        assert torch.equal(one.round().to(torch.uint8), px), n
        got = torch.empty(n, dtype=torch.float64, device="cuda")
        ichee.ichee_decrypt_batch(ctx.handle, [ct], [m], [got], ctx.stream())
        ref = torch.empty(n, dtype=torch.float64, device="cuda")
        ichee.ichee_decrypt_batch(warp.handle, [ct], [m], [ref], ctx.stream())
        assert torch.equal(one, ref), n                                     # the sums are exact: every shape the same bits
        assert torch.equal(got, ref), n
    warp.close()
    ctx.close()

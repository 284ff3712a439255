"""The mixed-radix upchannelizer's kernels give the same bits: whatever shape the
dispatch picks, every other (inputs per CTA; sums formed in the first pass or
before it) is forced by its tuning entry and compared, at lengths whose quads,
passes and rows come out uneven."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,n_input,taps,window", [
    (2400, 9, 4, None), (2400, 12, 1, (1190, 21)), (480, 3, 5, None), (6, 8, 2, None), (2, 1, 3, None),
    (1024, 5, 4, (0, 1)), (8192, 6, 2, None), (8192, 8, 1, (100, 1000)), (90, 33, 3, (7, 80)), (486, 2, 1, None),
    (4096, 4, 4, None)])
def test_every_shape_the_same_bits(lib, n, n_input, taps, window):
    g = torch.Generator(device="cuda")
    g.manual_seed(n + n_input)
    n_time = (taps + 2) * n + 1
    v = torch.randint(0, 256, (1, n_time, n_input), generator=g, device="cuda", dtype=torch.int16).to(torch.uint8)
    h = [torch.rand(taps * n, generator=g, device="cuda") - 0.3] if taps > 1 else None
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    key = f"k_upchan_mr/sm{sms}/{n}/{n_input}/{taps}/{window[1] if window else n}"

    def run():
        q, f = lib.upchan(v, [n], taps=h, window=window, want_f32=True)
        return q, f, lib.upchan(v, [n], taps=h, window=window)[0]

    lib.tune_clear()
    try:
        q, f, q1 = run()
        assert torch.equal(q, q1)
        tried = 0
        for c in range(4, 36):                 # inputs * 4 + kernel
            if c // 4 not in (1, 2, 4, 8):
                continue
            lib.tune_set(key, c)
            try:
                other = run()
            except lib.OvroError:              # a shape that does not fit
                continue
            tried += 1
            assert torch.equal(q, other[0]) and torch.equal(f, other[1]) and torch.equal(q, other[2])
        assert tried >= 2
    finally:
        lib.tune_clear()

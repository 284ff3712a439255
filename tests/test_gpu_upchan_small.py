"""A few spectra of a few inputs: the upchannelizer spreads them over the SMs, so the
transform is faster than with the most inputs a CTA can hold, and returns the same
bits with any number of them."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _kernel_ms(lib, fn):
    """Device time of the transform, the least of some calls."""
    best = float("inf")
    for _ in range(8):
        torch.cuda.synchronize()
        lib.profile(True)
        fn()
        torch.cuda.synchronize()
        best = min(best, lib.profile_query("k_upchan")[0])
        lib.profile(False)
    return best


@pytest.mark.parametrize("log2n,n_input,wide", [(13, 16, 8), (13, 18, 8), (13, 24, 8), (13, 40, 8), (12, 18, 16), (12, 40, 16)])
@pytest.mark.parametrize("f32", [False, True])
def test_few_spectra_fill_the_chip(lib, log2n, n_input, wide, f32):
    n = 1 << log2n
    g = torch.Generator(device="cuda")
    g.manual_seed(n_input)
    v = torch.randint(0, 256, (1, 9 * n, n_input), generator=g, device="cuda", dtype=torch.int16).to(torch.uint8)
    key = "k_upchan/sm%d/%d/%d" % (torch.cuda.get_device_properties(0).multi_processor_count, log2n, n_input)
    lib.tune_clear()
    q, f = lib.upchan(v, [n], want_f32=f32)
    t = _kernel_ms(lib, lambda: lib.upchan(v, [n], want_f32=f32))
    try:
        lib.tune_set(key, wide)
        qw, fw = lib.upchan(v, [n], want_f32=f32)
        tw = _kernel_ms(lib, lambda: lib.upchan(v, [n], want_f32=f32))
    finally:
        lib.tune_clear()
    assert torch.equal(q, qw) and (not f32 or torch.equal(f, fw))
    assert t <= 0.8 * tw, (t, tw)

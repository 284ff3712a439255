"""The upchannelizer on rows that do not start on a word: an odd number of
inputs with whole groups of them, and a voltage buffer that starts off 16 bytes.
Every input is transformed on its own, so the values are those of the same
inputs inside wider, aligned rows, bit for bit."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nfft,n_input,shift", [([2048], 23, 0), ([8192], 5, 0), ([1024, 256], 33, 0), ([4096], 17, 3),
                                                ([8192], 16, 1), ([1024], 48, 4), ([480], 9, 0), ([2400], 12, 2),
                                                ([16, 64], 31, 1), ([8192], 34, 0), ([1024], 574, 0),
                                                ([256], 4099, 0)])
def test_rows_off_a_word(lib, nfft, n_input, shift):
    g = torch.Generator(device="cuda")
    g.manual_seed(n_input)
    n_time, wide = 3 * max(nfft) + 7, (n_input + 63) // 32 * 32
    v = torch.randint(0, 256, (len(nfft), n_time, wide), generator=g, device="cuda", dtype=torch.int16).to(torch.uint8)
    flat = torch.zeros(len(nfft) * n_time * n_input + shift, dtype=torch.uint8, device="cuda")
    narrow = flat[shift:].view(len(nfft), n_time, n_input)
    narrow.copy_(v[:, :, :n_input])
    qw, fw = lib.upchan(v, nfft, want_f32=True)
    qn, fn = lib.upchan(narrow, nfft, want_f32=True)
    off_w = off_n = 0
    for n in nfft:
        k = n_time // n
        for a, b in ((qw, qn), (fw, fn)):
            w = a[off_w:off_w + n * k * wide * 2].view(n, k, wide, 2)[:, :, :n_input]
            assert torch.equal(w, b[off_n:off_n + n * k * n_input * 2].view(n, k, n_input, 2))
        off_w += n * k * wide * 2
        off_n += n * k * n_input * 2


@pytest.mark.parametrize("n_input", [3, 20])
@pytest.mark.parametrize("log2n", range(4, 15))
def test_every_power_of_two_both_ways(lib, log2n, n_input):
    """The int8 spectra are the same whether FP32 ones are asked for or not (the
    last passes differ), and the FP32 ones those of an FP64 transform.  Four passes,
    each at most 4 additions and 6 roundings of twiddles and their products deep:
    ||error|| <= 4 * 10 * 2^-24 ||X||."""
    n = 1 << log2n
    g = torch.Generator(device="cuda")
    g.manual_seed(log2n)
    v = torch.randint(0, 256, (1, 2 * n + 1, n_input), generator=g, device="cuda", dtype=torch.int16).to(torch.uint8)
    q, f = lib.upchan(v, [n], want_f32=True)
    q1, _ = lib.upchan(v, [n])
    assert torch.equal(q, q1)
    b = v[0, :2 * n].to(torch.int64).view(2, n, n_input)
    x = torch.complex(((b >> 4) ^ 8).double() - 8, ((b & 15) ^ 8).double() - 8)
    want = torch.fft.fftshift(torch.fft.fft(x, dim=1), dim=1).permute(1, 0, 2)
    got = torch.view_as_complex(f.double().view(n, 2, n_input, 2).contiguous())
    assert float((got - want).norm()) <= 40 * 2.0 ** -24 * float(want.norm())

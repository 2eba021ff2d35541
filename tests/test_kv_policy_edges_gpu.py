"""Edges of the KV4 quantizer's and the policy's packed arithmetic: NaN and infinities (no
value disturbs its neighbours in a word), ties, ragged group counts, tiny and infinite
scales."""
import numpy as np
import pytest

import parity

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_12487_gb300 import dptq
    dptq.load()
    return dptq


@pytest.mark.parametrize("rows,cols", [(1, 128), (3, 128), (5, 640), (257, 1024)])
def test_kv4_ties_and_non_finite_values(dp, orc, rows, cols):
    rng = np.random.default_rng(rows + cols)
    x = (rng.integers(-14, 15, (rows, cols)) * 0.5).astype(np.float16)   # half the values tie
    x[:, ::128] = 7.0                                                    # s = 1
    x[0, :128] = 0
    x[-1, 64:128] *= np.float16(2.0 ** -20)
    c_ref, s_ref = orc.kv4_quantize(x, 128)
    bad = x.copy()
    bad[-1, 5], bad[-1, 77] = np.nan, -np.nan
    for src in (x, bad):
        codes = torch.empty((rows, cols // 2), dtype=torch.uint8, device="cuda")
        sc = torch.empty((rows, cols // 128), dtype=torch.float32, device="cuda")
        dp.dptq_kv4_quantize(torch.from_numpy(src).cuda(), 128, codes, sc)
        c = parity.unpack_public_a4(codes.cpu().numpy(), cols)
        want = np.where(np.isnan(src), -1, c_ref)
        assert np.array_equal(c, want) and np.array_equal(sc.cpu().numpy(), s_ref)
    # an infinite value: infinite scale, code -1 for it and 0 for the other values of its group
    inf = x.copy()
    inf[-1, 9] = np.inf
    dp.dptq_kv4_quantize(torch.from_numpy(inf).cuda(), 128, codes, sc)
    c = parity.unpack_public_a4(codes.cpu().numpy(), cols)
    assert np.isinf(sc.cpu().numpy()[-1, 0]) and c[-1, 9] == -1 and np.all(np.delete(c[-1, :128], 9) == 0)
    assert np.array_equal(c[-1, 128:], c_ref[-1, 128:]) and np.array_equal(c[:-1], c_ref[:-1])


@pytest.mark.parametrize("offset", [2, 4, 6, 8])
@pytest.mark.parametrize("cols,group", [(640, 128), (512, 256)])
def test_kv4_codes_at_any_even_address(dp, offset, cols, group):
    rows = 9
    x = np.random.default_rng(offset).standard_normal((rows, cols)).astype(np.float16)
    x[2, 3] = np.nan
    want = torch.empty((rows, cols // 2), dtype=torch.uint8, device="cuda")
    buf = torch.full((rows * cols // 2 + 16,), 0xA5, dtype=torch.uint8, device="cuda")
    codes = buf[offset:offset + want.numel()].view(rows, cols // 2)
    sc = torch.empty((rows, cols // group), dtype=torch.float32, device="cuda")
    kv = torch.from_numpy(x).cuda()
    dp.dptq_kv4_quantize(kv, group, want, sc)
    dp.dptq_kv4_quantize(kv, group, codes, sc)
    assert torch.equal(codes, want) and torch.all(buf[:offset] == 0xA5) and torch.all(buf[offset + want.numel():] == 0xA5)


def test_kv4_codes_at_an_odd_address_are_refused(dp):
    buf = torch.empty((128,), dtype=torch.uint8, device="cuda")
    kv, sc = torch.zeros((1, 128), dtype=torch.float16, device="cuda"), torch.empty((1, 1), device="cuda")
    with pytest.raises(dp.DptqError):
        dp.dptq_kv4_quantize(kv, 128, buf[1:65].view(1, 64), sc)


@pytest.mark.parametrize("d", [4, 1028, 4096])
@pytest.mark.parametrize("bits", [4, 8])
def test_policy_ties_tiny_and_infinite_values(dp, orc, d, bits):
    L, T = 4, 9
    rng = np.random.default_rng(d + bits)
    x = (rng.integers(-14, 15, (L, T, d)) * 0.5).astype(np.float32)
    dx = (rng.integers(-3, 4, (L, T, d)) * 0.25).astype(np.float32)
    x[1] *= np.float32(1e-39)                       # subnormal sums: the reciprocal overflows
    dx[1] *= np.float32(1e-39)
    x[2] += rng.standard_normal((T, d)).astype(np.float32)
    ref = [orc.residual_stats(x[l], dx[l], bits, 1e-6) for l in range(L)]
    jr = torch.empty((L,), dtype=torch.float64, device="cuda")
    snr = torch.empty((L,), dtype=torch.float64, device="cuda")
    mask = torch.empty((L,), dtype=torch.uint8, device="cuda")
    dp.dptq_sensitivity_policy(torch.from_numpy(x).cuda(), torch.from_numpy(dx).cuda(), bits, 1e-6, 0.1, 20.0, jr, snr,
                               mask)
    for l in (0, 2, 3):
        assert abs(jr[l].item() - ref[l][0]) <= 1e-5 * abs(ref[l][0]) and abs(snr[l].item() - ref[l][1]) <= 1e-3
    # an infinite update: the scale is infinite, inf * 0 of the finite values' codes is NaN, and so
    # is its layer's SNR (IEEE, term by term); the other layers keep theirs
    dx[3, 2, 1] = np.inf
    before = snr.clone()
    dp.dptq_sensitivity_policy(torch.from_numpy(x).cuda(), torch.from_numpy(dx).cuda(), bits, 1e-6, 0.1, 20.0, jr, snr,
                               mask)
    assert np.isinf(jr[3].item()) and np.isnan(snr[3].item())
    assert np.allclose(snr[:3].cpu().numpy(), before[:3].cpu().numpy(), rtol=1e-12, equal_nan=True)
    dp.dptq_last_device_error()


# tokens of more than 4096 values: batches of 32 tokens that span layers, ragged last batches and
# widths, one token
@pytest.mark.parametrize("L,T,d", [(1, 1, 4100), (7, 5, 5120), (3, 700, 5120), (40, 33, 8192), (5, 9, 12292)])
def test_policy_of_wide_tokens(dp, L, T, d):
    g = torch.Generator(device="cuda").manual_seed(d + T)
    x = torch.randn((L, T, d), generator=g, device="cuda")
    dx = torch.randn((L, T, d), generator=g, device="cuda") * 0.3
    jr, snr = torch.empty(L, dtype=torch.float64, device="cuda"), torch.empty(L, dtype=torch.float64, device="cuda")
    bits = torch.empty(L, dtype=torch.uint8, device="cuda")
    dp.dptq_sensitivity_policy(x, dx, 4, 1e-6, 0.1, 20.0, jr, snr, bits)
    dp.dptq_last_device_error()
    xs, ds = x.double(), dx.double()
    u = x + dx
    s = u.abs().amax(-1, keepdim=True) / 7
    err = (s.double() * torch.clamp(torch.round(u / s), -8, 7).double() - ds - xs).pow(2).sum(-1)
    nx = xs.pow(2).sum(-1)
    # A thread sums up to d / 256 + 4 squares in fp32 (each step and the error's own roundings
    # within 2^-24), the rest is fp64: relative 2 (d / 256 + 8) 2^-24, twice over in a ratio.
    rel = 4 * (d / 256 + 8) * 2.0 ** -24
    torch.testing.assert_close(jr, (ds.pow(2).sum(-1).sqrt() / (nx.sqrt() + 1e-6)).mean(1), rtol=rel, atol=0)
    torch.testing.assert_close(snr, (10 * torch.log10(nx / (err + 1e-6))).mean(1), rtol=0, atol=10 * rel)

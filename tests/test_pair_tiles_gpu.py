"""192-token tiles multiplied by pairs of CTAs: accumulators equal the integer product."""
import pytest

from paper_2606_12487_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# whole waves and split tiles, one tile of tokens and many, a ragged last weight tile and token
# tile, an odd number of weight tiles (no pairs), K padded from 1152 to 1280
@pytest.mark.parametrize("M,N,K,pair", [(192, 38912, 4096, 2), (1000, 38912, 512, 2), (577, 12176, 4096, 2),
                                        (577, 12272, 2048, 2), (2048, 4096, 14336, 2), (1025, 12176, 1152, 2),
                                        (2048, 11904, 1024, 1)])
@pytest.mark.parametrize("bits", [4, 8])
def test_accumulators_of_pairs(M, N, K, pair, bits):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_12487_gb300 import dptq
    dptq.load()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if bits == 4:
        assert dptq.dptq_launch_plan(M, N, K, bits, sms, 0)["pair"] == pair
    g = torch.Generator(device="cuda").manual_seed(M + N)
    layer = dptq.dptq_pack_weights((torch.randn((N, K), generator=g, device="cuda") * 0.02).half(), 128)
    wq, sw = (torch.from_numpy(t).cuda() for t in dptq.dptq_get_packed(layer))
    w = torch.stack([((wq & 15) ^ 8).to(torch.int8) - 8, ((wq >> 4) ^ 8).to(torch.int8) - 8], -1).reshape(N, K)
    c = torch.from_numpy(inputs.random_codes(M, K, bits, seed=M + N)).cuda()
    packed = (c[:, 0::2] & 15).to(torch.uint8) | ((c[:, 1::2] & 15) << 4).to(torch.uint8) if bits == 4 else c
    ref = c.double() @ w.double().t()   # whole numbers below 2^53: exact
    sa = torch.rand(M, generator=g, device="cuda") * 0.1 + 0.01
    want = ((ref.float() * sa[:, None]) * sw[None, :]).half()
    for _ in range(2):   # split-tile sums are left clean
        out = torch.empty((M, N), dtype=torch.float16, device="cuda")
        acc = torch.empty((M, N), dtype=torch.int32, device="cuda")
        dptq.dptq_qgemm_codes(layer, packed.contiguous(), sa, bits, out, acc)
        assert torch.equal(acc.double(), ref)
        assert torch.equal(out.view(torch.int16), want.view(torch.int16))
    dptq.dptq_last_device_error()
    layer.close()

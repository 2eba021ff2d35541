"""GEMMs of more than 64 tokens on both kinds of token tiles, whole and split, ragged in both
dimensions: accumulators equal the integer product, outputs its scaled rounding."""
import numpy as np
import pytest

from test_launch_plan_cpu import units

from paper_2606_12487_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_12487_gb300 import dptq
    dptq.load()
    return dptq


# 64-token tiles whole, split, and with one k-block more than a stage; 192-token tiles whole in
# waves and split; K padded from 384 to 512
@pytest.mark.parametrize("M,N,K", [(65, 48, 512), (100, 1024, 4096), (129, 272, 768), (200, 4096, 1024),
                                   (333, 12288, 512), (449, 2064, 2048), (1000, 4096, 2048), (2048, 4096, 512),
                                   (700, 1024, 384)])
@pytest.mark.parametrize("bits", [4, 8])
def test_accumulators_on_every_plan(dp, M, N, K, bits):
    check_accumulators(dp, M, N, K, bits, 2)


# a split tile, a whole one and a split one in one CTA's share (single CTAs and pairs): the
# epilogue warps meet only in the split ones
@pytest.mark.parametrize("M,N,K,bits", [(193, 11904, 11008, 4), (129, 22016, 4096, 8), (200, 20480, 8192, 4),
                                        (333, 12176, 8192, 8)])
def test_split_tiles_with_whole_ones_between(dp, M, N, K, bits):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    p = dp.dptq_launch_plan(M, N, K, bits, sms)
    share = {}
    for c, _, _, _, slot, _ in units(p):
        share.setdefault(c, []).append(slot >= 0)
    if sms == 152:
        assert p["nt"] > 64 and any(s[i:i + 3] == [True, False, True] for s in share.values() for i in range(len(s)))
    check_accumulators(dp, M, N, K, bits, 20)


def check_accumulators(dp, M, N, K, bits, passes):
    layer = dp.dptq_pack_weights(torch.from_numpy(inputs.weights(N, K, layer=5)).cuda(), 128)
    wq, sw = dp.dptq_get_packed(layer)
    w = np.empty((N, K), dtype=np.int8)
    w[:, 0::2] = ((wq & 15) ^ 8).astype(np.int8) - 8
    w[:, 1::2] = ((wq >> 4) ^ 8).astype(np.int8) - 8
    codes = inputs.random_codes(M, K, bits, seed=M + N)
    sa = (np.random.default_rng(M).random(M) * 0.1 + 0.01).astype(np.float32)
    c = torch.from_numpy(codes).cuda()
    if bits == 4:
        packed = (c[:, 0::2] & 15).to(torch.uint8) | ((c[:, 1::2] & 15) << 4).to(torch.uint8)
    else:
        packed = c
    ref = (c.double() @ torch.from_numpy(w).cuda().double().t())   # whole numbers below 2^53: exact
    sad, swd = torch.from_numpy(sa).cuda(), torch.from_numpy(sw).cuda()
    want = ((ref.float() * sad[:, None]) * swd[None, :]).half()
    for _ in range(passes):   # split-tile sums are left clean
        out = torch.empty((M, N), dtype=torch.float16, device="cuda")
        acc = torch.empty((M, N), dtype=torch.int32, device="cuda")
        dp.dptq_qgemm_codes(layer, packed.contiguous(), sad, bits, out, acc)
        assert torch.equal(acc.double(), ref)
        assert torch.equal(out.view(torch.int16), want.view(torch.int16))
    dp.dptq_last_device_error()
    layer.close()

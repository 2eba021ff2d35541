"""The tensor-core rotation at the edges of its forms: units of 1024 elements, blocks over
1, 2 and 4 warps, tails in units of their own, rows over a cluster of CTAs, and rows whose
values leave the plain fp32-pair form."""
import numpy as np
import pytest

import parity
from paper_2606_12487_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def dp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_12487_gb300 import dptq
    dptq.load()
    return dptq


# one short unit; exactly one unit; a tail after it; a unit that holds whole blocks and
# part of the next; two- and four-warp blocks with and without tails; 17, 20 and 28 units
# (two CTAs a row), 33 with a tail, 40 and 48 (three: their first maxima meet right after the launch)
FORMS = [(32, 32), (160, 32), (1024, 1024), (1056, 1024), (2080, 64), (3072, 2048), (4096, 4096), (6144, 4096),
         (5888, 512), (17408, 1024), (20480, 2048), (28672, 4096), (33280, 1024), (40960, 4096), (49152, 256)]


def rows_of_every_kind(K):
    rng = np.random.default_rng(K)
    n = rng.standard_normal((7, K)).astype(np.float32)
    n[1] *= 1e-4                                   # near binary16's smallest values
    n[2] = 40.0 * rng.integers(-100, 101, K)       # large sums on a coarse grid: pairs with k > 0
    n[3, :3] = 60000.0                             # large sums and fine values: pairs with a list
    n[4] = 65504.0                                 # the largest sum: 64-bit integers
    n[5] = 0.0
    n[6, K // 2:] = 0.0                            # zero units
    return inputs.to_f16(n)


@pytest.mark.parametrize("K,B", FORMS)
def test_forms_match_the_oracle(dp, orc, K, B):
    x = rows_of_every_kind(K)
    M = x.shape[0]
    signs = np.where(np.random.default_rng(5).random(K) < 0.5, -1, 1).astype(np.int8)
    xd, sd = torch.from_numpy(x).to(DEV), torch.from_numpy(signs).to(DEV)
    exact = (B.bit_length() - 1) % 2 == 0 and K % B == 0   # even log2: no irrational factor
    for sg in (None, signs):
        y_ref = orc.rotate(x, B, sg)
        y = torch.empty((M, K), dtype=torch.float32, device=DEV)
        if sg is None:
            dp.dptq_rotate_act(xd, B, y)
        else:
            dp.dptq_rotate_act_rh(xd, B, sd, y)
        parity.check_rotation(y.cpu().numpy(), y_ref)
        if exact:
            assert np.array_equal(y.cpu().numpy(), y_ref)
        for bits in (4, 8):
            c_ref, s_ref = orc.rotate_quant_act(x, B, bits, sg)
            codes = torch.empty((M, K // 2) if bits == 4 else (M, K),
                                dtype=torch.uint8 if bits == 4 else torch.int8, device=DEV)
            sc = torch.empty((M,), dtype=torch.float32, device=DEV)
            if sg is None:
                dp.dptq_rotate_quant_act(xd, B, bits, codes, sc)
            else:
                dp.dptq_rotate_quant_act_rh(xd, B, bits, sd, codes, sc)
            c = codes.cpu().numpy()
            c = orc.unpack_nibbles(c, K) if bits == 4 else c
            parity.check_scales(sc.cpu().numpy(), s_ref)
            n = parity.check_codes(c, c_ref, y_ref, s_ref, bits)
            if exact:
                assert n == 0 and np.array_equal(sc.cpu().numpy(), s_ref)
    dp.dptq_last_device_error()


@pytest.mark.parametrize("K,B", [(160, 32), (1056, 1024), (4096, 4096), (14336, 2048), (17408, 1024)])
@pytest.mark.parametrize("bits", [4, 8])
def test_operand_planes_hold_the_public_codes(dp, K, B, bits):
    """The rotate-quantize launch of a layer (more rows than CTAs, padded token tiles) feeds
    the GEMM the codes and scales that the public call returns."""
    base = rows_of_every_kind(K)
    M = 700
    x = torch.from_numpy(base).to(DEV).repeat(M // 7, 1)
    x[7:] *= torch.linspace(0.1, 1.0, M - 7, device=DEV)[:, None].half()
    layer = dp.dptq_pack_weights(torch.from_numpy(inputs.weights(64, K)).to(DEV), B)
    got = torch.empty((M, 64), dtype=torch.float16, device=DEV)
    dp.dptq_qlinear(layer, x, bits, got)
    codes = torch.empty((M, K // 2) if bits == 4 else (M, K), dtype=torch.uint8 if bits == 4 else torch.int8, device=DEV)
    sc = torch.empty((M,), dtype=torch.float32, device=DEV)
    dp.dptq_rotate_quant_act(x, B, bits, codes, sc)
    ref = torch.empty((M, 64), dtype=torch.float16, device=DEV)
    dp.dptq_qgemm_codes(layer, codes, sc, bits, ref)
    assert torch.equal(got.view(torch.int16), ref.view(torch.int16))
    dp.dptq_last_device_error()
    layer.close()


# one row a CTA, two CTAs a row, several rows side by side in a CTA (1, 2 and 4 warps each, a
# last CTA that is not full), whole tiles and clusters of two and four CTAs
# (`rows` a CTA: 0 for half a row)
@pytest.mark.parametrize("M,N,K,B,rows", [(16, 512, 256, 256, 8), (13, 128, 1024, 1024, 8), (64, 512, 2048, 2048, 4),
                                          (33, 640, 4096, 4096, 2), (64, 1024, 4096, 2048, 2), (7, 4096, 11008, 256, 0),
                                          (32, 6144, 4096, 4096, 1), (21, 8192, 1536, 512, 1), (31, 512, 3072, 1024, 2)])
@pytest.mark.parametrize("bits", [4, 8])
def test_one_launch_equals_two(dp, M, N, K, B, rows, bits):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    items, _ = parity.one_launch_row_ctas(dp, M, N, K, B, bits, sms)
    assert items == (-(-M // rows) if rows else 2 * M)
    base = rows_of_every_kind(K)
    x = torch.from_numpy(np.concatenate([base] * (-(-M // 7)))[:M]).to(DEV)
    x[7:] *= torch.linspace(0.2, 1.0, max(1, M - 7), device=DEV)[:max(0, M - 7), None].half()
    layer = dp.dptq_pack_weights(torch.from_numpy(inputs.weights(N, K, layer=3)).to(DEV), B)
    one = torch.empty((M, N), dtype=torch.float16, device=DEV)
    two = torch.empty((M, N), dtype=torch.float16, device=DEV)
    for _ in range(2):
        dp.dptq_qlinear(layer, x, bits, one)
    dp.dptq_qlinear_quantize(layer, x, bits)
    dp.dptq_qlinear_gemm(layer, M, bits, two)
    assert torch.equal(one.view(torch.int16), two.view(torch.int16))
    dp.dptq_last_device_error()
    layer.close()

"""The plan a two-launch call takes: the operand planes do not depend on N (one quantized
matrix serves several layers), and every (tile, stage) is processed exactly once, with the
contributors and slots of split tiles consistent (the device's enumeration restated)."""
import itertools

import pytest

from paper_2606_12487_gb300 import dptq

NS = [16, 512, 1024, 4096, 5120, 12288, 28672]
KS = [256, 384, 4096, 11008, 28672]
MS = [1, 16, 33, 64, 65, 100, 128, 129, 200, 333, 512, 1000, 2048, 8192]


def units(p):
    """(tile, i0, i1, slot, contributors) of every CTA (a pair of CTAs: once, for its pair of
    tiles), as the kernel walks them."""
    G, KI, dp, sk, skG = p["grid"] // p["pair"], p["KI"], p["dp_tiles"], p["sk_iters"], p["sk_ctas"]
    begin = lambda c: c * sk // skG
    cta_of = lambda i: ((i + 1) * skG - 1) // sk
    for c in range(G):
        for t in range(c, dp, G):
            yield c, t, 0, KI, -1, 1
        if not sk or c >= skG:
            continue
        it, end = begin(c), begin(c + 1)
        while it < end:
            t, i0 = divmod(it, KI)
            i1 = min(KI, i0 + end - it)
            c0, c1 = cta_of(t * KI), cta_of(t * KI + KI - 1)
            yield c, dp + t, i0, i1, (-1 if c0 == c1 else c0), c1 - c0 + 1
            it += i1 - i0


@pytest.mark.parametrize("M,bits,sms", list(itertools.product(MS, (4, 8), (148, 152))))
def test_planes_do_not_depend_on_n(M, bits, sms):
    for K in KS:
        assert len({dptq.dptq_launch_plan(M, N, K, bits, sms)["M_pad"] for N in NS}) == 1
        wide = dptq.dptq_plan_info(M, 4096, K, bits, sms)
        assert dptq.dptq_launch_plan(M, 4096, K, bits, sms)["M_pad"] == wide["M_pad"]


@pytest.mark.parametrize("N,K", [(16, 256), (1024, 4096), (4096, 4096), (4096, 11008), (5120, 384), (5120, 5120), (6144, 4096),
                                 (8192, 8192), (12288, 4096), (28672, 4096)])
@pytest.mark.parametrize("bits", [4, 8])
@pytest.mark.parametrize("fused", [False, True])
def test_every_stage_once(N, K, bits, fused):
    for M in MS:
        rows = M * (2 if K > 8192 else 1) if fused else 0
        if fused:
            try:
                dptq.dptq_launch_plan(M, N, K, bits, 152, rows)
            except dptq.DptqError:   # refused only where no general one-launch plan exists either
                with pytest.raises(dptq.DptqError):
                    dptq.dptq_plan_info(M, N, K, bits, 152, fused=True)
                continue
        p = dptq.dptq_launch_plan(M, N, K, bits, 152, rows)
        assert p["fused"] == int(fused) and p["grid"] >= rows   # a CTA for every row's rotation
        tiles = p["n_wtiles"] * p["m_tiles"] // p["pair"]
        assert p["grid"] % p["pair"] == 0 and p["n_wtiles"] % p["pair"] == 0 and (p["pair"] == 1 or p["nt"] == 192)
        assert p["m_tiles"] * p["nt"] >= M and p["m_tiles"] * p["nt"] <= p["M_pad"]
        assert p["smem_bytes"] <= 232448 and p["grid"] <= 152 and p["kps"] * p["KI"] == -(-K // 256) * 2
        parts = {}
        for c, t, i0, i1, slot, n in units(p):
            parts.setdefault(t, []).append((i0, i1, slot, n))
        assert sorted(parts) == list(range(tiles))
        for t, q in parts.items():
            q.sort()
            assert q[0][0] == 0 and q[-1][1] == p["KI"] and all(a[1] == b[0] for a, b in zip(q, q[1:]))
            assert all(n == len(q) and slot == q[0][2] and (slot >= 0) == (len(q) > 1) for _, _, slot, n in q)
        slots = {t: q[0][2] for t, q in parts.items() if q[0][2] >= 0}
        assert len(set(slots.values())) == len(slots)          # a slot serves one tile
        n = p["cluster"]
        if n > 1:                                              # n CTAs per tile, one tile per CTA
            assert n in (2, 4) and p["grid"] == n * tiles and all(len(q) == n for q in parts.values())
            assert all(t == c // n for c, t, *_ in units(p))

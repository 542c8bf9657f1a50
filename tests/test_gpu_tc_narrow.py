"""Narrow single-CTA tiles (128 x 64, 128 x 32) of the dense tensor-core product: the same piece products in
the same chunks as 128 x 128 tiles, so the same sums bit for bit; and the runs that choose them."""
import pytest
import torch

from paper_1507_02087_gb300 import inputs

pytestmark = pytest.mark.gpu


def product(fmt, mats, upper, tile, lowprec):
    from paper_1507_02087_gb300 import sp2
    ld = mats[0].shape[0]
    if fmt == "bf16":
        planes = []
        for m in mats:
            p0 = m.bfloat16()
            p1 = (m - p0.float()).bfloat16()
            planes.append(torch.stack([p0, p1, (m - p0.float() - p1.float()).bfloat16()]))
    elif fmt == "fp16":
        planes = []
        for m in mats:
            p0 = (m * 2.0 ** 14).half()
            planes.append(torch.stack([p0, (m * 2.0 ** 14 - p0.float()).half()]))
    else:
        mask = ~0x1FFF
        planes = []
        for m in mats:
            hi = (m.view(torch.int32) & mask).view(torch.float32)
            lo = ((m - hi).view(torch.int32) & mask).view(torch.float32)
            planes.append(torch.stack([hi, lo]))
    arena = torch.stack(planes).contiguous()
    out = torch.full((ld, ld), float("nan"), device="cuda")
    sp2.sp2_test_tc_gemm(arena, ld, len(mats), 0, len(mats) - 1, upper, out, tile=tile, fmt=fmt, lowprec=lowprec)
    return out


@pytest.mark.parametrize("fmt", ["bf16", "fp16", "tf32"])
@pytest.mark.parametrize("lowprec", [False, True])
@pytest.mark.parametrize("ld", [128, 384, 1280])
def test_widths_agree_bit_for_bit(fmt, lowprec, ld):
    g = torch.Generator(device="cpu").manual_seed(ld)
    A = (torch.randn(ld, ld, generator=g) / ld ** 0.5).clamp(-1, 1).cuda()
    S = (0.5 * (A + A.T)).contiguous()
    for mats, upper in (([A, S], False), ([S], True)):
        wide = product(fmt, mats, upper, "128", lowprec)
        assert torch.isfinite(wide).all()
        for tile in ("64", "32"):
            assert torch.equal(product(fmt, mats, upper, tile, lowprec), wide)


@pytest.mark.parametrize("N", [100, 400, 1025, 1300])      # 32, 32, 64 and 64 columns
@pytest.mark.parametrize("prec", ["fp16x3", "bf16x6", "tf32x3"])
@pytest.mark.parametrize("norm", ["fro", "mixed"])
def test_runs_agree_with_wide_tiles(N, prec, norm):
    from paper_1507_02087_gb300 import sp2
    case = inputs.dense_gapped(N, N // 3, gap=0.05, seed=N, device="cuda", want_exact=False)
    out = {}
    for tile in ("auto", "128"):
        with sp2.Purifier(N, N // 3, prec, tile=tile, norm=norm) as P:
            D = P.run(case.F)
            out[tile] = D, P.info()
    (Da, ia), (Dw, iw) = out["auto"], out["128"]
    assert ia["status"] == 0 and ia["tile"] == "128"
    assert ia["n_iter"] == iw["n_iter"] and torch.equal(Da, Dw)
    # the same FP32 partials, summed in FP64 in another order
    assert abs(ia["v"] / iw["v"] - 1.0).max() < 1e-11 if (iw["v"] > 0).all() else True

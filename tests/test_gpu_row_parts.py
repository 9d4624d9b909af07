"""The row movers with a token's row split over several warps (few tokens, rows of
128 vectors and more) and the dispatch that ranks and copies in one launch (up to
512 slots), against float64: combine and its backward, the dispatch
backward, and the fused dispatch / router backward.  bf16 results are one
rounding of an fp32 sum (2^-9); fp32 sums of n terms stay within n 2^-24 of
sum |a b|, about sqrt(n) 2^-24 of the norm, of which four times is allowed."""
import pytest
import torch

from paper_2608_28511_gb300 import abi

pytestmark = pytest.mark.gpu


def _rel(a, b):
    return float((a.double() - b).norm() / b.norm())


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("T,K,E,D", [(1, 1, 4, 64), (3, 2, 5, 512), (13, 4, 33, 1088), (9, 8, 64, 2560),
                                     (7, 16, 100, 2048), (73, 7, 64, 576), (128, 4, 31, 1024),
                                     (171, 3, 256, 512), (512, 1, 2, 64), (1830, 3, 40, 1024), (3700, 2, 8, 512),
                                     (1823, 1, 16, 512), (1825, 1, 16, 1024), (2431, 1, 4, 2048)])
def test_row_movers(T, K, E, D, dtype):
    import __graft_entry__
    __graft_entry__.build()
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    tol = 2.0 ** -9 if dtype == "bf16" else 4.0 * (K + 1) ** 0.5 * 2.0 ** -24
    g = torch.Generator(device="cuda").manual_seed(T * K + D)
    rnd = lambda *s, d=dt: torch.randn(*s, generator=g, device="cuda").to(d)  # noqa: E731
    e = lambda *s, d=dt: torch.empty(*s, device="cuda", dtype=d)  # noqa: E731
    f32, i32 = torch.float32, torch.int32
    shp = abi.MoeShape.of(T, 1, K, D, E, 64, dtype)
    ws = torch.empty(abi.moe_workspace_size(shp), dtype=torch.uint8, device="cuda")
    x, w, y_perm, dy, dx_perm = rnd(T, D), rnd(E, D), rnd(T * K, D), rnd(T, D), rnd(T * K, D)
    top = torch.topk(rnd(T, E, d=f32), K, dim=1)
    idx, prob = top.indices.to(i32).contiguous(), torch.softmax(top.values, 1).contiguous()
    off, ros, tor, pp, xp = e(E + 1, d=i32), e(T * K, d=i32), e(T * K, d=i32), e(T * K, d=f32), e(T * K, D)
    abi.moe_dispatch(shp, x, idx, prob, off, ros, tor, xp, pp, ws)
    r = ros.view(T, K).long()
    assert torch.equal(xp[r], x[:, None].expand(T, K, D))
    y, dy_perm, dpp = e(T, D), e(T * K, D), e(T * K, d=f32)
    abi.moe_combine(shp, y_perm, pp, ros, y)
    assert _rel(y, (prob.double()[..., None] * y_perm[r].double()).sum(1)) < tol
    abi.moe_combine_bwd(shp, dy, y_perm, pp, ros, dy_perm, dpp)
    assert _rel(dy_perm[r], prob.double()[..., None] * dy.double()[:, None]) < tol
    assert _rel(dpp[r], (y_perm[r].double() * dy.double()[:, None]).sum(2)) < 4.0 * D ** 0.5 * 2.0 ** -24
    dx, dprob = e(T, D), e(T, K, d=f32)
    sum_dx = dx_perm[r].double().sum(1)
    abi.moe_dispatch_bwd(shp, dx_perm, dpp, ros, dx, dprob)
    assert _rel(dx, sum_dx) < tol and torch.equal(dprob, dpp[r])
    dz, dwr = e(T, E, d=f32), e(E, D, d=f32)
    abi.moe_dispatch_route_bwd(shp, dx_perm, dpp, ros, x, w, idx, prob, dx, dprob, dz, dwr, ws)
    dp = dpp[r].double()
    # p (dp - sum p dp) cancels: its fp32 error is relative to p |dp|
    zk = prob.double() * (dp - (prob.double() * dp).sum(1, keepdim=True))
    got = dz.gather(1, idx.long()).double()
    assert float((got - zk).norm()) < 4.0 * (K + 1) ** 0.5 * 2.0 ** -24 * float((prob.double() * dp).norm())
    assert int((dz != 0).sum()) <= T * K and torch.equal(dprob, dpp[r])
    # K more terms, dz w, on top of the K rows
    ref = sum_dx + torch.einsum("tk,tkd->td", got, w[idx.long()].double())
    assert _rel(dx, ref) < (2.0 ** -9 if dtype == "bf16" else 4.0 * (2 * K + 1) ** 0.5 * 2.0 ** -24)
    assert abi.moe_check_device_status() == 0

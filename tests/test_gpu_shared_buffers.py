"""Calls whose output takes the place of an input that the call has finished
with: the same bits as with buffers of their own."""
import itertools

import pytest
import torch

from paper_2608_28511_gb300 import abi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("counts,D,F", [([700, 0, 129, 300], 256, 256), ([5] * 40, 128, 128)])
@pytest.mark.parametrize("over", ["dy_perm", "x_perm", "act"])
def test_expert_backward_dx_over_an_input(over, counts, D, F, dtype):
    """moe_expert_ffn_bwd with dx_perm over an input of its size."""
    E, TK = len(counts), sum(counts)
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    g = torch.Generator(device="cuda").manual_seed(TK + D)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda").to(dt)  # noqa: E731
    shp = abi.MoeShape.of(TK, 1, 1, D, E, F, dtype)
    off = torch.tensor([0] + list(itertools.accumulate(counts)), dtype=torch.int32, device="cuda")
    inp = {"dy_perm": rnd(TK, D), "x_perm": rnd(TK, D), "h": rnd(TK, 2 * F), "act": rnd(TK, F)}
    w1, w2 = rnd(E, 2 * F, D), rnd(E, D, F)
    ws = torch.empty(abi.moe_workspace_size(shp), dtype=torch.uint8, device="cuda")
    out = []
    for shared in (False, True):
        b = {k: v.clone() for k, v in inp.items()}
        dx = b[over] if shared else torch.empty(TK, D, dtype=dt, device="cuda")
        dw1, dw2 = torch.empty(E, 2 * F, D, device="cuda"), torch.empty(E, D, F, device="cuda")
        abi.moe_expert_ffn_bwd(shp, b["dy_perm"], b["x_perm"], b["h"], b["act"], off, w1, w2, dx, dw1, dw2, ws)
        out.append((dx, dw1, dw2))
    assert abi.moe_check_device_status() == 0
    assert all(torch.equal(p, q) for p, q in zip(*out))


@pytest.mark.parametrize("T,K,D", [(1, 1, 64), (128, 4, 512), (500, 1, 1024), (300, 3, 256)])
def test_dispatch_rows_over_the_indices(T, K, D):
    """moe_dispatch with row_of_slot over topk_idx, on both sides of the size up
    to which ranking and row copies are one launch."""
    E = 64
    g = torch.Generator(device="cuda").manual_seed(T)
    shp = abi.MoeShape.of(T, 1, K, D, E, 64)
    x = torch.randn(T, D, generator=g, device="cuda").bfloat16()
    top = torch.topk(torch.randn(T, E, generator=g, device="cuda"), K, dim=1)
    prob = torch.softmax(top.values, 1).contiguous()
    ws = torch.empty(abi.moe_workspace_size(shp), dtype=torch.uint8, device="cuda")
    i32 = dict(dtype=torch.int32, device="cuda")
    out = []
    for shared in (False, True):
        idx = top.indices.to(torch.int32).contiguous()
        ros = idx.view(-1) if shared else torch.empty(T * K, **i32)
        off, tor, pp = torch.empty(E + 1, **i32), torch.empty(T * K, **i32), torch.empty(T * K, device="cuda")
        xp = torch.empty(T * K, D, dtype=torch.bfloat16, device="cuda")
        abi.moe_dispatch(shp, x, idx, prob, off, ros, tor, xp, pp, ws)
        out.append((off, ros, tor, xp, pp))
    assert abi.moe_check_device_status() == 0
    assert all(torch.equal(p, q) for p, q in zip(*out))


@pytest.mark.parametrize("T,K,D", [(1, 1, 1024), (300, 8, 2048), (150, 16, 1024), (900, 2, 2560), (700, 4, 256)])
def test_probability_gradient_over_the_probabilities(T, K, D):
    """The dispatch backwards with dtopk_prob over topk_prob, and over row_of_slot,
    with a token's row moved by one warp or by eight."""
    E = 64
    g = torch.Generator(device="cuda").manual_seed(T)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")  # noqa: E731
    shp = abi.MoeShape.of(T, 1, K, D, E, 64)
    x, w, dxp, dpp = rnd(T, D).bfloat16(), rnd(E, D).bfloat16(), rnd(T * K, D).bfloat16(), rnd(T * K)
    top = torch.topk(rnd(T, E), K, dim=1)
    idx, p0 = top.indices.to(torch.int32).contiguous(), torch.softmax(top.values, 1).contiguous()
    ros0 = torch.randperm(T * K, generator=g, device="cuda").to(torch.int32)
    ws = torch.empty(abi.moe_workspace_size(shp), dtype=torch.uint8, device="cuda")
    out = []
    for shared in (False, True):
        prob, ros = p0.clone(), ros0.clone()
        dprob = prob if shared else torch.empty_like(prob)
        dx, dz, dwr = torch.empty_like(x), torch.empty(T, E, device="cuda"), torch.empty(E, D, device="cuda")
        abi.moe_dispatch_route_bwd(shp, dxp, dpp, ros, x, w, idx, prob, dx, dprob, dz, dwr, ws)
        dx2, dp2 = torch.empty_like(x), ros.view(torch.float32) if shared else torch.empty(T * K, device="cuda")
        abi.moe_dispatch_bwd(shp, dxp, dpp, ros, dx2, dp2)
        out.append((dx, dprob, dz, dwr, dx2, dp2))
    assert abi.moe_check_device_status() == 0
    assert all(torch.equal(p, q) for p, q in zip(*out))

"""The fp32 expert block: the forward on each of the tiles that its SwiGLU epilogue
takes (32, 64 and 128 rows of 128 columns), and the backward, whose three products that depend on dH run in one
launch and whose SwiGLU backward runs in the epilogue of dA's product, on every
tile size that the row counts select, with empty experts.  Each output against
float64, those after h and a from the GPU's own; a sum of n fp32 products is within
n 2^-24 of sum |a b|, about sqrt(n) 2^-24 of the result's norm for random signs,
and dH carries the sum over D and about ten roundings of its own: four times the
sum of both is allowed."""
import itertools

import pytest
import torch

from paper_2608_28511_gb300 import abi

pytestmark = pytest.mark.gpu

EDGES = [0, 1, 31, 32, 33, 0, 63, 64, 65, 130]


@pytest.mark.parametrize("counts,D,F", [([1], 64, 64), (EDGES, 64, 64), (EDGES, 192, 128), (EDGES, 64, 1216),
                                        ([0, 700, 129, 1], 512, 448), ([5] * 40, 128, 192),
                                        ([900, 0, 1, 1100], 320, 768), ([300, 0, 150, 50], 128, 1216)])
def test_fp32_expert_backward(counts, D, F):
    import __graft_entry__
    __graft_entry__.build()
    E, TK = len(counts), sum(counts)
    g = torch.Generator(device="cuda").manual_seed(D + F + TK)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")  # noqa: E731
    shp = abi.MoeShape.of(TK, 1, 1, D, E, F, "f32")
    off = torch.tensor([0] + list(itertools.accumulate(counts)), dtype=torch.int32, device="cuda")
    x, dy, w1, w2 = rnd(TK, D), rnd(TK, D), rnd(E, 2 * F, D) * D ** -0.5, rnd(E, D, F) * F ** -0.5
    h, act, y, dx = (torch.empty(TK, n, device="cuda") for n in (2 * F, F, D, D))
    dw1, dw2 = torch.full_like(w1, 3.0), torch.full_like(w2, 3.0)
    ws = torch.empty(abi.moe_workspace_size(shp), dtype=torch.uint8, device="cuda")
    abi.moe_expert_ffn(shp, x, off, w1, w2, h, act, y, ws)
    abi.moe_expert_ffn_bwd(shp, dy, x, h, act, off, w1, w2, dx, dw1, dw2, ws)
    assert abi.moe_check_device_status() == 0

    def near(got, ref, n):
        tol = 4.0 * 2.0 ** -24 * (max(n, 16) ** 0.5 + max(D, 16) ** 0.5 + 10.0)
        assert float((got.double() - ref).norm()) <= tol * float(ref.norm()), (n, float(ref.norm()))

    for e, n in enumerate(counts):
        r = slice(int(off[e]), int(off[e]) + n)
        if not n:
            assert not dw1[e].any() and not dw2[e].any()
            continue
        he = h[r].double().view(n, F // 64, 2, 64)
        gate, up = he[:, :, 0].reshape(n, F), he[:, :, 1].reshape(n, F)
        s = torch.sigmoid(gate)
        near(h[r], x[r].double() @ w1[e].double().T, D)
        near(act[r], gate * s * up, 1)
        near(y[r], act[r].double() @ w2[e].double().T, F)
        dA = dy[r].double() @ w2[e].double()
        dg, du = dA * up * s * (1 + gate * (1 - s)), dA * gate * s
        dH = torch.stack([dg.view(n, F // 64, 64), du.view(n, F // 64, 64)], 2).reshape(n, 2 * F)
        near(dx[r], dH @ w1[e].double(), 2 * F)
        near(dw1[e], dH.T @ x[r].double(), n)
        near(dw2[e], dy[r].double().T @ act[r].double(), n)

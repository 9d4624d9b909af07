"""Expert GEMMs at the edges of the row steps in which a short tile's A rows are
copied (16 rows, all 128 of a CTA's from 65 on; a tile is two CTAs): experts of
every such row count side by side, each compared alone with float64 products of
the same bf16 operands, forward and input gradient.  One bf16 rounding of an fp32
sum is within 2^-9; dH is rounded to bf16 from a hardware tanh (2^-7)."""
import itertools

import pytest
import torch

from paper_2608_28511_gb300 import abi

pytestmark = pytest.mark.gpu

COUNTS = [0, 1, 15, 16, 17, 47, 48, 49, 63, 64, 65, 80, 127, 128, 129, 143, 144, 145, 191, 192, 193, 208, 0, 256, 272,
          320, 321, 5]


@pytest.mark.parametrize("D,F", [(256, 128), (192, 320)])
def test_expert_rows_at_copy_steps(D, F):
    import __graft_entry__
    __graft_entry__.build()
    E, TK, bf = len(COUNTS), sum(COUNTS), torch.bfloat16
    g = torch.Generator(device="cuda").manual_seed(D)
    shp = abi.MoeShape.of(TK, 1, 1, D, E, F, "bf16")
    off = torch.tensor([0] + list(itertools.accumulate(COUNTS)), dtype=torch.int32, device="cuda")
    x, w1, w2 = (torch.randn(*s, generator=g, device="cuda").to(bf) for s in ((TK, D), (E, 2 * F, D), (E, D, F)))
    h, act, y = (torch.empty(*s, dtype=bf, device="cuda") for s in ((TK, 2 * F), (TK, F), (TK, D)))
    ws = torch.empty(abi.moe_workspace_size(shp), dtype=torch.uint8, device="cuda")
    abi.moe_expert_ffn(shp, x, off, w1, w2, h, act, y, ws)
    dy, dx = torch.randn(TK, D, generator=g, device="cuda").to(bf), torch.empty(TK, D, dtype=bf, device="cuda")
    dw1, dw2 = torch.empty(E, 2 * F, D, device="cuda"), torch.empty(E, D, F, device="cuda")
    abi.moe_expert_ffn_bwd(shp, dy, x, h, act, off, w1, w2, dx, dw1, dw2, ws)
    assert abi.moe_check_device_status() == 0
    for e, n in enumerate(COUNTS):
        r = slice(int(off[e]), int(off[e]) + n)
        if not n:
            continue
        for got, a, w in ((h[r], x[r], w1[e]), (y[r], act[r], w2[e])):
            ref = a.double() @ w.double().T
            assert float((got.double() - ref).norm() / ref.norm()) < 2.0 ** -9, (e, n)
        he = h[r].double().view(n, F // 64, 2, 64)
        gate, up = he[:, :, 0].reshape(n, F), he[:, :, 1].reshape(n, F)
        s = torch.sigmoid(gate)
        dA = dy[r].double() @ w2[e].double()
        dH = torch.stack([(dA * up * s * (1 + gate * (1 - s))).view(n, F // 64, 64),
                          (dA * gate * s).view(n, F // 64, 64)], 2).reshape(n, 2 * F)
        ref = dH @ w1[e].double()
        assert float((dx[r].double() - ref).norm() / ref.norm()) < 2.0 ** -7, (e, n)

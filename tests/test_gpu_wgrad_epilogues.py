"""Expert weight gradients in each of the forms that the average rows per expert
select (stores by the copy engine, by eight and by four epilogue warps), with
empty and ragged experts and widths that end inside a tile.  dw2 against float64
products of the same bf16 operands: a sum of n products in fp32 is within
n 2^-24 of sum |a b|, about sqrt(n) 2^-24 of the norm, of which four times is
allowed; dw1's operand dH, which dx_perm shares, is rounded to bf16 from a
hardware tanh (2^-7)."""
import itertools

import pytest
import torch

from paper_2608_28511_gb300 import abi

pytestmark = pytest.mark.gpu

COUNTS = {"bulk": [0, 1, 63, 64, 65, 0, 128, 200, 255, 129, 700],
          "eight": [0, 1, 640, 641, 700, 129, 704, 0, 577],
          "four": [0, 900, 1, 1025, 0, 2048]}


@pytest.mark.parametrize("form", list(COUNTS))
@pytest.mark.parametrize("D,F", [(64, 64), (320, 448), (576, 192), (1088, 128)])
def test_weight_gradients(form, D, F):
    import __graft_entry__
    __graft_entry__.build()
    counts, bf = COUNTS[form], torch.bfloat16
    E, TK = len(counts), sum(counts)
    g = torch.Generator(device="cuda").manual_seed(D + F + TK)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda").to(bf)  # noqa: E731
    shp = abi.MoeShape.of(TK, 1, 1, D, E, F, "bf16")
    off = torch.tensor([0] + list(itertools.accumulate(counts)), dtype=torch.int32, device="cuda")
    x, dy, h, act = rnd(TK, D), rnd(TK, D), rnd(TK, 2 * F), rnd(TK, F)
    w1, w2, dx = rnd(E, 2 * F, D), rnd(E, D, F), torch.empty(TK, D, dtype=bf, device="cuda")
    # one expert's block more at the end, which stays as it was
    dw1, dw2 = torch.full((E + 1, 2 * F, D), 3.0, device="cuda"), torch.full((E + 1, D, F), 3.0, device="cuda")
    ws = torch.empty(abi.moe_workspace_size(shp), dtype=torch.uint8, device="cuda")
    abi.moe_expert_ffn_bwd(shp, dy, x, h, act, off, w1, w2, dx, dw1[:E], dw2[:E], ws)
    assert abi.moe_check_device_status() == 0
    assert bool((dw1[E] == 3.0).all()) and bool((dw2[E] == 3.0).all())
    for e, n in enumerate(counts):
        r = slice(int(off[e]), int(off[e]) + n)
        if not n:
            assert not dw1[e].any() and not dw2[e].any()
            continue
        ref = dy[r].double().T @ act[r].double()
        assert float((dw2[e].double() - ref).norm() / ref.norm()) < 4.0 * max(n, 16) ** 0.5 * 2.0 ** -24, (e, n)
        he = h[r].double().view(n, F // 64, 2, 64)
        gate, up = he[:, :, 0].reshape(n, F), he[:, :, 1].reshape(n, F)
        s = torch.sigmoid(gate)
        dA = dy[r].double() @ w2[e].double()
        dg, du = dA * up * s * (1 + gate * (1 - s)), dA * gate * s
        dH = torch.stack([dg.view(n, F // 64, 64), du.view(n, F // 64, 64)], 2).reshape(n, 2 * F)
        for got, ref in ((dw1[e], dH.T @ x[r].double()), (dx[r], dH @ w1[e].double())):
            assert float((got.double() - ref).norm() / ref.norm()) < 2.0 ** -7, (e, n)

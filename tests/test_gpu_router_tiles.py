"""Router logits at the edges of the tensor-core GEMM's row tiles, whose height
follows from the number of tokens (whole 8-row steps, one round of the SM pairs
up to 128 rows each), against float64.  A sum of D bf16 products in fp32 is
within D 2^-24 of sum |a b|, about sqrt(D) 2^-24 of the result's norm for random
signs; four times that is allowed."""
import pytest
import torch

from paper_2608_28511_gb300 import abi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("E", [4, 36, 64, 100, 128, 200, 256])
@pytest.mark.parametrize("T", [1, 8, 9, 17, 1215, 1217, 2045, 19456, 19457, 20001])
def test_router_logits(T, E):
    import __graft_entry__
    __graft_entry__.build()
    D, K = 320, 2
    g = torch.Generator(device="cuda").manual_seed(T + E)
    shp = abi.MoeShape.of(T, 1, K, D, E, 64, "bf16")
    x, w = (torch.randn(*s, generator=g, device="cuda").bfloat16() for s in ((T, D), (E, D)))
    bias = torch.randn(E, generator=g, device="cuda")
    z = torch.full((T + 1, E), 7.0, device="cuda")  # one row past the end stays as it was
    idx, p = torch.empty(T, K, dtype=torch.int32, device="cuda"), torch.empty(T, K, device="cuda")
    ws = torch.empty(abi.moe_workspace_size(shp), dtype=torch.uint8, device="cuda")
    for b in (None, bias):
        abi.moe_route(shp, x, w, b, z[:T], idx, p, ws)
        ref = x.double() @ w.double().T + (0.0 if b is None else b.double())
        assert float((z[:T].double() - ref).norm() / ref.norm()) < 4.0 * D ** 0.5 * 2.0 ** -24
    assert bool((z[T] == 7.0).all()) and abi.moe_check_device_status() == 0

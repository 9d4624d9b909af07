"""The CUDA-core GEMM engine at the edges of its tiles, against float64.

fp32 projections and their backward reach every operand layout (rows of k
contiguous, rows of m or n contiguous) and every tile size, the routers with an
odd number of experts its unaligned and split reductions.  Bound: a sum of n
fp32 products in any order is within n 2^-24 of sum |a b|, about sqrt(n) 2^-24 of
the result's norm for random signs; four times that is allowed.
"""
import pytest
import torch

from paper_2608_28511_gb300 import abi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _rel(a, b):
    return float((a.double() - b).norm() / b.norm())


def _tol(n):
    return 4.0 * max(n, 16) ** 0.5 * 2.0 ** -24


@pytest.mark.parametrize("T,n_in,n_out", [(1, 64, 64), (31, 64, 128), (33, 192, 64), (127, 128, 192), (129, 64, 1088),
                                          (1000, 320, 512), (2049, 576, 1344), (5000, 64, 1024)])
@pytest.mark.parametrize("accumulate", [False, True])
def test_fp32_projection(T, n_in, n_out, accumulate):
    g = torch.Generator(device="cuda").manual_seed(T + n_in)
    shp = abi.MoeShape.of(T, 1, 1, 64, 1, 64, "f32", n_in)
    x, w, dout, din0 = (torch.randn(*s, generator=g, device="cuda")
                        for s in ((T, n_in), (n_out, n_in), (T, n_out), (T, n_in)))
    out = torch.empty(T, n_out, device="cuda")
    ws = torch.empty(abi.moe_workspace_size(shp), dtype=torch.uint8, device="cuda")
    abi.moe_latent_proj(shp, n_in, n_out, x, w, out, ws)
    assert _rel(out, x.double() @ w.double().T) < _tol(n_in)
    din, dw = din0.clone(), torch.empty(n_out, n_in, device="cuda")
    abi.moe_latent_proj_bwd(shp, n_in, n_out, dout, x, w, din, accumulate, dw, ws)
    ref = dout.double() @ w.double() + (din0.double() if accumulate else 0.0)
    assert _rel(din, ref) < _tol(n_out)
    assert _rel(dw, dout.double().T @ x.double()) < _tol(T)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("T,E,D", [(1, 3, 64), (511, 5, 128), (513, 13, 192), (3001, 60, 256), (5000, 129, 64),
                                   (4096, 12, 512), (4096, 12, 1024), (3700, 31, 2048), (2100, 33, 1088)])
def test_router_with_odd_experts(T, E, D, dtype):
    """Logits, and the weight gradient with and without the split over tokens."""
    K = min(3, E)
    g = torch.Generator(device="cuda").manual_seed(T + E)
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    shp = abi.MoeShape.of(T, 1, K, D, E, 64, dtype)
    x = torch.randn(T, D, generator=g, device="cuda").to(dt)
    w = torch.randn(E, D, generator=g, device="cuda").to(dt)
    bias = torch.randn(E, generator=g, device="cuda")
    ws = torch.empty(abi.moe_workspace_size(shp), dtype=torch.uint8, device="cuda")
    z, dz, dwr = (torch.empty(*s, device="cuda") for s in ((T, E), (T, E), (E, D)))
    idx, p = torch.empty(T, K, dtype=torch.int32, device="cuda"), torch.empty(T, K, device="cuda")
    abi.moe_route(shp, x, w, bias, z, idx, p, ws)
    assert _rel(z, x.double() @ w.double().T + bias.double()) < max(_tol(D), 1e-5 if dtype == "bf16" else 0.0)
    dp = torch.randn(T, K, generator=g, device="cuda")
    dx = torch.zeros(T, D, device="cuda").to(dt)
    abi.moe_route_bwd(shp, x, w, idx, p, dp, dx, dwr, dz, ws)
    # fp32 dz everywhere but on the tensor cores (bf16 and E a multiple of 8)
    ref = dz.double().T @ x.double()
    assert _rel(dwr, ref) < (_tol(T) if dtype == "f32" or E % 8 else 4e-3)
    assert abi.moe_check_device_status() == 0

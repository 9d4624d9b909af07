"""The warp-per-token top-K selection where its lists are short or ragged and
where keys are equal, infinite or NaN: indices against a plain sort of the same
keys (NaN as -inf, -0 as +0, ties to the lower expert)."""
import numpy as np
import pytest
import torch

from paper_2608_28511_gb300 import abi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("E,K", [(1, 1), (2, 2), (5, 5), (16, 16), (31, 3), (33, 8), (63, 16), (65, 4), (100, 7),
                                 (129, 9), (255, 16), (256, 1)])
def test_selection(E, K):
    T = 333
    z = torch.randn(T, E, generator=torch.Generator().manual_seed(E * 17 + K))
    z[0] = float("-inf")                               # every key equal
    z[1] = 0.0
    z[1, ::2] = -0.0                                   # -0 ties with +0
    z[2, : E // 2 + 1] = float("nan")
    z[3, -1] = float("inf")
    z[4] = torch.round(z[4])                           # many ties, in and across lists
    z[5::9] = torch.round(z[5::9] * 2)
    z[6, :] = z[6, 0]
    z[6, -1] = float("nan")
    idx = torch.empty(T, K, dtype=torch.int32, device="cuda")
    prob = torch.empty(T, K, device="cuda")
    abi.moe_topk(abi.MoeShape.of(T, 1, K, 64, E, 64), z.cuda(), idx, prob)
    key = np.where(np.isnan(z.numpy()), -np.inf, z.numpy()) + 0.0
    ref = np.argsort(-key, axis=1, kind="stable")[:, :K]
    assert (idx.cpu().numpy() == ref).all()
    top = np.take_along_axis(key, ref, 1).astype(np.float64)
    fine = np.isfinite(top[:, 0])                      # an infinite best key has no softmax
    w = np.exp(top[fine] - top[fine][:, :1])
    assert np.abs(prob.cpu().numpy()[fine] - w / w.sum(1, keepdims=True)).max() <= 1e-6
    assert abi.moe_check_device_status() == 0


@pytest.mark.parametrize("K", [5, 8, 16])
def test_probabilities_are_summed_best_first(K):
    """One logit 17 above the others, whose terms (4.1e-8 and less, of a best one
    of 1) are each below half a unit in the last place of the running sum when
    added best first: the sum is exactly 1.  Added to each other first they move
    it.  The same for the sigmoid scores, of which the best is exactly 1."""
    T, E = 40, 64
    z = -17.0 - 0.01 * torch.rand(T, E, generator=torch.Generator().manual_seed(K))
    best = torch.arange(T) % E
    z[torch.arange(T), best] = 0.0
    idx = torch.empty(T, K, dtype=torch.int32, device="cuda")
    prob = torch.empty(T, K, device="cuda")
    shp = abi.MoeShape.of(T, 1, K, 64, E, 64)
    abi.moe_topk(shp, z.cuda(), idx, prob)
    assert torch.equal(idx[:, 0].cpu().long(), best) and bool((prob[:, 0] == 1.0).all())
    z[torch.arange(T), best] = 40.0
    f, loss = torch.empty(1, E, device="cuda"), torch.empty(4, device="cuda")
    ws = torch.empty(abi.moe_workspace_size(shp), dtype=torch.uint8, device="cuda")
    abi.moe_topk_sigmoid(shp, z.cuda(), None, 1e-4, None, idx, prob, f, loss, ws)
    assert torch.equal(idx[:, 0].cpu().long(), best) and bool((prob[:, 0] == 1.0).all())
    assert abi.moe_check_device_status() == 0


@pytest.mark.parametrize("E,K", [(3, 3), (4, 1), (7, 7), (8, 2), (9, 2), (15, 9), (16, 16), (17, 3), (24, 6),
                                 (31, 7), (32, 16), (40, 8), (64, 5), (128, 16), (200, 8), (256, 16)])
def test_equal_keys_in_every_place(E, K):
    """Pairs and runs of equal keys at each rank up to past the last chosen one, in
    one lane (experts 32 apart) and across lanes, and rows that hold few distinct
    keys: the lower expert comes first."""
    g = torch.Generator().manual_seed(E + K)
    rows = []
    for r in range(min(K + 1, E - 1)):
        for run in (2, 3, 40):
            for shift in (1, 32):
                z = torch.randn(E, generator=g).sort(descending=True).values
                z[r : r + run] = z[r].clone()                      # ranks r .. r + run - 1 are equal
                order = torch.randperm(E, generator=g)
                place = torch.empty(E)
                if shift == 32:                                    # ... and lie 32 experts apart
                    order = torch.arange(E).view(-1, 1) if E <= 32 else torch.argsort(torch.arange(E) % 32, stable=True)
                    order = order.reshape(-1).roll(int(torch.randint(E, (1,), generator=g)))
                place[order] = z
                rows.append(place)
    for n in (1, 2, 3):
        rows += list(torch.randint(0, n, (20, E), generator=g).float())
    z = torch.stack(rows)
    T = z.shape[0]
    idx, prob = torch.empty(T, K, dtype=torch.int32, device="cuda"), torch.empty(T, K, device="cuda")
    shp = abi.MoeShape.of(T, 1, K, 64, E, 64)
    ref = np.argsort(-z.numpy(), axis=1, kind="stable")[:, :K]
    abi.moe_topk(shp, z.cuda(), idx, prob)
    assert (idx.cpu().numpy() == ref).all()
    keys, f, loss = torch.empty(T, E, device="cuda"), torch.empty(1, E, device="cuda"), torch.empty(4, device="cuda")
    ws = torch.empty(abi.moe_workspace_size(shp), dtype=torch.uint8, device="cuda")
    abi.moe_topk_sigmoid(shp, z.cuda(), None, 1e-4, keys, idx, prob, f, loss, ws)
    ref = np.argsort(-keys.cpu().numpy(), axis=1, kind="stable")[:, :K]
    assert (idx.cpu().numpy() == ref).all() and abi.moe_check_device_status() == 0


@pytest.mark.parametrize("E", [3, 5, 16, 20, 64, 130])
@pytest.mark.parametrize("S,GBS", [(1, 3), (4, 5), (15, 2), (17, 2), (33, 1), (63, 2), (65, 3), (100, 1)])
def test_sigmoid_statistics_of_short_sequences(S, GBS, E):
    """Choice counts and the balance loss where a sequence does not give every warp
    of a block the same number of tokens: f exactly from the choices, the loss
    against float64 (a mean of T fp32 quotients: within 1e-6)."""
    K, T = min(E, 3), S * GBS
    g = torch.Generator().manual_seed(S * E)
    z, b = torch.randn(T, E, generator=g), torch.randn(E, generator=g) * 0.05
    shp = abi.MoeShape.of(S, GBS, K, 64, E, 64)
    idx, prob = torch.empty(T, K, dtype=torch.int32, device="cuda"), torch.empty(T, K, device="cuda")
    f, loss = torch.empty(GBS, E, device="cuda"), torch.empty(4, device="cuda")
    keys = torch.empty(T, E, device="cuda")
    ws = torch.empty(abi.moe_workspace_size(shp), dtype=torch.uint8, device="cuda")
    abi.moe_topk_sigmoid(shp, z.cuda(), b.cuda(), 0.5, keys, idx, prob, f, loss, ws)
    assert abi.moe_check_device_status() == 0
    i = idx.cpu().long()
    assert (i.numpy() == np.argsort(-keys.cpu().numpy(), axis=1, kind="stable")[:, :K]).all()
    s = torch.sigmoid(z.double())
    cnt = torch.zeros(T, E, dtype=torch.float64).scatter_(1, i, 1.0).view(GBS, S, E).sum(1)
    assert float((f.cpu().double() - cnt * E / (K * S)).abs().max()) <= 1e-6 * E
    sel = s.gather(1, i)
    assert float((prob.cpu().double() - sel / sel.sum(1, keepdim=True)).abs().max()) <= 1e-6
    P = (s / s.sum(1, keepdim=True)).view(GBS, S, E).mean(1)
    want = 0.5 / GBS * float((cnt * E / (K * S) * P).sum())
    assert abs(float(loss[0]) - want) <= 2e-6 * abs(want)


@pytest.mark.parametrize("T", [4096, 4097])
@pytest.mark.parametrize("E,K", [(17, 3), (32, 8)])
def test_both_forms_for_up_to_32_experts(T, E, K):
    """A warp per token up to 4096 tokens, eight lanes per token above: the same
    indices and bits of the probabilities for the rows that both have."""
    z = torch.round(torch.randn(8000, E, generator=torch.Generator().manual_seed(T)) * 8) / 8
    idx, prob = torch.empty(8000, K, dtype=torch.int32, device="cuda"), torch.empty(8000, K, device="cuda")
    abi.moe_topk(abi.MoeShape.of(8000, 1, K, 64, E, 64), z.cuda(), idx, prob)
    i2, p2 = torch.empty(T, K, dtype=torch.int32, device="cuda"), torch.empty(T, K, device="cuda")
    abi.moe_topk(abi.MoeShape.of(T, 1, K, 64, E, 64), z[:T].cuda(), i2, p2)
    assert torch.equal(i2, idx[:T]) and torch.equal(p2, prob[:T])
    assert (i2.cpu().numpy() == np.argsort(-z[:T].numpy(), axis=1, kind="stable")[:, :K]).all()

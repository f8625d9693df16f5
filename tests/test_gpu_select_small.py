"""Selection of few rows by one cluster, and of more or longer ones by the general way: both against the oracle's rule, over
row counts and lengths on both sides of the lines between them, with a capacity that is too small and with masses that are none."""
import numpy as np
import pytest
import torch

from oracle import losa_oracle as orc

pytestmark = pytest.mark.gpu


def lib():
    import paper_2608_12032_b200 as losa
    return losa


def masses(rows, nKb, seed):
    g = torch.Generator("cpu").manual_seed(seed)
    m = torch.exp(2.5 * torch.randn(rows, nKb, generator=g))
    return (m / m.sum(1, keepdim=True)).reshape(1, 1, rows, nKb)


@pytest.mark.parametrize("rows", [1, 7, 8, 9, 15, 16, 17, 64, 65, 128, 129, 255, 256, 257])
@pytest.mark.parametrize("nKb", [1, 4, 32, 33, 128, 129, 256, 257, 512, 513, 1024, 1025])
def test_row_counts_around_the_cluster(rows, nKb):
    losa = lib()
    m = masses(rows, nKb, rows + nKb)
    offsets, idx = losa.losa_select(m.cuda(), 0.9)
    ref = orc.select(m.reshape(rows, nKb).numpy().astype(np.float64), 0.9)
    assert np.array_equal(offsets.cpu().numpy(), ref.offsets)
    assert np.array_equal(idx.cpu().numpy()[:ref.offsets[-1]], ref.kv_idx)
    k = (2 * nKb + 2) // 3
    offsets, idx = losa.losa_select_topk(m.cuda(), k)
    assert offsets.tolist() == [k * i for i in range(rows + 1)]
    order = torch.sort(m.reshape(rows, nKb), dim=1, descending=True, stable=True)[1][:, :k]
    assert torch.equal(idx.cpu().reshape(rows, k).long(), order.sort(1)[0])
    assert losa.losa_async_status() == 0


def test_a_capacity_that_is_too_small_and_masses_that_are_none():
    losa = lib()
    m = masses(40, 64, 7).cuda()
    offsets, idx = losa.losa_select(m, 0.9)
    n = int(offsets[-1])
    out = (torch.zeros(41, dtype=torch.int32, device="cuda"), torch.full((n,), -1, dtype=torch.int32, device="cuda"))
    losa.losa_select(m, 0.9, kv_capacity=n - 5, out=out)
    assert losa.losa_status_string(losa.losa_async_status()) == "LOSA_ERR_CAPACITY"
    assert torch.equal(out[0], offsets) and torch.equal(out[1][:n - 5], idx[:n - 5]) and (out[1][n - 5:] == -1).all()
    m[0, 0, 3, 5] = float("nan")
    m[0, 0, 39, 0] = -1.0
    offsets2, idx2 = losa.losa_select(m, 0.9)
    assert losa.losa_status_string(losa.losa_async_status()) == "LOSA_ERR_BAD_MASS"
    a, b = offsets.tolist(), offsets2.tolist()
    for r in set(range(40)) - {3, 39}:  # the other rows are untouched
        assert torch.equal(idx[a[r]:a[r + 1]], idx2[b[r]:b[r + 1]])


@pytest.mark.parametrize("rows,nKb", [(8, 256), (64, 1024), (128, 512), (256, 128), (65, 1024), (129, 130)])
def test_thresholds_among_many_close_masses(rows, nKb):
    """Masses within a few per cent of each other, of which half are kept: the threshold's bin holds most of the row, so
    that its list is long and split again.  The last two by the general way."""
    losa = lib()
    g = torch.Generator("cpu").manual_seed(rows + nKb)
    m = torch.exp(0.01 * torch.randn(rows, nKb, generator=g))
    m = (m / m.sum(1, keepdim=True)).reshape(1, 1, rows, nKb)
    offsets, idx = losa.losa_select(m.cuda(), 0.5)
    ref = orc.select(m.reshape(rows, nKb).numpy().astype(np.float64), 0.5)
    assert np.array_equal(offsets.cpu().numpy(), ref.offsets)
    assert np.array_equal(idx.cpu().numpy()[:ref.offsets[-1]], ref.kv_idx)
    k = nKb // 2
    offsets, idx = losa.losa_select_topk(m.cuda(), k)
    order = torch.sort(m.reshape(rows, nKb), dim=1, descending=True, stable=True)[1][:, :k]
    assert torch.equal(idx.cpu().reshape(rows, k).long(), order.sort(1)[0])
    assert losa.losa_async_status() == 0


@pytest.mark.parametrize("nKb", [2, 8, 31, 32, 33])
@pytest.mark.parametrize("tau", [1e-7, 0.25, 0.5, 0.515625, 1.0])
def test_ties_zeros_and_sums_that_just_reach_tau(nKb, tau):
    """Masses in units of 2^-6, many of them equal or zero, some rows adding up to less than tau: whole in every arithmetic."""
    losa = lib()
    rng = np.random.default_rng(nKb)
    m = rng.integers(0, 4, (20, nKb)).astype(np.float64)
    m[0], m[1], m[2] = 0.0, 1.0, 0.0
    m[2, nKb // 2] = 64.0
    for r in range(3, 20):
        m[r, rng.integers(nKb)] += max(0.0, 64.0 - m[r].sum()) if r < 17 else 0.0
    m /= 64.0
    offsets, idx = losa.losa_select(torch.from_numpy(m).float().reshape(1, 1, 20, nKb).cuda(), tau)
    ref = orc.select(m, tau)
    assert np.array_equal(offsets.cpu().numpy(), ref.offsets)
    assert np.array_equal(idx.cpu().numpy()[:ref.offsets[-1]], ref.kv_idx)
    assert losa.losa_async_status() == 0

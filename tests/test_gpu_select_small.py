"""Selection of few rows by one cluster, and of one row more by the general way: both against the oracle's rule, over row
counts around a warp's, a CTA's and the cluster's, with a capacity that is too small and with masses that are none."""
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


@pytest.mark.parametrize("rows", [1, 15, 16, 17, 128, 129, 255, 256, 257])
@pytest.mark.parametrize("nKb", [1, 33, 256, 257, 1024])
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

"""Items that a single wave is cut into: their parts run in one cluster and are merged through its CTAs' shared memory
(or, where the device does not hold all these clusters at once, by a launch behind: 10 items), from two parts to as many as
there can be, of an odd number of query tiles with a short last one; some parts outgrow their reference and are run again,
the others of their cluster wait for them.  Against the fp64 oracle."""
import numpy as np
import pytest
import torch

from oracle import losa_oracle as orc
from tests import util
from tests.test_gpu_units import check, lib, problem

pytestmark = pytest.mark.gpu

N = 1100  # 9 query tiles, of 5 items to a head; 9 K/V tiles


@pytest.mark.parametrize("D,R,C", [(64, 64, 64), (64, 128, 32), (128, 128, 128), (128, 64, 64)])
@pytest.mark.parametrize("H", [1, 2, 3, 4, 7])
def test_parts_of_an_item_are_merged_in_their_cluster(D, R, C, H):
    losa = lib()
    prob = losa.make_problem(torch.empty((1, H, N, D), dtype=torch.bfloat16, device="cuda"), R, C)
    assert 2 <= losa.losa_work_slots(losa.binding.LOSA_OP_ATTN, prob) // (5 * H)
    check(H, N, D, R, C, (0, H - 1), 1700 + H)


@pytest.mark.parametrize("D,R,C", [(64, 64, 64), (128, 128, 64)])
def test_cut_items_of_a_batched_call_and_of_token_major_tensors(D, R, C):
    """Two layers of two heads in one wave equal the single calls where both are cut alike; rows a head apart, a batch of
    two, bf16 and fp32 output (the same, rounded once)."""
    losa = lib()
    nQb, nKb = -(-N // R), -(-N // C)
    layers = []
    for i in range(2):
        q, k, v = (util.rand_bf16((2, N, 1, D), 1720 + 3 * i + j).cuda().transpose(1, 2) for j in range(3))
        off, idx = util.random_csr(2 * nQb, nKb, 1730 + i, 0.6)
        layers.append((q, k, v, torch.from_numpy(off).cuda(), torch.from_numpy(idx).cuda()))
    outs = losa.losa_sparse_attn_batched(layers, R, C, out_dtype=torch.float32)
    for (q, k, v, off, idx), o in zip(layers, outs):
        single = losa.losa_sparse_attn(q, k, v, off, idx, R, C, out_dtype=torch.float32)
        assert torch.equal(single.bfloat16(), losa.losa_sparse_attn(q, k, v, off, idx, R, C))
        # 10 items in 7 parts, 20 in 3: P rounds against another reference, 2^-9 each at random
        assert (o - single).norm() <= 4e-3 * single.norm()
    assert losa.losa_async_status() == 0


@pytest.mark.parametrize("D,R,C", [(64, 64, 64), (64, 128, 32), (128, 128, 128), (128, 64, 64)])
@pytest.mark.parametrize("H", [1, 2])
def test_parts_that_list_nothing(D, R, C, H):
    """Lists of one to three key blocks cut into eight parts (5 items, in clusters) or seven (10 items at D = 128 and 64,
    merged by a launch behind): most units have no K/V tile and end as soon as their query tile is there, and others
    list blocks of one of their query blocks only, so that the other's rows have no weight in that part."""
    losa = lib()
    nQb, nKb = -(-N // R), -(-N // C)
    q, k, v = (util.rand_bf16((1, H, N, D), 1740 + i) for i in range(3))
    rng = np.random.default_rng(1750 + H)
    rows = [np.sort(rng.choice(nKb, rng.integers(1, 4), replace=False)) for _ in range(H * nQb)]
    off = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int32)
    idx = np.concatenate(rows).astype(np.int32)
    args = [x.cuda() for x in (q, k, v, torch.from_numpy(off), torch.from_numpy(idx))]
    outs = [losa.losa_sparse_attn(*args, R, C, out_dtype=torch.float32) for _ in range(20)]
    assert losa.losa_async_status() == 0
    want = orc.blocks_to_tokens(orc.sparse_attn(*(util.to_np(x) for x in (q, k, v)), R, C, off, idx), 1, H, N)
    util.assert_output_close(outs[0], want, "short lists")
    assert all(torch.equal(outs[0], o) for o in outs[1:])


@pytest.mark.parametrize("D,R,C", [(64, 64, 64), (64, 128, 32), (128, 128, 128), (128, 64, 64)])
@pytest.mark.parametrize("H", [1, 2])
def test_a_unit_whose_two_query_tiles_are_run_again_counts_once(D, R, C, H):
    """One row of each query tile of an item meets its far key in the second K/V tile of the item's last part, in every head;
    merged in clusters (5 items) and by a launch behind (10)."""
    losa = lib()
    q, k, v = problem(H, N, D, 1760, range(H))
    q[0, :, 128 + 7] = q[0, :, 7]
    prob = losa.make_problem(q.cuda(), R, C)
    for fill in (0, 255):  # whatever the workspace held before
        ws = torch.full((losa.losa_workspace_bytes(losa.binding.LOSA_OP_ATTN, prob),), fill, dtype=torch.uint8, device="cuda")
        o = losa.losa_attn(q.cuda(), k.cuda(), v.cuda(), R, C, out_dtype=torch.float32, ws=ws)
        assert losa.losa_async_status() == 0
        assert util.units_run_again(losa, ws, prob) == H
        util.assert_output_close(o, orc.dense_attn(*(util.to_np(x) for x in (q, k, v))), "two tiles again")

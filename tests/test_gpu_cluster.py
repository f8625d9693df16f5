"""Items that a single wave is cut into: their parts run in one cluster and are merged through its CTAs' shared memory, or,
where the device does not hold all these clusters at once, by a launch behind (the library says how many kernels a call
takes): from two parts to as many as there can be, of an odd number of query tiles with a short last one, and parts that
outgrow their reference and are run again while the others of their cluster wait for them.  Against the fp64 oracle."""
import numpy as np
import pytest
import torch

from oracle import losa_oracle as orc
from tests import util
from tests.test_gpu_units import check, lib, problem

pytestmark = pytest.mark.gpu

N = 1100  # 9 query tiles, of 5 items to a head; 9 K/V tiles


def merged_in_cluster(losa, prob, op):
    """Of a call that is one wave and cut: whether it takes one kernel or a second one that merges."""
    launches = losa.losa_kernel_launches(op, prob)
    assert launches in (1, 2)
    return launches == 1


# 5, 10, 15, 20 and 35 items in 8, 7, 4, 3 and 2 parts.  Of the first a B200 holds more clusters than there are, of the second
# (14 CTAs, or 7) fewer whichever of its SMs are there; the others fit on some.
@pytest.mark.parametrize("D,R,C", [(64, 64, 64), (64, 128, 32), (128, 128, 128), (128, 64, 64)])
@pytest.mark.parametrize("H,clusters", [(1, True), (2, False), (3, None), (4, None), (7, None)])
def test_parts_of_an_item_are_merged_in_their_cluster(D, R, C, H, clusters):
    """Heads whose first query block has a row that meets a far key in the last part only, which is run again."""
    losa = lib()
    prob = losa.make_problem(torch.empty((1, H, N, D), dtype=torch.bfloat16, device="cuda"), R, C)
    assert 2 <= losa.losa_work_slots(losa.binding.LOSA_OP_ATTN, prob) // (5 * H)
    for op in (losa.binding.LOSA_OP_ATTN, losa.binding.LOSA_OP_SPARSE_ATTN):
        assert clusters is None or merged_in_cluster(losa, prob, op) == clusters
    check(H, N, D, R, C, (0, H - 1), 1700 + H, again=len({0, H - 1}))


@pytest.mark.parametrize("D,R,C", [(64, 64, 64), (128, 128, 64)])
@pytest.mark.parametrize("layers,B,H", [(2, 2, 1), (2, 1, 2), (3, 1, 1)])
def test_cut_items_of_a_batched_call_and_of_token_major_tensors(D, R, C, layers, B, H):
    """20 or 15 items of all the layers together in one wave, rows a head apart: against the oracle, in bf16 the fp32 output
    rounded once, and bit for bit what one call on all the layers as one batch gives, which is cut alike."""
    losa = lib()
    nQb, nKb = -(-N // R), -(-N // C)
    args, want = [], []
    for i in range(layers):
        q, k, v = (util.rand_bf16((B, N, H, D), 1720 + 3 * i + j).transpose(1, 2) for j in range(3))
        off, idx = util.random_csr(B * H * nQb, nKb, 1730 + i, 0.6)
        want.append(orc.blocks_to_tokens(orc.sparse_attn(*(util.to_np(x) for x in (q, k, v)), R, C, off, idx), B, H, N))
        args.append((*(x.cuda() for x in (q, k, v)), torch.from_numpy(off).cuda(), torch.from_numpy(idx).cuda()))
    outs = losa.losa_sparse_attn_batched(args, R, C, out_dtype=torch.float32)
    low = losa.losa_sparse_attn_batched(args, R, C)
    assert losa.losa_async_status() == 0
    for o, ref in zip(outs, want):
        util.assert_output_close(o, ref, "batched")
    assert all(torch.equal(o.bfloat16(), x) for o, x in zip(outs, low))
    q, k, v = (torch.cat([a[j] for a in args]) for j in range(3))
    off = torch.cat([torch.zeros(1, dtype=torch.int32, device="cuda")] + [a[3].diff() for a in args]).cumsum(0).int()
    one = losa.losa_sparse_attn(q, k, v, off, torch.cat([a[4] for a in args]), R, C, out_dtype=torch.float32)
    assert torch.equal(torch.cat(outs), one)


@pytest.mark.parametrize("D,R,C", [(64, 64, 64), (64, 128, 32), (128, 128, 128), (128, 64, 64)])
@pytest.mark.parametrize("H", [1, 2])
def test_parts_that_list_nothing(D, R, C, H):
    """Lists of one to three key blocks cut into eight parts (5 items, in clusters) or seven (10 items at D = 128 and 64,
    merged by a launch behind): most units have no K/V tile and end as soon as their query tile is there, and others
    list blocks of one of their query blocks only, so that the other's rows have no weight in that part."""
    losa = lib()
    nQb, nKb = -(-N // R), -(-N // C)
    q, k, v = (util.rand_bf16((1, H, N, D), 1740 + i) for i in range(3))
    assert merged_in_cluster(losa, losa.make_problem(q.cuda(), R, C), losa.binding.LOSA_OP_SPARSE_ATTN) == (H == 1)
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
    assert merged_in_cluster(losa, prob, losa.binding.LOSA_OP_ATTN) == (H == 1)
    for fill in (0, 255):  # whatever the workspace held before
        ws = torch.full((losa.losa_workspace_bytes(losa.binding.LOSA_OP_ATTN, prob),), fill, dtype=torch.uint8, device="cuda")
        o = losa.losa_attn(q.cuda(), k.cuda(), v.cuda(), R, C, out_dtype=torch.float32, ws=ws)
        assert losa.losa_async_status() == 0
        assert util.units_run_again(losa, ws, prob) == H
        util.assert_output_close(o, orc.dense_attn(*(util.to_np(x) for x in (q, k, v))), "two tiles again")

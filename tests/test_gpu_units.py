"""Work units around the number of work slots: a call with no more units than slots prepares nothing (each slot takes
the unit at its position and makes its own list), one with more draws them; and the shortest units that a last wave
is cut into.  Some rows outgrow their reference, in the first unit, the last and one in between, so that units are
run again next to others.  Against the fp64 oracle."""
import numpy as np
import pytest
import torch

from oracle import losa_oracle as orc
from tests import util

pytestmark = pytest.mark.gpu


def lib():
    import paper_2608_12032_b200 as losa
    return losa


def problem(H, N, D, seed, heads):
    g = torch.Generator("cpu").manual_seed(seed)
    q, k, v = (torch.randn(1, H, N, D, generator=g) for _ in range(3))
    far = torch.zeros(D)
    far[3] = (120.0 * D ** 0.5) ** 0.5  # a score of 120 with itself, of a few with the other rows
    for h in heads:
        q[0, h, 7] = far
        k[0, h, N - 2] = far
    return tuple(x.bfloat16() for x in (q, k, v))


def check(H, N, D, R, C, heads, seed, again=None):
    """again: how many units of the dense call are run again (None: not counted, in one uncut wave)"""
    losa = lib()
    q, k, v = problem(H, N, D, seed, heads)
    qd, kd, vd = q.cuda(), k.cuda(), v.cuda()
    qn, kn, vn = (util.to_np(x) for x in (q, k, v))
    nQb, nKb = -(-N // R), -(-N // C)
    off, idx = util.random_csr(H * nQb, nKb, seed, 0.6)
    prob = losa.make_problem(qd, R, C)
    ws = torch.empty(losa.losa_workspace_bytes(losa.binding.LOSA_OP_ATTN, prob), dtype=torch.uint8, device="cuda")
    o = losa.losa_attn(qd, kd, vd, R, C, out_dtype=torch.float32, ws=ws)
    if again is not None:
        assert util.units_run_again(losa, ws, prob) == again
    o_s = losa.losa_sparse_attn(qd, kd, vd, torch.from_numpy(off).cuda(), torch.from_numpy(idx).cuda(), R, C,
                                out_dtype=torch.float32)
    mass = losa.losa_block_mass(qd, kd, R, C)
    o_f, mass_f = losa.losa_attn_mass(qd, kd, vd, R, C, out_dtype=torch.float32)
    assert losa.losa_async_status() == 0
    ref, ref_m = orc.dense_attn(qn, kn, vn), orc.block_mass(qn, kn, R, C)
    util.assert_output_close(o, ref, "dense")
    util.assert_output_close(o_f, ref, "fused")
    util.assert_output_close(
        o_s, orc.blocks_to_tokens(orc.sparse_attn(qn, kn, vn, R, C, off, idx), 1, H, N), "sparse")
    for m in (mass, mass_f):
        assert np.abs(m.cpu().numpy().reshape(ref_m.shape) - ref_m).max() <= util.MASS_TOL


@pytest.mark.parametrize("D,R,C", [(64, 64, 64), (64, 128, 32), (128, 128, 128), (128, 64, 64)])
@pytest.mark.parametrize("more", [-1, 0, 1])
def test_as_many_units_as_slots_and_one_more_or_less(D, R, C, more):
    losa = lib()
    prob = losa.make_problem(torch.empty((1, 1, 256, D), dtype=torch.bfloat16, device="cuda"), R, C)
    H = losa.losa_work_slots(losa.binding.LOSA_OP_ATTN, prob) + more  # one pair of query tiles per head
    # (of one more than slots the last is cut into parts of one K/V tile, which takes its reference from all its keys)
    check(H, 250, D, R, C, (0, H // 2, H - 1), 1200 + more, again=2 if more > 0 else None)


@pytest.mark.parametrize("D,R,C", [(64, 64, 64), (64, 128, 128), (128, 128, 32), (128, 64, 64)])
@pytest.mark.parametrize("tiles", [2, 9])
def test_short_items_cut_into_as_many_parts_as_there_can_be(D, R, C, tiles):
    """One item of one head in parts of one key block, which never outgrow their reference; five in parts of two K/V
    tiles at most, of which the first query block's last part meets its far key in the second and is run again."""
    check(1, 128 * tiles - 30, D, R, C, (0,), 1300 + tiles, again=1 if tiles == 9 else 0)


@pytest.mark.parametrize("D,R,C", [(64, 64, 64), (64, 128, 32), (128, 128, 128), (128, 64, 64)])
def test_units_run_again_with_and_without_their_maxima(D, R, C):
    """Keys 60 nats above the first tile leave finite row sums, which the unit's rows are run again against; keys 150
    nats above do not, and their maxima are taken first.  Both, and units that are not run again, in turn and several of
    a kind behind one another, more than one to a work slot."""
    losa = lib()
    H, N = 2 * losa.losa_work_slots(losa.binding.LOSA_OP_ATTN, losa.make_problem(
        torch.empty((1, 1, 256, D), dtype=torch.bfloat16, device="cuda"), R, C)) + 40, 250
    g = torch.Generator("cpu").manual_seed(1600)
    q = torch.randn(1, H, N, D, generator=g) * 0.3 + 1.0
    k = torch.randn(1, H, N, D, generator=g) * 0.3
    v = torch.randn(1, H, N, D, generator=g)
    nats = torch.tensor([0.0, 60.0, 60.0, 150.0, 60.0, 150.0, 150.0])[torch.arange(H) * 5 // 3 % 7]
    k[0, :, 140:] += (nats * D ** 0.5 / D)[:, None, None]
    q, k, v = q.bfloat16(), k.bfloat16(), v.bfloat16()
    qd, kd, vd = q.cuda(), k.cuda(), v.cuda()
    qn, kn, vn = (util.to_np(x) for x in (q, k, v))
    ref, ref_m = orc.dense_attn(qn, kn, vn), orc.block_mass(qn, kn, R, C)
    off, idx = util.all_blocks_csr(H * -(-N // R), -(-N // C))
    o = losa.losa_attn(qd, kd, vd, R, C, out_dtype=torch.float32)
    o_s = losa.losa_sparse_attn(qd, kd, vd, torch.from_numpy(off).cuda(), torch.from_numpy(idx).cuda(), R, C,
                                out_dtype=torch.float32)
    mass, lse = losa.losa_block_mass(qd, kd, R, C, return_lse=True)
    o_f, mass_f, lse_f = losa.losa_attn_mass(qd, kd, vd, R, C, return_lse=True, out_dtype=torch.float32)
    assert losa.losa_async_status() == 0
    for name, x in (("dense", o), ("sparse", o_s), ("fused", o_f)):
        util.assert_output_close(x, ref, name)
    for m in (mass, mass_f):
        assert np.abs(m.cpu().numpy().reshape(ref_m.shape) - ref_m).max() <= util.MASS_TOL
    want = torch.logsumexp(q[0].double() @ k[0].double().transpose(1, 2) / D ** 0.5, -1)
    for x in (lse, lse_f):
        assert (x[0].cpu().double() - want).abs().max() <= 1e-4  # 150 + 64 sums in fp32: 150 * 2^-23 each


@pytest.mark.parametrize("H", [2, 80])
@pytest.mark.parametrize("sparse", [False, True])
def test_captured_behind_a_memset_and_behind_another_stream(H, sparse):
    """The first launch of a call is a dependent of whatever is ahead of it in the stream: a kernel, a memset, a copy
    and the join with another stream, in a captured graph as well."""
    losa = lib()
    N, blk = 250, 64
    q, k, v = (x.cuda() for x in problem(H, N, 64, 1400, (0,)))
    nb = -(-N // blk)
    csr = tuple(torch.from_numpy(x).cuda() for x in util.random_csr(H * nb, nb, 1401, 0.6)) if sparse else ()
    call = losa.losa_sparse_attn if sparse else losa.losa_attn
    op = losa.binding.LOSA_OP_SPARSE_ATTN if sparse else losa.binding.LOSA_OP_ATTN
    prob = losa.make_problem(q, blk, blk)
    assert (H > losa.losa_work_slots(op, prob)) == (H == 80)  # 80: a launch ahead of the kernel prepares the units
    want = call(q, k, v, *csr, blk, blk)
    outs = [torch.full_like(want, 7.0) for _ in range(3)]
    q2, v2 = torch.empty_like(q), v.clone()
    ws = torch.empty(losa.losa_workspace_bytes(op, prob), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph):
        q2.zero_()
        v2.zero_()  # directly ahead of the call that reads it: o is 0
        call(q, k, v2, *csr, blk, blk, out=outs[0], ws=ws)
        v2.copy_(v)
        call(q, k, v2, *csr, blk, blk, out=outs[1], ws=ws)
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            q2.copy_(q)
        torch.cuda.current_stream().wait_stream(side)
        call(q2, k, v, *csr, blk, blk, out=outs[2], ws=ws)
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    assert losa.losa_async_status() == 0
    assert not outs[0].any() and torch.equal(outs[1], want) and torch.equal(outs[2], want)

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
        k[0, h, N - 5] = far
    return tuple(x.bfloat16() for x in (q, k, v))


def check(H, N, D, R, C, heads, seed):
    losa = lib()
    q, k, v = problem(H, N, D, seed, heads)
    qd, kd, vd = q.cuda(), k.cuda(), v.cuda()
    qn, kn, vn = (util.to_np(x) for x in (q, k, v))
    nQb, nKb = -(-N // R), -(-N // C)
    off, idx = util.random_csr(H * nQb, nKb, seed, 0.6)
    o = losa.losa_attn(qd, kd, vd, R, C, out_dtype=torch.float32)
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
    check(H, 250, D, R, C, (0, H // 2, H - 1), 1200 + more)


@pytest.mark.parametrize("D,R,C", [(64, 64, 64), (64, 128, 128), (128, 128, 32), (128, 64, 64)])
@pytest.mark.parametrize("tiles", [2, 9])
def test_short_items_cut_into_as_many_parts_as_there_can_be(D, R, C, tiles):
    """One or five items of one head: parts of one K/V tile or less, made, run, run again and merged."""
    check(1, 128 * tiles - 30, D, R, C, (0,), 1300 + tiles)


def test_captured_behind_a_memset_and_behind_another_stream():
    """The first launch of a call is a dependent of whatever is ahead of it in the stream: a kernel, a memset, a copy
    and the join with another stream, in a captured graph as well."""
    losa = lib()
    q, k, v = (x.cuda() for x in problem(2, 700, 64, 1400, (0,)))
    want = losa.losa_attn(q, k, v, 64, 64)
    o, q2 = torch.empty_like(want), torch.empty_like(q)
    ws = torch.empty(losa.losa_workspace_bytes(losa.binding.LOSA_OP_ATTN, losa.make_problem(q, 64, 64)), dtype=torch.uint8,
                     device="cuda")
    torch.cuda.synchronize()
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph):
        o.zero_()
        losa.losa_attn(q, k, v, 64, 64, out=o, ws=ws)
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            q2.zero_()
            q2.copy_(q)
        torch.cuda.current_stream().wait_stream(side)
        losa.losa_attn(q2, k, v, 64, 64, out=o, ws=ws)
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    assert losa.losa_async_status() == 0
    assert torch.equal(o, want)

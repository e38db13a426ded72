"""GPU parity of the hard layer and its popcount head on rows of any number
of words (bit-exact): word counts around the 32-word lane groups, the
128-word stages and the three-stage chunks of the staged kernels, with and
without a partial last word, at every fan-in, and rows that start off a
16-byte boundary."""
import os

import numpy as np
import pytest
import torch

import oracle
import paper_2602_07400_gb300 as bl
from paper_2602_07400_gb300 import synth
from parity_util import check_exact

pytestmark = pytest.mark.gpu

oracle.set_threads(os.cpu_count() or 1)


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _case(W, tail, k, w_in, w, C, offset=0):
    N = 32 * W - tail
    xp = synth.random_words(w_in, W, seed=W + k)
    if tail:
        xp[:, -1] &= np.uint32((1 << (32 - tail)) - 1)
    conn = synth.connectivity(w, k, w_in, seed=2)
    table = synth.random_tables(w, seed=3)
    if k < 6:
        table &= np.uint64((1 << (1 << k)) - 1)
    buf = torch.zeros(w_in * W + 8, dtype=torch.int32, device="cuda")
    x = buf[offset:offset + w_in * W].view(w_in, W)
    x.copy_(dev(xp.view(np.int32)))
    yp = torch.full((w, W), -1, dtype=torch.int32, device="cuda")
    tab = dev(table.view(np.int64))
    bl.bitlogic_hard_forward(x, N, dev(conn), tab, yp=yp)
    want = oracle.hard_forward(xp, N, conn, table)
    check_exact(yp.cpu().numpy().view(np.uint32), want, "words")
    yp2 = torch.full((w, W), -1, dtype=torch.int32, device="cuda")
    counts = torch.full((N, C), -1, dtype=torch.int32, device="cuda")
    pred = torch.full((N,), -1, dtype=torch.int32, device="cuda")
    bl.bitlogic_hard_forward(x, N, dev(conn), tab, yp=yp2, C=C, counts=counts, pred=pred)
    wc, wp = oracle.popcount_head(want, N, C)
    check_exact(yp2.cpu().numpy().view(np.uint32), want, "words (head)")
    check_exact(counts.cpu().numpy(), wc, "counts")
    check_exact(pred.cpu().numpy(), wp, "pred")
    assert bl.bitlogic_device_error() == 0


@pytest.mark.parametrize("W", [1, 31, 33, 63, 65, 97, 127, 129, 255, 313, 383, 385, 513, 769])
@pytest.mark.parametrize("k,tail", [(6, 0), (6, 17), (4, 31)])
def test_any_word_count(W, k, tail):
    _case(W, tail, k, 50, 180, 6)


@pytest.mark.parametrize("k", [1, 2, 3, 5])
def test_every_fan_in(k):
    _case(193, 5, k, 40, 90, 9)


@pytest.mark.parametrize("W,offset", [(132, 1), (384, 3), (4, 2)])
def test_rows_off_a_16_byte_boundary(W, offset):
    # a multiple of four words per row whose first row is not 16-byte aligned
    _case(W, 3, 6, 30, 64, 4, offset)


def test_large_groups_and_few_classes():
    # more nodes per class than one block's slice: several splits
    _case(161, 9, 6, 200, 3000, 2)


def _node_words(x, table):
    """Output words of one fan-in-2 node on the words x [2, W] (device int32)."""
    a, b = x[0], x[1]
    corner = [~a & ~b, a & ~b, ~a & b, a & b]
    out = torch.zeros_like(a)
    for i in range(4):
        if table >> i & 1:
            out |= corner[i]
    return out


@pytest.mark.parametrize("W,head", [(65535 * 128 + 1, True), (65535 * 384 + 1, False)])
def test_rows_of_more_stages_than_grid_y_holds(W, head):
    # no multiple of four words, and longer than the staged kernels' grids take
    N = 32 * W - 5
    g = torch.Generator(device="cuda").manual_seed(W)
    x = torch.randint(-2 ** 31, 2 ** 31, (2, W), generator=g, device="cuda", dtype=torch.int64).to(torch.int32)
    x[:, -1] &= (1 << 27) - 1
    conn, tables = np.array([[0, 1], [1, 0], [0, 1]], np.int32), [0b0110, 0b1011, 0b0001]
    want = torch.stack([_node_words(x[c], t) for c, t in zip(conn.tolist(), tables)])
    want[:, -1] &= (1 << 27) - 1
    yp = torch.full((3, W), -1, dtype=torch.int32, device="cuda")
    kw = {}
    if head:
        kw = dict(C=1, counts=torch.full((N, 1), -1, dtype=torch.int32, device="cuda"))
    bl.bitlogic_hard_forward(x, N, dev(conn), dev(np.array(tables, np.int64)), yp=yp, **kw)
    assert torch.equal(yp, want)
    if head:
        bit = torch.arange(32, device="cuda", dtype=torch.int32)
        for w0 in range(0, W, 1 << 20):
            part = want[:, w0:w0 + (1 << 20)]
            count = sum((row[:, None] >> bit & 1) for row in part).reshape(-1)
            got = kw["counts"][32 * w0:32 * w0 + count.numel(), 0]
            assert torch.equal(got, count[:got.numel()])
    assert bl.bitlogic_device_error() == 0

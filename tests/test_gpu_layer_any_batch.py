"""GPU parity of the fp32 layer kernels on batches that are no multiple of
four and on rows off a 16-byte boundary: forward, backward with per-edge
terms (from rows and from upstream terms, at given positions) and the CSR
reduction, around the 32- and 128-sample edges of their stages, and the head's group sums likewise."""
import os

import numpy as np
import pytest
import torch

import oracle
import paper_2602_07400_gb300 as bl
from paper_2602_07400_gb300 import synth
from parity_util import check_exact, check_fwd, check_grad

pytestmark = pytest.mark.gpu

oracle.set_threads(os.cpu_count() or 1)


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def off_boundary(a, offset):
    """The rows of a on the device, starting `offset` floats past an aligned address."""
    buf = torch.empty(a.size + 8, device="cuda")
    t = buf[offset:offset + a.size].view(a.shape)
    t.copy_(dev(a))
    return t


@pytest.mark.parametrize("k", [3, 4, 5, 6])
@pytest.mark.parametrize("B,offset", [(1, 0), (31, 0), (33, 0), (127, 0), (129, 0), (258, 0), (515, 0), (1030, 0), (128, 1), (260, 3)])
@pytest.mark.parametrize("node", ["soft", "st"])
def test_layer_on_any_batch(k, B, offset, node):
    w_in, w = 40, 70
    X = synth.uniform_activations(w_in, B, seed=B)
    conn = synth.connectivity(w, k, w_in, seed=1)
    theta = synth.table_logits(w, 1 << k, seed=2)
    dY = synth.uniform_gradients(w // 2, B, seed=3, scale=1e-2)
    Xd, dYd = off_boundary(X, offset), off_boundary(dY, offset)
    off, edge = bl.bitlogic_build_csr(conn, w_in)
    pos = bl.bitlogic_csr_positions(edge)
    Y = torch.full((w, B), np.nan, device="cuda")
    bl.bitlogic_lut_forward_node(Xd, dev(conn), dev(theta), Y, node)
    X64 = X.astype(np.float64)
    check_fwd(Y, oracle.lut_forward(X64, conn, theta, node), "y", atol=1e-6 if node == "st" else 0.0)
    dth = torch.full((w, 1 << k), np.nan, device="cuda")
    P = torch.full((w * k, B), np.nan, device="cuda")
    out = torch.full((w, B), np.nan, device="cuda")
    bl.bitlogic_lut_backward_node(Xd, dev(conn), dev(theta), dth, node, dY=dYd, dy_group=2, edge_terms=P,
                                  edge_pos=dev(pos), dY_out=out)
    dX = torch.full((w_in, B), np.nan, device="cuda")
    bl.bitlogic_csr_reduce(P, dev(off), None, dX)
    full = np.repeat(dY, 2, axis=0)
    check_exact(out.cpu().numpy(), full, "gradient used")
    wth, wdx = oracle.lut_backward(X64, conn, theta, full.astype(np.float64), want_dx=True, node=node)
    check_grad(dth, wth, "dtheta")
    check_grad(dX, wdx, "dX")
    # the gradient as one upstream term row per node: the same sums
    dth_t, P_t = torch.empty_like(dth), torch.full_like(P, np.nan)
    bl.bitlogic_lut_backward_node(Xd, dev(conn), dev(theta), dth_t, node, up_terms=dev(full),
                                  up_off=dev(np.arange(w + 1, dtype=np.int32)), edge_terms=P_t, edge_pos=dev(pos))
    check_exact(dth_t.cpu().numpy(), dth.cpu().numpy(), "dtheta from terms")
    check_exact(P_t.cpu().numpy(), P.cpu().numpy(), "edge terms from terms")
    assert bl.bitlogic_device_error() == 0


@pytest.mark.parametrize("C,g,B,offset", [(10, 64, 1, 0), (10, 129, 127, 0), (1, 257, 131, 0), (10, 513, 158, 0),
                                          (100, 90, 907, 0), (3, 1025, 256, 1)])
def test_head_on_any_batch(C, g, B, offset):
    rng = np.random.default_rng(C + B)
    Y = rng.random((C * g, B)).astype(np.float32)
    labels = rng.integers(0, C, size=B).astype(np.int32)
    loss = torch.zeros(1, device="cuda")
    logits = torch.full((B, C), np.nan, device="cuda")
    dY = torch.full((C * g, B), np.nan, device="cuda")
    ws = torch.empty(bl.bitlogic_head_loss_workspace(B, C), dtype=torch.uint8, device="cuda")
    bl.bitlogic_head_loss(off_boundary(Y, offset), dev(labels), C, 20.0, loss, ws, logits=logits, dY=dY)
    wl, wloss, wdy = oracle.head_loss(Y.astype(np.float64), labels, C, 20.0)
    check_fwd(logits, wl, "logits")
    check_fwd(loss, np.array([wloss]), "loss")
    check_grad(dY, wdy, "dY")
    assert bl.bitlogic_device_error() == 0


@pytest.mark.parametrize("w_in,deg", [(1, 32), (3, 63), (7, 500), (900, 33)])
@pytest.mark.parametrize("B,offset", [(1, 0), (4, 0), (130, 0), (256, 0), (300, 1), (515, 0)])
def test_csr_reduce_of_few_rows(w_in, deg, B, offset):
    # several warps per row: runs of unequal length, rows without a term
    rng = np.random.default_rng(w_in + deg + B)
    n = w_in * deg
    owner = np.sort(rng.integers(0, w_in, size=n))
    if w_in > 2:
        owner[owner == 1] = 0
    csr_off = np.searchsorted(owner, np.arange(w_in + 1)).astype(np.int32)
    P = rng.standard_normal((n, B), dtype=np.float32)
    total, size = np.zeros((w_in, B)), np.zeros((w_in, B))
    np.add.at(total, owner, P.astype(np.float64))
    np.add.at(size, owner, np.abs(P).astype(np.float64))
    perm = rng.permutation(n).astype(np.int32)
    shuffled = np.empty_like(P)
    shuffled[perm] = P
    outs = []
    for rows, edge in ((P, None), (shuffled, dev(perm))):
        dX = torch.full((w_in, B), np.nan, device="cuda")
        bl.bitlogic_csr_reduce(off_boundary(rows, offset), dev(csr_off), edge, dX)
        outs.append(dX.cpu().numpy())
    check_exact(outs[1], outs[0], "with an edge map")
    # fp32 sums of m terms: error below m 2^-24 of the terms' magnitudes
    m = np.diff(csr_off)[:, None] + 8
    assert np.all(np.abs(outs[0] - total) <= size * m * 2.0 ** -24)
    assert bl.bitlogic_device_error() == 0


@pytest.mark.parametrize("k,w", [(3, 5000), (4, 5200), (6, 3000)])
@pytest.mark.parametrize("B,offset", [(129, 0), (260, 0), (260, 1), (37, 0)])
def test_backward_over_several_nodes_per_block(k, w, B, offset):
    # more nodes than two waves of the persistent blocks: what a block carries
    # from one node to the next (ring slots, rows, logits, positions), for the
    # gradient from rows and summed from several upstream terms per node
    w_in = 300
    X = synth.uniform_activations(w_in, B, seed=B)
    conn = synth.connectivity(w, k, w_in, seed=1)
    theta = synth.table_logits(w, 1 << k, seed=2)
    Xd = off_boundary(X, offset)
    off, edge = bl.bitlogic_build_csr(conn, w_in)
    pos = bl.bitlogic_csr_positions(edge)
    rng = np.random.default_rng(k + B)
    # upstream terms: 0 to 4 per node, their rows in any order
    deg = rng.integers(0, 5, size=w)
    up_off = np.concatenate(([0], np.cumsum(deg))).astype(np.int32)
    n = int(up_off[-1])
    up_edge = rng.permutation(n).astype(np.int32)
    terms = synth.uniform_gradients(n, B, seed=4, scale=1e-2)
    summed = np.zeros((w, B))
    np.add.at(summed, np.repeat(np.arange(w), deg), terms[up_edge].astype(np.float64))
    dY = synth.uniform_gradients(w // 2, B, seed=3, scale=1e-2)
    sources = [(dict(dY=off_boundary(dY, offset), dy_group=2), np.repeat(dY, 2, axis=0).astype(np.float64)),
               (dict(up_terms=off_boundary(terms, offset), up_off=dev(up_off), up_edge=dev(up_edge)), summed)]
    for source, full in sources:
        dth = torch.full((w, 1 << k), np.nan, device="cuda")
        P = torch.full((w * k, B), np.nan, device="cuda")
        used = torch.full((w, B), np.nan, device="cuda")
        bl.bitlogic_lut_backward_node(Xd, dev(conn), dev(theta), dth, "soft", edge_terms=P, edge_pos=dev(pos),
                                      dY_out=used, **source)
        dX = torch.full((w_in, B), np.nan, device="cuda")
        bl.bitlogic_csr_reduce(P, dev(off), None, dX)
        wth, wdx = oracle.lut_backward(X.astype(np.float64), conn, theta, full, want_dx=True)
        # up to four fp32 terms of at most 0.06: three roundings of at most 2^-24 x 0.24
        check_fwd(used, full, "gradient used", atol=5e-8)
        check_grad(dth, wth, "dtheta")
        check_grad(dX, wdx, "dX")
    assert bl.bitlogic_device_error() == 0


@pytest.mark.parametrize("w_in,deg", [(1, 40), (7, 500), (60, 70), (900, 33), (3, 20)])
@pytest.mark.parametrize("B,offset", [(4, 0), (130, 0), (256, 0), (300, 1), (515, 0)])
def test_upstream_terms_are_the_csr_reduction_bit_for_bit(w_in, deg, B, offset):
    # the gradient that a layer sums from the next layer's terms is
    # bitlogic_csr_reduce of them, also where few rows have many terms
    rng = np.random.default_rng(w_in + deg + B)
    n = w_in * deg
    off = np.searchsorted(np.sort(rng.integers(0, w_in, size=n)), np.arange(w_in + 1)).astype(np.int32)
    terms = rng.standard_normal((n, B), dtype=np.float32)
    edge = rng.permutation(n).astype(np.int32)
    Pd = off_boundary(terms, offset)
    dX = torch.full((w_in, B), np.nan, device="cuda")
    bl.bitlogic_csr_reduce(Pd, dev(off), dev(edge), dX)
    X = synth.uniform_activations(8, B, seed=5)
    for k in (1, 2, 4):
        conn = synth.connectivity(w_in, k, 8, seed=6)
        theta = dev(synth.table_logits(w_in, 1 << k, seed=7))
        for terms_out in (None, torch.empty(w_in * k, B, device="cuda")):
            used = torch.full((w_in, B), np.nan, device="cuda")
            bl.bitlogic_lut_backward_node(dev(X), dev(conn), theta, torch.empty_like(theta), "soft", up_terms=Pd,
                                          up_off=dev(off), up_edge=dev(edge), edge_terms=terms_out, dY_out=used)
            check_exact(used.cpu().numpy(), dX.cpu().numpy(), "gradient used")
    assert bl.bitlogic_device_error() == 0


@pytest.mark.parametrize("k", [3, 4, 5, 6])
@pytest.mark.parametrize("B,offset", [(256, 0), (260, 0), (132, 1)])
@pytest.mark.parametrize("node", ["soft", "st"])
def test_upstream_terms_with_input_gradient(k, B, offset, node):
    # aligned and other rows, nodes without a term and with more than 32 (two
    # chunks of row ids): against the oracle, with and without given positions
    w_in, w = 40, 300
    X = synth.uniform_activations(w_in, B, seed=B)
    conn = synth.connectivity(w, k, w_in, seed=1)
    theta = synth.table_logits(w, 1 << k, seed=2)
    off, edge = bl.bitlogic_build_csr(conn, w_in)
    pos = bl.bitlogic_csr_positions(edge)
    rng = np.random.default_rng(k)
    deg = rng.integers(0, 6, size=w)
    deg[7], deg[-1] = 33, 70
    up_off = np.concatenate(([0], np.cumsum(deg))).astype(np.int32)
    n = int(up_off[-1])
    up_edge = rng.permutation(n).astype(np.int32)
    terms = synth.uniform_gradients(n, B, seed=4, scale=1e-2)
    full = np.zeros((w, B))
    np.add.at(full, np.repeat(np.arange(w), np.diff(up_off)), terms[up_edge].astype(np.float64))
    wth, wdx = oracle.lut_backward(X.astype(np.float64), conn, theta, full, want_dx=True, node=node)
    rows = []
    for epos, csr_edge in ((None, dev(edge)), (dev(pos), None)):
        dth, P = torch.full((w, 1 << k), np.nan, device="cuda"), torch.full((w * k, B), np.nan, device="cuda")
        bl.bitlogic_lut_backward_node(off_boundary(X, offset), dev(conn), dev(theta), dth, node,
                                      up_terms=off_boundary(terms, offset), up_off=dev(up_off), up_edge=dev(up_edge),
                                      edge_terms=P, edge_pos=epos)
        dX = torch.full((w_in, B), np.nan, device="cuda")
        bl.bitlogic_csr_reduce(P, dev(off), csr_edge, dX)
        check_grad(dth, wth, "dtheta")
        check_grad(dX, wdx, "dX")
        rows.append(P.cpu().numpy())
    check_exact(rows[1], rows[0][edge], "term rows at CSR positions")
    assert bl.bitlogic_device_error() == 0


@pytest.mark.parametrize("k", [3, 4])
@pytest.mark.parametrize("B", [512, 516])
@pytest.mark.parametrize("over", [False, True])
def test_large_inputs_take_the_staged_kernel(k, B, over):
    # both sides of the line, for both sources of the gradient
    w_in, w = -(-16000000 // B) - (0 if over else 1), 90
    X = synth.uniform_activations(w_in, B, seed=B)
    conn = synth.connectivity(w, k, w_in, seed=1)
    theta = synth.table_logits(w, 1 << k, seed=2)
    dY = synth.uniform_gradients(w, B, seed=3, scale=1e-2)
    Xd, rows = dev(X), np.unique(conn)
    small = np.searchsorted(rows, conn).astype(np.int32)   # the same layer on the rows that it reads
    wth, wdx = oracle.lut_backward(X[rows].astype(np.float64), small, theta, dY.astype(np.float64), want_dx=True)
    off, edge = bl.bitlogic_build_csr(small, len(rows))
    outs = []
    for source in (dict(dY=dev(dY)), dict(up_terms=dev(dY), up_off=dev(np.arange(w + 1, dtype=np.int32)))):
        dth, P = torch.full((w, 1 << k), np.nan, device="cuda"), torch.full((w * k, B), np.nan, device="cuda")
        bl.bitlogic_lut_backward_node(Xd, dev(conn), dev(theta), dth, "soft", edge_terms=P, **source)
        dX = torch.full((len(rows), B), np.nan, device="cuda")
        bl.bitlogic_csr_reduce(P, dev(off), dev(edge), dX)
        check_grad(dth, wth, "dtheta")
        check_grad(dX, wdx, "dX")
        outs.append((dth.cpu().numpy(), P.cpu().numpy()))
    for a, b in zip(*outs):
        check_exact(a, b, "gradient from rows and from terms")
    assert bl.bitlogic_device_error() == 0


@pytest.mark.parametrize("C,g,B", [(100, 10, 907), (10, 63, 130), (10, 64, 31), (7, 1, 5), (10, 120, 67)])
def test_head_of_short_groups(C, g, B):
    # both sides of the group size from which long batches of rows are read
    Y = np.random.default_rng(C + B).random((C * g, B)).astype(np.float32)
    labels = np.random.default_rng(B).integers(0, C, size=B).astype(np.int32)
    loss, logits = torch.zeros(1, device="cuda"), torch.full((B, C), np.nan, device="cuda")
    ws = torch.empty(bl.bitlogic_head_loss_workspace(B, C), dtype=torch.uint8, device="cuda")
    bl.bitlogic_head_loss(dev(Y), dev(labels), C, 20.0, loss, ws, logits=logits)
    wl, wloss, _ = oracle.head_loss(Y.astype(np.float64), labels, C, 20.0)
    check_fwd(logits, wl, "logits")
    check_fwd(loss, np.array([wloss]), "loss")
    assert bl.bitlogic_device_error() == 0


@pytest.mark.parametrize("B", [4, 60, 124, 128, 132, 256, 260])
def test_routing_input_gradient_around_its_slices(B):
    # one group of samples per lane up to 128, two beyond; rows with no, few and
    # more than 32 readers
    w_in, slots, Kc = 30, 90, 8
    X, G = synth.uniform_activations(w_in, B, seed=1), synth.uniform_gradients(slots, B, seed=2, scale=1e-2)
    cand = synth.candidate_pools(slots, Kc, w_in - 1, seed=3)
    cand[:50, 0] = 5
    r = synth.table_logits(slots, Kc, seed=4)
    off, edge = bl.bitlogic_build_csr(cand, w_in)
    p, dr = torch.empty(slots, Kc, device="cuda"), torch.empty(slots, Kc, device="cuda")
    bl.bitlogic_route_forward(dev(X), dev(cand), dev(r), torch.empty(slots, B, device="cuda"), p)
    dX = torch.full((w_in, B), np.nan, device="cuda")
    bl.bitlogic_route_backward(dev(X), dev(cand), dev(r), dev(G), dr, p, dev(off), dev(edge), dX)
    wdr, wdX = oracle.route_backward(X.astype(np.float64), cand, r, G.astype(np.float64))
    check_grad(dX, wdX, "dX")
    check_grad(dr, wdr, "dr")
    assert bl.bitlogic_device_error() == 0

"""GPU parity of layer 2 on corner codes of layer 1: the codes and tables
against the bit-row forward (bit for bit), the layer-2 forward and backward
and the corner reduction against the oracle on the decoded rows, at the edges
of the kernels' stages (64 and 128 samples), fan-ins and table sizes."""
import os

import numpy as np
import pytest
import torch

import oracle
import paper_2602_07400_gb300 as bl
from paper_2602_07400_gb300 import synth
from paper_2602_07400_gb300.pipeline import Network, TrainStep
from parity_util import check_exact, check_fwd, check_grad
from test_gpu_bitrows import dev, pack_rows

pytestmark = pytest.mark.gpu

oracle.set_threads(os.cpu_count() or 1)


def _layer1(w_in, w1, k1, B, node, seed=0):
    """Codes and table of a layer on random binary wires, and its fp32 rows."""
    bits = synth.binary_activations(w_in, B, seed=seed + B)
    conn = synth.connectivity(w1, k1, w_in, seed=seed + 1)
    theta = synth.table_logits(w1, 1 << k1, seed=seed + 2)
    X = dev(pack_rows(bits))
    codes = torch.full((w1, bl.code_bytes(B)), 255, dtype=torch.uint8, device="cuda")
    table = torch.empty(w1, 1 << k1, device="cuda")
    bl.bitlogic_lut_forward_codes(X, B, dev(conn), dev(theta), codes, table, node)
    Y = torch.empty(w1, B, device="cuda")
    bl.bitlogic_lut_forward_bitrows(X, B, dev(conn), dev(theta), Y, node)
    corner = (bits[conn].astype(np.int64) << np.arange(k1)[None, :, None]).sum(axis=1)
    return codes, table, Y, corner, theta


@pytest.mark.parametrize("k1,B,node", [(1, 5, "soft"), (2, 128, "st"), (3, 1024, "soft"), (4, 1027, "st"),
                                       (5, 2049, "soft"), (6, 907, "soft"), (6, 1024, "st")])
def test_codes_and_decode(k1, B, node):
    codes, table, Y, corner, theta = _layer1(50, 37, k1, B, node)
    got = codes.cpu().numpy()
    check_exact(got[:, :B], (4 * corner).astype(np.uint8), "codes")
    assert not got[:, B:].any()                       # padding
    out = torch.full_like(Y, np.nan)
    bl.bitlogic_codes_decode(codes, table, out)
    check_exact(out.cpu().numpy(), Y.cpu().numpy(), "decoded rows vs bit-row forward")
    assert bl.bitlogic_device_error() == 0


# B: below a stage, at its edges, ragged and unaligned rows, several stages;
# w: fewer and more nodes than one wave of the persistent warps
SHAPES = [(6, 6, 40, 30, 1), (6, 6, 90, 60, 64), (6, 6, 120, 3000, 132), (6, 4, 300, 200, 1027), (6, 1, 60, 40, 907),
          (5, 5, 80, 50, 63), (5, 6, 200, 4000, 200), (5, 2, 70, 36, 128), (4, 4, 100, 3000, 65), (4, 6, 64, 40, 1000),
          (4, 3, 50, 24, 37), (6, 5, 100, 80, 2048)]


@pytest.mark.parametrize("k,k1,w1,w,B", SHAPES)
@pytest.mark.parametrize("node", ["soft", "st"])
def test_layer2_on_codes(k, k1, w1, w, B, node):
    codes, table, Y1, corner, theta1 = _layer1(64, w1, k1, B, node)
    conn = synth.connectivity(w, k, w1, seed=11)
    theta = synth.table_logits(w, 1 << k, seed=12)
    X = Y1.cpu().numpy().astype(np.float64)
    Y = torch.full((w, B), np.nan, device="cuda")
    bl.bitlogic_lut_forward_coded(codes, table, dev(conn), dev(theta), Y, node)
    want = oracle.lut_forward(X, conn, theta, node)
    if node == "st":
        check_exact(Y.cpu().numpy().astype(np.float64), want, "y (binary inputs)")
    else:
        check_fwd(Y, want, "y")
    # the fp32-row forward evaluates the same expressions (at fan-in 4 on ragged
    # rows it is the lerp tree of the scalar kernel, which rounds differently)
    Yr = torch.empty_like(Y)
    if B % 4 == 0 or k >= 5:
        bl.bitlogic_lut_forward_node(Y1, dev(conn), dev(theta), Yr, node)
        check_exact(Y.cpu().numpy(), Yr.cpu().numpy(), "y vs fp32 rows")
    group = 2
    dYg = synth.uniform_gradients(w // group, B, seed=13, scale=1e-2)
    off, edge = bl.bitlogic_build_csr(conn, w1)
    pos = bl.bitlogic_csr_positions(edge)
    dth = torch.full((w, 1 << k), np.nan, device="cuda")
    H = torch.full((w * k, 1 << k1), np.nan, device="cuda")
    bl.bitlogic_lut_backward_coded(codes, table, B, dev(conn), dev(theta), dth, H, dev(dYg), group, node)
    Hp = torch.full_like(H, np.nan)
    dth_p = torch.empty_like(dth)
    bl.bitlogic_lut_backward_coded(codes, table, B, dev(conn), dev(theta), dth_p, Hp, dev(dYg), group, node,
                                   edge_pos=dev(pos))
    check_exact(dth_p.cpu().numpy(), dth.cpu().numpy(), "dtheta with positions (and run to run)")
    check_exact(Hp.cpu().numpy(), H.cpu().numpy()[edge], "corner sums at CSR positions")
    dY = np.repeat(dYg.astype(np.float64), group, axis=0)
    wth, wdx = oracle.lut_backward(X, conn, theta, dY, want_dx=True, node=node)
    check_grad(dth, wth, "dtheta")
    # corner sums of an edge add up to the edge's terms: their totals per input
    # node and corner are those of the input gradient
    tot = np.zeros((w1, 1 << k1))
    np.add.at(tot, conn.reshape(-1), H.cpu().numpy().astype(np.float64))
    want_tot = np.zeros((w1, 1 << k1))
    for a in range(1 << k1):
        want_tot[:, a] = np.where(corner == a, wdx, 0.0).sum(axis=1)
    check_grad(tot, want_tot, "corner sums")
    d1 = torch.full((w1, 1 << k1), np.nan, device="cuda")
    bl.bitlogic_corner_reduce(Hp, dev(off), None, dev(theta1), d1)
    d1e = torch.empty_like(d1)
    bl.bitlogic_corner_reduce(H, dev(off), dev(edge), dev(theta1), d1e)
    check_exact(d1e.cpu().numpy(), d1.cpu().numpy(), "corner reduction with an edge map")
    s = 1.0 / (1.0 + np.exp(-theta1.astype(np.float64)))
    check_grad(d1, s * (1 - s) * want_tot, "layer-1 dtheta")
    assert bl.bitlogic_device_error() == 0


def test_out_of_range_indices_are_flagged():
    codes, table, Y1, corner, theta1 = _layer1(64, 40, 4, 100, "soft")
    conn = synth.connectivity(20, 4, 40, seed=3)
    theta = dev(synth.table_logits(20, 16, seed=4))
    bad = conn.copy()
    bad[3, 1] = 40
    bad[7, 0] = -1
    zero = conn.copy()
    zero[3, 1] = zero[7, 0] = 0
    outs = []
    for c in (bad, zero):
        Y, dth = torch.empty(20, 100, device="cuda"), torch.empty(20, 16, device="cuda")
        H = torch.empty(80, 16, device="cuda")
        bl.bitlogic_lut_forward_coded(codes, table, dev(c), theta, Y)
        bl.bitlogic_lut_backward_coded(codes, table, 100, dev(c), theta, dth, H, Y)
        outs.append((Y.cpu().numpy(), dth.cpu().numpy(), H.cpu().numpy()))
        assert bl.bitlogic_device_error() == (-8 if c is bad else 0)
    for a, b in zip(*outs):
        check_exact(a, b, "row 0 in place of an index out of range")
    # codes beyond the table are taken modulo its size
    wild = codes.clone()
    wild |= 0xC3
    Y, Yw = torch.empty(20, 100, device="cuda"), torch.empty(20, 100, device="cuda")
    bl.bitlogic_lut_forward_coded(codes, table, dev(conn), theta, Y)
    bl.bitlogic_lut_forward_coded(wild, table, dev(conn), theta, Yw)
    check_exact(Yw.cpu().numpy(), Y.cpu().numpy(), "code bits outside the table")


@pytest.mark.parametrize("B,k,node", [(256, 6, "soft"), (127, 6, "soft"), (255, 4, "st"), (130, 5, "soft"), (37, 4, "soft")])
def test_training_step_on_codes(B, k, node):
    # the whole step, ragged batches included, against the oracle, and with
    # dY1 kept (formed from the terms) the same outputs
    wl = synth.Workload("codes", B, 60, 5, 40.0, (64, 128, 192), (300, 200), k, 5.0)
    conn1, th1, conn2, th2 = synth.network(wl, seed=3)
    x, labels = synth.blob_batch(B, wl.d, wl.classes, wl.sigma, seed=4)
    net = Network(conn1, th1, conn2, th2, wl.w_in)
    steps = []
    for keep in (False, True):
        st = TrainStep(net, B, wl.d, wl.thresholds, wl.classes, wl.tau, node=node, keep_dy1=keep)
        # a ragged batch offers dY1 with or without keep_dy1
        assert st.codes1 and st.bits1 and st.fuse_dy1 and (st.dy1 is not None) == (keep or B % 4 != 0)
        st.load(x.cuda(), labels.cuda())
        st.run()
        steps.append(st)
    torch.cuda.synchronize()
    r = oracle.train_step(x.numpy(), labels.numpy(), wl.thresholds, conn1, th1, conn2, th2, wl.classes, wl.tau,
                          want_dx1=False, node=node)
    a, b = steps
    check_fwd(a.y1, r["y1"], "y1")
    check_fwd(a.y2, r["y2"], "y2", atol=1e-6 if node == "st" else 0.0)
    check_fwd(a.logits, r["logits"], "logits", atol=1e-6)
    for name in ("dth1", "dth2"):
        check_grad(getattr(a, name), r[name], name)
        check_exact(getattr(a, name).cpu().numpy(), getattr(b, name).cpu().numpy(), name)
    check_grad(b.dy1, r["dy1"], "dy1")
    assert bl.bitlogic_device_error() == 0


def test_ragged_batch_refuses_other_binary_wires():
    wl = synth.Workload("codes", 37, 60, 5, 40.0, (64, 128, 192), (300, 200), 4, 5.0)
    net = Network(*synth.network(wl, seed=3), wl.w_in)
    for kw in (dict(bytes1=True), dict(bits1=True), dict(bytes1=True, bits1=True)):
        with pytest.raises(ValueError):
            TrainStep(net, 37, wl.d, wl.thresholds, wl.classes, wl.tau, **kw)
    st = TrainStep(net, 37, wl.d, wl.thresholds, wl.classes, wl.tau, codes1=False)
    assert not st.codes1 and not st.bytes1 and st.bits.dtype == torch.float32


@pytest.mark.parametrize("k1", [1, 4, 6])
@pytest.mark.parametrize("w,deg", [(1, 4), (5, 8), (3, 63), (7, 32), (13, 100), (2500, 9)])
def test_corner_reduce_with_few_nodes(k1, w, deg):
    # several warps per node: runs of unequal length, nodes without a reader
    rng = np.random.default_rng(w + deg)
    n, K = w * deg, 1 << k1
    owner = np.sort(rng.integers(0, w, size=n))
    if w > 2:
        owner[owner == 1] = 0
    off = np.searchsorted(owner, np.arange(w + 1)).astype(np.int32)
    H = rng.standard_normal((n, K), dtype=np.float32)
    theta = synth.table_logits(w, K, seed=2)
    total = np.zeros((w, K))
    np.add.at(total, owner, H.astype(np.float64))
    size = np.zeros((w, K))
    np.add.at(size, owner, np.abs(H).astype(np.float64))
    s = 1.0 / (1.0 + np.exp(-theta.astype(np.float64)))
    perm = rng.permutation(n).astype(np.int32)
    shuffled = np.empty_like(H)
    shuffled[perm] = H
    outs = []
    for rows, edge in ((H, None), (shuffled, dev(perm))):
        d = torch.full((w, K), np.nan, device="cuda")
        bl.bitlogic_corner_reduce(dev(rows), dev(off), edge, dev(theta), d)
        outs.append(d.cpu().numpy())
    check_exact(outs[1], outs[0], "with an edge map")
    # fp32 sums of m terms: error below m 2^-24 of the terms' magnitudes
    bound = s * (1 - s) * (size * (deg * 8 + 8) * 2.0 ** -24 + 2.0 ** -20 * np.abs(total)) + 1e-30
    assert np.all(np.abs(outs[0] - s * (1 - s) * total) <= bound)
    assert bl.bitlogic_device_error() == 0


@pytest.mark.parametrize("k,k1,B", [(6, 6, 5), (6, 6, 64), (6, 5, 100), (6, 1, 131), (6, 6, 256), (6, 6, 1001), (5, 5, 200),
                                    (5, 3, 333), (5, 6, 260), (6, 6, 1030), (4, 4, 127), (4, 2, 37), (4, 6, 190),
                                    (4, 5, 385)])
def test_nan_logits_reach_only_the_samples_that_select_them(k, k1, B):
    # a table entry that no sample selects changes nothing, whatever it holds:
    # lanes past the batch must not stand for a sample at entry 0
    rng = np.random.default_rng(k + B)
    w1, w, K1 = 20, 24, 1 << k1
    a = rng.integers(0, K1, size=(w1, B))
    a[3] = rng.integers(1, K1, size=B)
    padded = np.zeros((w1, bl.code_bytes(B)), np.uint8)
    padded[:, :B] = 4 * a
    conn = synth.connectivity(w, k, w1, seed=1)
    conn[2, 0], conn[2, 1:] = 3, np.arange(4, 3 + k)
    theta = synth.table_logits(w, 1 << k, seed=2)
    table = rng.random((w1, K1)).astype(np.float32)
    dY = synth.uniform_gradients(w, B, seed=3, scale=1e-2)

    def backward(table, theta):
        dth, H = torch.empty(w, 1 << k, device="cuda"), torch.empty(w * k, K1, device="cuda")
        bl.bitlogic_lut_backward_coded(dev(padded), dev(table), B, dev(conn), dev(theta), dth, H, dev(dY))
        return dth.cpu().numpy(), H.cpu().numpy()

    dth, H = backward(table, theta)
    assert np.isfinite(dth).all() and np.isfinite(H).all()
    hole = table.copy()
    hole[3, 0] = np.nan
    for got, want, name in zip(backward(hole, theta), (dth, H), ("dtheta", "corner sums")):
        check_exact(got, want, name + " with an unselected NaN entry")
    bad = theta.copy()
    bad[2, 1] = np.nan
    dth_b, H_b = backward(table, bad)
    others = np.arange(w) != 2
    check_exact(dth_b[others], dth[others], "other nodes' dtheta")
    check_exact(H_b[np.repeat(others, k)], H[np.repeat(others, k)], "other nodes' corner sums")
    for i in range(k):
        unread = np.setdiff1d(np.arange(K1), a[conn[2, i]])
        assert not H_b[2 * k + i, unread].any(), "corners that no sample is on"


@pytest.mark.parametrize("k", [6, 5, 4])
@pytest.mark.parametrize("B", [256, 37])
def test_step_on_parameters_off_an_aligned_address(k, B):
    # logits that are slices of one parameter vector, starting at any float
    wl = synth.Workload("codes", B, 60, 5, 40.0, (64, 128, 192), (300, 200), k, 5.0)
    params = synth.network(wl, seed=3)
    x, labels = synth.blob_batch(B, wl.d, wl.classes, wl.sigma, seed=4)
    outs = []
    for offset in (0, 1, 3):
        net = Network(*params, wl.w_in)
        for name in ("theta1", "theta2"):
            t = getattr(net, name)
            flat = torch.zeros(t.numel() + 4, device="cuda")
            view = flat[offset:offset + t.numel()].view(t.shape)
            view.copy_(t)
            setattr(net, name, view)
        st = TrainStep(net, B, wl.d, wl.thresholds, wl.classes, wl.tau)
        st.load(x.cuda(), labels.cuda())
        st.run()
        outs.append([t.cpu().numpy() for t in (st.logits, st.dth1, st.dth2)])
    for got in outs[1:]:
        for a, b in zip(got, outs[0]):
            check_exact(a, b, "as with aligned logits")
    assert bl.bitlogic_device_error() == 0


@pytest.mark.parametrize("B,k,node", [(127, 6, "soft"), (37, 4, "st"), (257, 5, "soft")])
def test_ragged_step_offers_the_gradient_of_layer_1(B, k, node):
    # without keep_dy1, eager and replayed, also once the logits have moved on
    wl = synth.Workload("codes", B, 60, 5, 40.0, (64, 128, 192), (300, 200), k, 5.0)
    params = synth.network(wl, seed=3)
    x, labels = synth.blob_batch(B, wl.d, wl.classes, wl.sigma, seed=4)
    conn1, th1, conn2, th2 = params
    r = oracle.train_step(x.numpy(), labels.numpy(), wl.thresholds, conn1, th1, conn2, th2, wl.classes, wl.tau,
                          want_dx1=False, node=node)
    for captured in (False, True):
        st = TrainStep(Network(*params, wl.w_in), B, wl.d, wl.thresholds, wl.classes, wl.tau, node=node)
        assert st.dy1.shape == (300, B)
        st.load(x.cuda(), labels.cuda())
        if captured:
            st.capture().replay()
        else:
            st.run()
        before = st.dy1
        check_grad(before, r["dy1"], "dy1")
        st.update(lr=0.5)
        st.x.zero_()
        check_exact(st.dy1.cpu().numpy(), before.cpu().numpy(), "dy1 after the update")
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        st.load(x.cuda(), labels.cuda())
        torch.cuda.synchronize()
        st.run(stream=side)
        side.synchronize()
        want = oracle.train_step(x.numpy(), labels.numpy(), wl.thresholds, conn1, st.net.theta1.cpu().numpy(), conn2,
                                 st.net.theta2.cpu().numpy(), wl.classes, wl.tau, want_dx1=False, node=node)
        check_grad(st.dy1, want["dy1"], "dy1 of a step on another stream")
    assert bl.bitlogic_device_error() == 0

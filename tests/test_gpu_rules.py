"""The Muon comparison rule of Eq. (6) and the Eq. (11) direction counters,
CUDA path vs the fp64 oracle through the C ABI (needs a GB300)."""
import numpy as np
import pytest

import parity as PT
from oracle import meqmuon as O
from paper_2609_35701_gb300 import workloads as W

pytestmark = pytest.mark.gpu

LR, MU, WD, EPS = 0.02, 0.95, 0.1, 1e-7


@pytest.fixture(scope="module")
def meq():
    import __graft_entry__

    __graft_entry__.build()
    import torch

    assert torch.cuda.is_available()
    from paper_2609_35701_gb300 import meq as m

    return m


def _to_dev(ts):
    return [t.contiguous().cuda() for t in ts]


@pytest.mark.parametrize("nesterov", [0, 1])
def test_muon_rule_matches_oracle(meq, nesterov):
    """Eq. (6) on tall, wide, square and ragged shapes (several tiles and a
    tail), three steps, each matrix staged from the GPU's own W and B."""
    wl = W.custom_workload([(320, 576), (576, 320), (256, 256), (200, 1000), (96, 40)], pattern="both", seed=21)
    shapes = [(r, c) for _, r, c in wl.shapes]
    opt = meq.MeqMuon(shapes, update_rule=meq.RULE_MUON, nesterov=nesterov)
    params = _to_dev(W.initial_weights(wl))
    B_prev = [np.zeros(s) for s in shapes]
    for t in range(3):
        Gs = W.gradients(wl, t)
        W0 = [p.cpu().double().numpy() for p in params]
        opt.step(params, _to_dev(Gs), LR, MU, WD, EPS)
        opt.sync()
        for i in range(len(shapes)):
            B = opt.read_momentum(i)
            PT.check_muon_step(W0[i], Gs[i].double().numpy(), B_prev[i], params[i].cpu().numpy(), B,
                               opt.read_ns_output(i), opt.read_stats(i), LR, MU, WD, EPS, nesterov=bool(nesterov),
                               Ut_gpu=opt.read_update(i))
            B_prev[i] = B
            assert opt.read_direction_counts(i) == (0, 0)
    opt.close()


def test_muon_rule_update_rms(meq):
    """Eq. (6) keeps the update RMS near rho for every shape: the applied
    update divided by eta has RMS rho sqrt(max(m, n)) ||U||_F / sqrt(m n),
    which the oracle's U fixes; for these well-conditioned gradients NS
    output singular values lie in the quintic's band [0.68, 1.2]."""
    wl = W.custom_workload([(128, 512), (512, 128), (384, 384)], pattern="none", seed=5)
    shapes = [(r, c) for _, r, c in wl.shapes]
    opt = meq.MeqMuon(shapes, update_rule=meq.RULE_MUON)
    params = _to_dev(W.initial_weights(wl))
    W0 = [p.cpu().double().numpy() for p in params]
    G = W.gradients(wl, 0)
    opt.step(params, _to_dev(G), LR, MU, 0.0, EPS)
    opt.sync()
    for i, (m, n) in enumerate(shapes):
        upd = (W0[i] - params[i].cpu().double().numpy()) / LR
        U = O.newton_schulz(G[i].double().numpy())
        want = O.RHO * np.sqrt(max(m, n)) * np.linalg.norm(U) / np.sqrt(m * n)
        got = np.sqrt((upd * upd).mean())
        assert abs(got - want) / want < 1e-2, (m, n, got, want)
        assert 0.68 * O.RHO < got < 1.21 * O.RHO
    opt.close()


def test_direction_counts(meq):
    """Device counters of Eq. (11): after T steps each hidden weight's row and
    column counts are the tallies of the directions the steps reported, and
    they sum to T; a reset zeroes them."""
    wl = W.custom_workload([(192, 448), (448, 192), (256, 256), (320, 320)], pattern="both", seed=8)
    shapes = [(r, c) for _, r, c in wl.shapes]
    opt = meq.MeqMuon(shapes)
    params = _to_dev(W.initial_weights(wl))
    tally = np.zeros((len(shapes), 2), np.int64)
    T = 7
    for t in range(T):
        opt.step(params, _to_dev(W.gradients(wl, t)), LR, MU, WD, EPS)
        opt.sync()
        for i in range(len(shapes)):
            tally[i, opt.read_stats(i)["direction"]] += 1
    for i in range(len(shapes)):
        assert opt.read_direction_counts(i) == tuple(tally[i]), i
        assert sum(opt.read_direction_counts(i)) == T
    opt.reset_direction_counts()
    opt.sync()
    assert all(opt.read_direction_counts(i) == (0, 0) for i in range(len(shapes)))
    opt.step(params, _to_dev(W.gradients(wl, T)), LR, MU, WD, EPS)
    opt.sync()
    assert all(sum(opt.read_direction_counts(i)) == 1 for i in range(len(shapes)))
    opt.close()


def test_direction_counts_follow_the_orthogonality_constraint(meq):
    """Section 3.1: orthogonalising a wide matrix (m < n) equalises its rows,
    a tall one its columns, so with row / column imbalance on the free side
    Eq. (11) picks column for wide and row for tall weights at every step."""
    wl = W.custom_workload([(256, 768), (768, 256)], pattern="both", seed=13)
    shapes = [(r, c) for _, r, c in wl.shapes]
    opt = meq.MeqMuon(shapes)
    params = _to_dev(W.initial_weights(wl))
    for t in range(5):
        opt.step(params, _to_dev(W.gradients(wl, t)), LR, MU, WD, EPS)
    opt.sync()
    assert opt.read_direction_counts(0) == (0, 5)   # wide: column-wise
    assert opt.read_direction_counts(1) == (5, 0)   # tall: row-wise
    opt.close()


def test_ns_cv_trajectory_matches_oracle(meq):
    """Section 3.1 replay of Eq. (5) through the CUDA path: the row and column
    CVs of X_0..X_20 agree with the fp64 oracle's trajectory (the GPU runs
    its 16-bit NS, so the CVs carry its ~1e-3 relative output error)."""
    import torch

    wl = W.custom_workload([(256, 640), (640, 256), (384, 384)], pattern="both", seed=17)
    for i, (_, m, n) in enumerate(wl.shapes):
        G = W.gradient(wl, i, 0)
        gr, gc = meq.ns_cv_trajectory(G.cuda().contiguous(), steps=20)
        orr, oc = O.ns_cv_trajectory(G.double().numpy(), steps=20)
        assert gr.shape == (21,) and gc.shape == (21,)
        assert abs(gr[0] - orr[0]) <= 1e-4 * orr[0] and abs(gc[0] - oc[0]) <= 1e-4 * max(oc[0], 1e-6)
        assert np.all(np.abs(gr - orr) <= 5e-3 + 2e-2 * orr), (m, n, np.abs(gr - orr).max())
        assert np.all(np.abs(gc - oc) <= 5e-3 + 2e-2 * oc), (m, n, np.abs(gc - oc).max())
        # Section 3.1: orthogonalisation equalises the rows of a wide matrix
        # and the columns of a tall one, leaving the other side's imbalance;
        # a square matrix has both sides constrained
        if m < n:
            assert gr[20] < 0.1 * gr[0] and gr[20] < 0.2 * gc[20], (m, n, gr[[0, 20]], gc[[0, 20]])
        elif m > n:
            assert gc[20] < 0.1 * gc[0] and gc[20] < 0.2 * gr[20], (m, n, gr[[0, 20]], gc[[0, 20]])
        else:
            assert gr[20] < 0.1 * gr[0] and gc[20] < 0.1 * gc[0], (m, n, gr[[0, 20]], gc[[0, 20]])
    torch.cuda.synchronize()


@pytest.mark.parametrize("shape", [(200, 333), (333, 200), (256, 256), (64, 9000)])
@pytest.mark.parametrize("opts", [{}, {"ns_x0_fused": 0}, {"ns_fp16_mask": 0}, {"ns_fp16_mask": 0b01101},
                                  {"nesterov": 1, "ns_cta_pair": 0}], ids=str)
def test_ns_cv_trajectory_is_that_of_separate_steps(meq, shape, opts):
    """Point k of the trajectory equals, bit for bit, the CVs that a k-iteration step from the same
    matrix reports (tall and wide, operand formats that change between iterations)."""
    import torch

    H = torch.randn(shape, generator=torch.Generator().manual_seed(5)) * torch.logspace(-1, 1, shape[0])[:, None]
    gr, gc = meq.ns_cv_trajectory(H.cuda(), steps=6, **opts)
    for k in (1, 2, 5, 6):
        opt = meq.MeqMuon([shape], ns_steps=k, **opts)
        opt.step([torch.zeros(shape, device="cuda")], [H.cuda()], 0.0, 0.0, 0.0)
        st = opt.read_stats(0)
        assert (gr[k], gc[k]) == (st["gamma_r"], st["gamma_c"]), k
        opt.close()


def test_ns_cv_trajectory_threshold_applies_to_x0(meq):
    """Section 3.1 replays Eq. (5) from X_0 = H / ||H||_F, and Eq. (8)
    counts the rows and columns whose RMS exceeds delta: the threshold is on
    X_0's RMS, not H's. H here has a large norm, one row at 3 delta and one
    at delta / 10 in X_0, and one column at delta / 10 (still below delta
    after one iteration, whose slope at zero is a = 3.4445); the oracle's
    CVs (that row and column left out) must be reproduced, and reading the
    threshold on H instead would be caught."""
    import torch

    rng = np.random.default_rng(3)
    m, n = 64, 96
    H = rng.standard_normal((m, n)) * 1e3 * np.exp(rng.uniform(-1, 1, (m, 1)))
    H[5] = H[6] = 0.0
    H[:, 7] = 0.0
    nrm = np.sqrt((H * H).sum())
    u = rng.standard_normal(n)
    H[5] = u / np.linalg.norm(u) * 3e-7 * np.sqrt(n) * nrm
    H[6] = u / np.linalg.norm(u) * 1e-8 * np.sqrt(n) * nrm
    v = rng.standard_normal(m)
    v[[5, 6]] = 0.0
    H[:, 7] = v / np.linalg.norm(v) * 1e-8 * np.sqrt(m) * nrm
    H = H.astype(np.float32).astype(np.float64)
    orr, oc = O.ns_cv_trajectory(H, steps=1)
    r_h, c_h = O.row_col_rms(H)
    # the other reading differs well beyond the tolerance
    assert abs(O.coefficient_of_variation(r_h) - orr[0]) > 1e-2 * orr[0]
    assert abs(O.coefficient_of_variation(c_h) - oc[0]) > 1e-2 * oc[0]
    gr, gc = meq.ns_cv_trajectory(torch.from_numpy(H.astype(np.float32)).cuda(), steps=1)
    assert abs(gr[0] - orr[0]) <= 1e-4 * orr[0], (gr[0], orr[0])
    assert abs(gc[0] - oc[0]) <= 1e-4 * oc[0], (gc[0], oc[0])
    assert abs(gr[1] - orr[1]) <= 5e-3 + 2e-2 * orr[1] and abs(gc[1] - oc[1]) <= 5e-3 + 2e-2 * oc[1]


def test_ns_cv_trajectory_large_matrix(meq):
    """8192 x 8192 (beyond the allocation-free entry point's fixed scratch:
    the replay has its own), k = 0 and 1 against the oracle."""
    import torch

    gen = torch.Generator().manual_seed(11)
    m = n = 8192
    H = torch.randn(m, n, generator=gen) * torch.exp(torch.empty(1, n).uniform_(-2.0, 2.0, generator=gen))
    gr, gc = meq.ns_cv_trajectory(H.cuda(), steps=1)
    orr, oc = O.ns_cv_trajectory(H.double().numpy(), steps=1)
    assert abs(gr[0] - orr[0]) <= 1e-4 * max(orr[0], 1e-6) and abs(gc[0] - oc[0]) <= 1e-4 * oc[0], (gr, gc, orr, oc)
    assert np.all(np.abs(gr - orr) <= 5e-3 + 2e-2 * orr) and np.all(np.abs(gc - oc) <= 5e-3 + 2e-2 * oc)
    torch.cuda.synchronize()

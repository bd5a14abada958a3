"""One filter update at the sizes where the kernels split their work differently, against the FP64 oracle,
and layouts symmetric about 0 against the general kernels on the same problem.

Tolerances.  The message table, the existence probabilities and the noise weights: those of the parity tests.  Log
likelihoods: 2e-3 nats (FP32 geometry and amplitudes) plus 1e-6 of the PF log ratio's size (an
amplitude carries some 5e-7 and enters squared), 1e-3 nats plus 1e-6 of the MT log likelihood's
size, and an FP32 MT value (from 24 PFs on, unless selected) its own reported bound.  Two GPU paths:
twice these.
"""
import dataclasses

import numpy as np
import pytest

from oracle import beliefs, messages_woodbury, model, resample, synth
from paper_2604_19723_gb300 import workload as W

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::RuntimeWarning")]

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2604_19723_gb300 import bp  # noqa: E402

PAPER = dict(J=2, Nf=10, My=4, Mz=4)
# (geometry, PFs, particles)
CASES = [
    (dict(J=1, Nf=10, My=4, Mz=4), 1, 127), (PAPER, 2, 128), (PAPER, 3, 129),      # no other PF, one particle tile
    (PAPER, 8, 130), (PAPER, 9, 130), (PAPER, 16, 257), (PAPER, 17, 130),          # column groups, accumulator sets
    (PAPER, 23, 130), (PAPER, 24, 130), (PAPER, 32, 130), (PAPER, 33, 130),        # MT variants, A in tensor memory
    (PAPER, 40, 130), (PAPER, 41, 130), (PAPER, 48, 130), (PAPER, 49, 130),        # second MMA parts, 48 / 64 rows
    (dict(J=2, Nf=7, My=1, Mz=1), 3, 130), (dict(J=2, Nf=1, My=3, Mz=3), 3, 130),  # one antenna, one frequency
    (dict(J=2, Nf=9, My=1, Mz=7), 5, 130), (dict(J=3, Nf=5, My=3, Mz=3), 26, 130),  # odd everywhere
    (dict(J=2, Nf=8, My=2, Mz=3), 26, 130), (dict(J=2, Nf=75, My=2, Mz=2), 26, 130),  # odd rows; many frequencies
    (dict(J=1, Nf=16, My=8, Mz=8), 25, 66), (dict(J=1, Nf=9, My=9, Mz=5), 6, 66),   # many elements per frequency
]


def problem(geom_kw, S, P, seed):
    g, prm = W.make_geometry(**geom_kw), W.Params()
    scn = W.make_scenario(g, prm, N=3, K=max(S - 1, 1), seed=seed, snr_db=20.0)
    eta = synth.noise_variance(scn)
    z = synth.observe(scn, 1, eta, seed + 100).astype(np.complex64).astype(np.complex128)
    st = W.state_near_truth(scn, P=P, S=S, n=0, seed=seed + 1, eta_true=eta, pos_std=0.005, sfv_std=0.005,
                            uniform_weights=True)
    return g, prm, z, st


def update(g, prm, z, pred, P, S_max, seed):
    f = bp.Filter(g, prm, P=P, S_max=S_max, seed=seed)
    f.set_predicted(pred.n, pred.S, pred.x, pred.phi, pred.eta, pred.w_beta, pred.w_alpha, pred.w_xi, pred.zeta)
    f.update(torch.from_numpy(np.ascontiguousarray(z.astype(np.complex64))).cuda())
    torch.cuda.synchronize()
    return f


def loglik_tolerances(f, S, li, dk):
    tol_i = 1e-3 + 1e-6 * np.abs(li)
    if S >= 24:
        di = f.diag_iota()
        rest = np.ones(len(li), bool)
        rest[di["selected"]] = False
        tol_i = np.where(rest, np.maximum(tol_i, di["err"]), tol_i)
    return tol_i, 2e-3 + 1e-6 * np.abs(dk)


@pytest.mark.parametrize("case", CASES, ids=lambda c: "%dx%dx%d-S%d-P%d" % (c[0]["Nf"], c[0]["My"], c[0]["Mz"], c[1], c[2]))
def test_update_at_the_edges_of_the_splits(case):
    geom_kw, S, P = case
    g, prm, z, st = problem(geom_kw, S, P, 500 + S)
    S_max = 16 if S <= 16 else 64
    # the predicted belief without births keeps the PF count
    pred = model.predict(st, dataclasses.replace(prm, Q=0), g.J, seed=7, S_max=S_max)
    assert pred.S == S
    f = update(g, dataclasses.replace(prm, Q=0), z, pred, P, S_max, 7)
    msg = messages_woodbury.update_messages(pred, prm, g, z)
    tab, ll, gw = f.diag_table(S), f.diag_loglik(S), f.diag_weights(S)
    for key in ("m", "mw", "mu3", "mu4"):
        ref = getattr(msg.table, key)
        assert np.max(np.abs(tab[key] - ref)) <= 1e-5 * max(np.max(np.abs(ref)), 1e-300), key
    li, dk = msg.log_iota.sum(0), (msg.log_kappa1 - msg.log_kappa0[:, :, None]).sum(1)
    tol_i, tol_k = loglik_tolerances(f, S, li, dk)
    assert np.all(np.abs(ll["log_iota"] - li) <= tol_i), np.max(np.abs(ll["log_iota"] - li) / tol_i)
    assert np.all(np.abs(ll["delta_kappa"] - dk) <= tol_k), np.max(np.abs(ll["delta_kappa"] - dk) / tol_k)
    w_eta = beliefs.beliefs(pred, msg).w_eta
    for j in range(g.J):
        assert np.max(np.abs(gw["w_eta"][j] - w_eta[j])) < 1e-4 * np.max(w_eta[j]), j
    # estimates: FP64 sums of the FP32 particles with the weights that the update reports
    est = f.estimate()
    scale = np.max(np.abs(pred.x), axis=1)
    assert np.all(np.abs(est["x_hat"] - pred.x.astype(float) @ gw["w_x"]) <= 1e-9 * (1.0 + scale))
    for s in range(S):
        if gw["p_s"][s] > 0 and gw["w_y"][s].sum() > 0:
            w = gw["w_y"][s] / gw["w_y"][s].sum()
            want = pred.phi[s].astype(float) @ w
            assert np.all(np.abs(est["phi_hat"][s] - want) <= 1e-9 * (1.0 + np.max(np.abs(pred.phi[s]), axis=1))), s
    f.close()


@pytest.mark.parametrize("geom_kw, S", [(PAPER, 5), (PAPER, 26), (PAPER, 36), (PAPER, 60), (dict(J=2, Nf=5, My=3, Mz=3), 27),
                                        (dict(J=2, Nf=9, My=3, Mz=2), 12), (dict(J=1, Nf=16, My=8, Mz=8), 25)])
def test_symmetric_layouts_agree_with_the_general_kernels(geom_kw, S):
    """A picometre on one element makes the layout asymmetric (and changes its phase by 1e-10)."""
    P = 131
    g, prm, z, st = problem(geom_kw, S, P, 900 + S)
    prm = dataclasses.replace(prm, Q=0)
    off = np.zeros(g.My)
    off[0] = 1e-12
    pred = model.predict(st, prm, g.J, seed=9, S_max=64)
    a = update(g, prm, z, pred, P, 64, 9)
    b = update(dataclasses.replace(g, p_y=g.p_y + off), prm, z, pred, P, 64, 9)
    ta, tb = a.diag_table(S), b.diag_table(S)
    for key in ("m", "mw", "mu3", "mu4"):
        assert np.max(np.abs(ta[key] - tb[key])) <= 2e-5 * max(np.max(np.abs(tb[key])), 1e-300), key
    la, lb = a.diag_loglik(S), b.diag_loglik(S)
    tol_a, tol_k = loglik_tolerances(a, S, lb["log_iota"], lb["delta_kappa"])
    tol_b, _ = loglik_tolerances(b, S, lb["log_iota"], lb["delta_kappa"])
    assert np.all(np.abs(la["log_iota"] - lb["log_iota"]) <= tol_a + tol_b)
    assert np.all(np.abs(la["delta_kappa"] - lb["delta_kappa"]) <= 2.0 * tol_k)
    assert np.all(np.abs(a.diag_weights(S)["p_pr"] - b.diag_weights(S)["p_pr"]) < 2e-5)
    a.close()
    b.close()


@pytest.mark.parametrize("P", [1, 31, 2047, 2048, 2049, 4097])
def test_resampling_at_tile_edges(P):
    """Each index is the first whose cumulative weight reaches (U + i) / P, from the GPU's own weights."""
    g, prm, z, st = problem(dict(J=2, Nf=4, My=2, Mz=1), 2, P, 41)
    prm = dataclasses.replace(prm, Q=0, T_pru=0.0)
    pred = model.predict(st, prm, g.J, seed=41, S_max=8)
    f = update(g, prm, z, pred, P, 8, 41)
    gw, gi = f.diag_weights(pred.S), f.diag_indices(pred.S)
    triples = [(gw["w_x"], gi["x"], (0, 0))] + [(gw["w_eta"][j], gi["eta"][j], (2, j)) for j in range(g.J)] + \
        [(gw["w_y"][s], gi["y"][s], (1, s)) for s in range(pred.S)]
    for w, idx, (kind, index) in triples:
        u = (resample.resample_uniform(41, pred.n, kind, index) + np.arange(P)) / P
        c = np.cumsum(w) / np.sum(w)
        c[-1] = 1.0
        assert np.all(c[idx] >= u - 1e-12)
        assert np.all(np.where(idx > 0, c[np.maximum(idx - 1, 0)], 0.0) < u + 1e-12)
    f.close()

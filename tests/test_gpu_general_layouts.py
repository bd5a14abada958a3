"""One filter update on layouts that are not symmetric about 0, and on the largest arrays, against the FP64 oracle.

Element positions start at the corner element, or lie at irregular spacings, so that no element mirrors another and
the kernels for symmetric layouts would be wrong.  Tolerances: those of the symmetric layouts' tests.
"""
import dataclasses

import numpy as np
import pytest

from oracle import beliefs, messages_woodbury, model
from paper_2604_19723_gb300 import workload as W

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::RuntimeWarning")]

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from oracle import synth  # noqa: E402
from paper_2604_19723_gb300 import bp  # noqa: E402


def layout(kind, **kw):
    g = W.make_geometry(**kw)
    if kind == "symmetric":
        return g
    if kind == "corner":          # the first element is the origin of the array
        return dataclasses.replace(g, p_y=g.p_y - g.p_y[0] + 0.2 * g.wavelength, p_z=g.p_z - g.p_z[0] - 0.1 * g.wavelength)
    rng = np.random.default_rng(3)
    jitter = lambda p: p + rng.uniform(-0.15, 0.15, p.shape) * g.wavelength  # noqa: E731
    return dataclasses.replace(g, p_y=jitter(g.p_y), p_z=jitter(g.p_z))


def problem(kind, geom_kw, S, P, seed, twins=False):
    g, prm = layout(kind, **geom_kw), W.Params(Q=0)
    scn = W.make_scenario(g, prm, N=3, K=max(S - 1, 1), seed=seed, snr_db=20.0)
    eta = synth.noise_variance(scn)
    z = synth.observe(scn, 1, eta, seed + 100).astype(np.complex64)
    st = W.state_near_truth(scn, P=P, S=S, n=0, seed=seed + 1, eta_true=eta, pos_std=0.005, sfv_std=0.005,
                            uniform_weights=True)
    if twins:
        # the last PF a few millimetres from the one before it: its steering vectors lie close to the span of the others
        off = np.random.default_rng(seed).normal(0.0, 2e-3, (3, P)).astype(np.float32)
        st.phi[S - 1, :3] = st.phi[S - 2, :3] + off
    return g, prm, z, model.predict(st, prm, g.J, seed=9, S_max=64)


CASES = [("corner", dict(J=1, Nf=10, My=4, Mz=4), 1, 131), ("corner", dict(J=2, Nf=10, My=4, Mz=4), 5, 131),
         ("irregular", dict(J=2, Nf=9, My=3, Mz=3), 12, 130), ("irregular", dict(J=2, Nf=10, My=4, Mz=4), 23, 130),
         ("corner", dict(J=2, Nf=10, My=4, Mz=4), 24, 130), ("irregular", dict(J=2, Nf=8, My=2, Mz=3), 26, 130),
         ("irregular", dict(J=2, Nf=75, My=2, Mz=2), 33, 130), ("corner", dict(J=2, Nf=10, My=4, Mz=4), 40, 130),
         ("irregular", dict(J=2, Nf=10, My=4, Mz=4), 60, 130), ("corner", dict(J=1, Nf=9, My=9, Mz=5), 6, 66),
         ("irregular", dict(J=1, Nf=16, My=8, Mz=8), 25, 66),
         # (for the CUDA-core PF likelihood: middle elements, one antenna, one frequency, all columns)
         ("symmetric", dict(J=2, Nf=9, My=3, Mz=3), 21, 130), ("symmetric", dict(J=2, Nf=7, My=1, Mz=1), 4, 63),
         ("symmetric", dict(J=2, Nf=1, My=3, Mz=5), 3, 65), ("symmetric", dict(J=2, Nf=10, My=4, Mz=4), 64, 64),
         ("irregular", dict(J=1, Nf=37, My=1, Mz=1), 5, 129)]

# up to the largest array, the last two PFs millimetres apart: sums of the steering vectors' products over all elements
LARGE = [(kind, geom_kw, 5, 66, True) for kind in ("corner", "irregular", "symmetric")
         for geom_kw in (dict(J=1, Nf=12, My=8, Mz=8), dict(J=1, Nf=24, My=8, Mz=8), dict(J=1, Nf=32, My=8, Mz=8),
                         dict(J=1, Nf=128, My=4, Mz=4), dict(J=1, Nf=8, My=16, Mz=16))]


def check(kind, geom_kw, S, P, twins=False):
    g, prm, z, pred = problem(kind, geom_kw, S, P, 300 + S, twins)
    f = bp.Filter(g, prm, P=P, S_max=16 if S <= 16 else 64, seed=9)
    zd = torch.from_numpy(np.ascontiguousarray(z)).cuda()

    def update(**tiles):
        f.set_tiles(**tiles)
        f.set_predicted(pred.n, pred.S, pred.x, pred.phi, pred.eta, pred.w_beta, pred.w_alpha, pred.w_xi, pred.zeta)
        f.update(zd)
        return f.diag_loglik(S)

    cuda_cores = update(kappa_tc=-1)
    ll = update(kappa_tc=0)
    msg = messages_woodbury.update_messages(pred, prm, g, z.astype(np.complex128))
    tab, gw = f.diag_table(S), f.diag_weights(S)
    for key in ("m", "mw", "mu3", "mu4"):
        ref = getattr(msg.table, key)
        assert np.max(np.abs(tab[key] - ref)) <= 1e-5 * max(np.max(np.abs(ref)), 1e-300), key
    li, dk = msg.log_iota.sum(0), (msg.log_kappa1 - msg.log_kappa0[:, :, None]).sum(1)
    tol_i = 1e-3 + 1e-6 * np.abs(li)
    if S >= 24:                   # an FP32 value, unless selected, within its own reported bound
        di = f.diag_iota()
        rest = np.ones(P, bool)
        rest[di["selected"]] = False
        tol_i = np.where(rest, np.maximum(tol_i, di["err"]), tol_i)
    tol_k = 2e-3 + 1e-6 * np.abs(dk)
    assert np.all(np.abs(ll["log_iota"] - li) <= tol_i), np.max(np.abs(ll["log_iota"] - li) / tol_i)
    for got in (ll["delta_kappa"], cuda_cores["delta_kappa"]):
        assert np.all(np.abs(got - dk) <= tol_k), np.max(np.abs(got - dk) / tol_k)
    w_eta = beliefs.beliefs(pred, msg).w_eta
    for j in range(g.J):
        assert np.max(np.abs(gw["w_eta"][j] - w_eta[j])) < 1e-4 * np.max(w_eta[j]), j
    f.close()


@pytest.mark.parametrize("case", CASES + LARGE, ids=lambda c: "%s-%dx%dx%d-S%d" % (c[0], c[1]["Nf"], c[1]["My"], c[1]["Mz"], c[2]))
def test_update_on_a_general_layout(case):
    check(*case)


@pytest.mark.parametrize("kind", ["symmetric", "corner"])
def test_the_ill_conditioned_particles_are_counted_and_listed(kind):
    """Below 24 PFs: particles in which the last two PFs nearly coincide, on both layouts' routes."""
    P, S = 200, 5
    g, prm, z, pred = problem(kind, dict(J=2, Nf=10, My=4, Mz=4), S, P, 305, True)
    pred.phi[S - 1, :3, ::2] += np.float32(0.5)      # every other particle apart
    f = bp.Filter(g, prm, P=P, S_max=16, seed=9)
    f.set_predicted(pred.n, pred.S, pred.x, pred.phi, pred.eta, pred.w_beta, pred.w_alpha, pred.w_xi, pred.zeta)
    f.update(torch.from_numpy(np.ascontiguousarray(z)).cuda())
    listed = f.diag_iota()["selected"]
    assert len(listed) == f.estimate()["iota_repaired"] > 50
    assert len(np.unique(listed)) == len(listed) and listed[0] >= 0 and listed[-1] < P
    assert np.mean(listed % 2) > 0.9
    f.close()

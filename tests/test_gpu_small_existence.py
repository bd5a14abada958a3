"""Noise weights when existence probabilities vanish, against the FP64 oracle.

The m-vectors carry the existence weights in FP64, so the Gram matrix behind the noise likelihood has
entries whose squares leave the range of FP64.  What vanishes must drop out of the weights of the noise
variance; tolerance of the parity tests on those weights.
"""
import dataclasses

import numpy as np
import pytest

from oracle import beliefs, messages_woodbury, model, synth
from paper_2604_19723_gb300 import workload as W

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::RuntimeWarning")]

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2604_19723_gb300 import bp  # noqa: E402

P, S = 130, 6
SCALES = {
    "los": [(10.0 ** -e, 1.0, 1.0, 1.0, 1.0, 1.0) for e in range(130, 170, 3)],
    "second": [(1.0, 10.0 ** -e, 1.0, 1.0, 1.0, 1.0) for e in range(130, 170, 3)],
    "three": [(1.0, 1.0, 1.0) + (10.0 ** -e,) * 3 for e in range(60, 90, 2)],
    "graded": [(1.0, 1e-3, 1e-20, 1e-60, 1e-97, 1e-99), (1e-99, 1e-97, 1e-60, 1e-20, 1e-3, 1.0),
               (1e-30, 1e-60, 1e-90, 1e-120, 1e-150, 1e-180)],
    "all": [(10.0 ** -e,) * 6 for e in (20, 40, 60, 77, 80, 120, 160)],
}


@pytest.mark.parametrize("which", SCALES)
def test_noise_weights_with_vanishing_pfs(which):
    g, prm = W.make_geometry(J=2, Nf=10, My=4, Mz=4), W.Params(Q=0)
    scn = W.make_scenario(g, prm, N=3, K=S - 1, seed=71, snr_db=20.0)
    eta = synth.noise_variance(scn)
    z = synth.observe(scn, 1, eta, 171).astype(np.complex64)
    st = W.state_near_truth(scn, P=P, S=S, n=0, seed=72, eta_true=eta, pos_std=0.005, sfv_std=0.005, uniform_weights=True)
    pred = model.predict(st, prm, g.J, seed=7, S_max=16)
    f = bp.Filter(g, prm, P=P, S_max=16, seed=7)
    zd = torch.from_numpy(np.ascontiguousarray(z)).cuda()
    for scale in SCALES[which]:
        p = dataclasses.replace(pred, w_alpha=pred.w_alpha * np.array(scale)[:, None])
        f.set_predicted(p.n, p.S, p.x, p.phi, p.eta, p.w_beta, p.w_alpha, p.w_xi, p.zeta)
        f.update(zd)
        want = beliefs.beliefs(p, messages_woodbury.update_messages(p, prm, g, z.astype(np.complex128))).w_eta
        got = f.diag_weights(S)["w_eta"]
        assert np.all(np.isfinite(got)), scale
        for j in range(g.J):
            assert np.max(np.abs(got[j] - want[j])) < 1e-4 * np.max(want[j]), (scale, j)
    f.close()

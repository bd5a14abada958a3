"""An observation that holds NaN or Inf leaves no PF with a finite log ratio (and the estimate refuses it)."""
import numpy as np
import pytest

from oracle import model, synth
from paper_2604_19723_gb300 import workload as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2604_19723_gb300 import bp  # noqa: E402


@pytest.mark.parametrize("S", [1, 5, 26, 40])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("tensor_cores", [0, -1])
def test_no_log_ratio_from_an_observation_that_is_not_finite(S, bad, tensor_cores):
    g, prm, P = W.make_geometry(J=2), W.Params(Q=0), 130
    scn = W.make_scenario(g, prm, N=3, K=max(S - 1, 1), seed=5, snr_db=20.0)
    eta = synth.noise_variance(scn)
    z = synth.observe(scn, 1, eta, 171).astype(np.complex64)
    z[0, 3] = bad
    st = W.state_near_truth(scn, P=P, S=S, n=0, seed=72, eta_true=eta, pos_std=0.005, sfv_std=0.005)
    pred = model.predict(st, prm, g.J, seed=7, S_max=64)
    f = bp.Filter(g, prm, P=P, S_max=64, seed=7)
    f.set_tiles(kappa_tc=tensor_cores)
    f.set_predicted(pred.n, pred.S, pred.x, pred.phi, pred.eta, pred.w_beta, pred.w_alpha, pred.w_xi, pred.zeta)
    f.update(torch.from_numpy(z).cuda())
    assert not np.any(np.isfinite(f.diag_loglik(S)["delta_kappa"]))
    with pytest.raises(bp.BPError) as e:
        f.estimate()
    assert e.value.status == 4
    f.close()

"""FP32 with infinite and very large parameters: tanh of an infinite sum is +-1, on the tensor cores as
on the FMA pipe, so log|psi| and its sign stay what they are without derivatives; the derivatives
meet 0 x inf there, E_L is not finite and fn_sync reports it.  The value of log|psi| is compared between
local_energy (tensor cores for h1 = 128) and log_psi (FMA pipe) within the FP32 bound of 1e-4."""
import numpy as np
import pytest
import torch

import paper_2401_10287_gb300 as P
import workloads as W
from oracle import ansatz, mcmc
from gpu_helpers import make_pair, need_gpu, oracle_params, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("value", [np.inf, -np.inf, 3.4e38])
@pytest.mark.parametrize("where", ["layer 0", "layer", "mean field", "bias"])
def test_log_psi_with_a_saturated_column(where, value):
    need_gpu()
    sysm, ans = W.lih(1), W.Ansatz(3, 128, 16, 4, "aniso")
    net, gpu = make_pair(sysm, ans, 1)
    p = oracle_params(net, 2, 0.05).astype(np.float32)
    d = ansatz.unpack(net, p)                             # views of p
    if where == "bias":
        d["b1"][7] = value
    else:
        d["V0" if where == "layer 0" else "V1"][7, 140 if where == "mean field" else 3] = value
    r, _ = mcmc.init_walkers(sysm.nuclei, sysm.charges, sysm.n_up, sysm.n_down, sysm.partial_charges, 200, 3, 0.8,
                             dtype=np.float32)
    pd, rd = to_dev(p, torch.float32), to_dev(r, torch.float32)
    lv, sv = gpu.log_psi(pd, rd)
    gpu.sync()
    assert torch.isfinite(lv).all()
    e, lp, sg = gpu.local_energy(pd, rd)
    if where == "bias":                                   # no product with it: the derivatives of the column are zero
        gpu.sync()
        assert torch.isfinite(e).all()
    else:
        with pytest.raises(P.FnError, match="NUMERIC"):
            gpu.sync()
        assert not torch.isfinite(e).any()
    assert torch.equal(sg, sv)
    assert float(((lp - lv).abs() / lv.abs().clamp(min=1.0)).max()) <= 1e-4


def test_a_nan_parameter_is_reported():
    need_gpu()
    sysm, ans = W.lih(1), W.Ansatz(3, 128, 16, 4, "aniso")
    net, gpu = make_pair(sysm, ans, 1)
    p = oracle_params(net, 2, 0.05).astype(np.float32)
    ansatz.unpack(net, p)["V1"][7, 3] = np.nan
    r, _ = mcmc.init_walkers(sysm.nuclei, sysm.charges, sysm.n_up, sysm.n_down, sysm.partial_charges, 20, 3, 0.8,
                             dtype=np.float32)
    e, lp, _ = gpu.local_energy(to_dev(p, torch.float32), to_dev(r, torch.float32))
    with pytest.raises(P.FnError, match="NUMERIC"):
        gpu.sync()
    assert torch.isnan(e).all() and torch.isnan(lp).all()

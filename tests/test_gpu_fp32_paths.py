"""FP32 energies with h1 a multiple of 128 on both of their paths: the tensor cores, and the FMA pipe that
a handle takes where those kernels cannot run (FN_LAYER_KERNEL=fma when it is created).  Bounds of the
FP32 tests: relative to the terms that E_L is a difference of, max(1, |E_L|, (|grad log psi|^2 + |lap
log psi|) / 2), every walker 1e-4 and the median 5e-6; log|psi| 1e-4 of max(1, |log|psi||).  The handle
without the tensor cores has no three-part weights in its workspace."""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import ansatz, mcmc
from gpu_helpers import make_pair, need_gpu, oracle_params, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("make,ans,B", [
    (lambda: W.lih(1), W.Ansatz(3, 128, 9, 5, "aniso"), 301),
    (W.n2, W.Ansatz(2, 256, 32, 3, "iso"), 45),
    (W.hydrogen_atom, W.Ansatz(1, 128, 8, 2, "iso"), 1),
])
def test_both_paths_against_oracle(make, ans, B, monkeypatch):
    need_gpu()
    sysm = make()
    monkeypatch.delenv("FN_LAYER_KERNEL", raising=False)
    net, tensor = make_pair(sysm, ans, 1)
    monkeypatch.setenv("FN_LAYER_KERNEL", "fma")
    _, fma = make_pair(sysm, ans, 1)
    monkeypatch.delenv("FN_LAYER_KERNEL")
    assert fma.workspace_bytes(B) < tensor.workspace_bytes(B)
    p = oracle_params(net, 2, 0.05).astype(np.float32)
    r, _ = mcmc.init_walkers(sysm.nuclei, sysm.charges, sysm.n_up, sysm.n_down, sysm.partial_charges, B, 3, 0.8,
                             dtype=np.float32)
    p64, r64 = p.astype(np.float64), r[:45].astype(np.float64)
    e_ref, lp_ref, sg_ref = ansatz.local_energy(net, p64, sysm.nuclei, sysm.charges, r64)
    _, _, grad, lap = ansatz.log_psi_derivatives(net, p64, sysm.nuclei, r64)
    scale = np.maximum(np.maximum(1.0, np.abs(e_ref)), 0.5 * (np.sum(grad * grad, -1) + np.abs(lap)))
    for gpu in (tensor, fma):
        e, lp, sg = (x.cpu().numpy()[:45] for x in gpu.local_energy(to_dev(p, torch.float32), to_dev(r, torch.float32)))
        gpu.sync()
        np.testing.assert_array_equal(sg, sg_ref)
        assert np.all(np.abs(lp - lp_ref) <= 1e-4 * np.maximum(1.0, np.abs(lp_ref)))
        err = np.abs(e - e_ref) / scale
        assert np.median(err) <= 5e-6 and np.all(err <= 1e-4), (np.median(err), err.max())

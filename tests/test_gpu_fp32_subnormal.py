"""FP32 local energies with orbitals below the normal FP32 range.

E_L does not change when every envelope weight pi is scaled by one factor.  With pi = 1e-39
the orbital values are subnormal, 3e-39 to 8e-39; their reciprocals are still FP32 numbers, so an FP32
determinant stage took them, and the FP64 one has to.  Subnormal numbers are multiples of 2^-149 =
1.4e-45: an envelope of 3e-40 is off by 2.3e-6 of itself, and so are its derivatives, E_L by a few times that
of its kinetic scale; the bound is 1e-3."""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import ansatz
from gpu_helpers import make_pair, need_gpu, oracle_params, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("make,ans", [
    (W.hydrogen_atom, W.Ansatz(2, 32, 8, 1, "iso")),
    (lambda: W.atom(2, 1), W.Ansatz(2, 128, 8, 2, "iso")),
])
def test_subnormal_orbitals_keep_their_energy(make, ans):
    need_gpu()
    sysm = make()
    net, gpu = make_pair(sysm, ans, 1)
    p = oracle_params(net, 3, 0.02).astype(np.float32)
    d = ansatz.unpack(net, p)                             # views of p
    d["w_up"][:] = np.abs(d["w_up"])
    d["g_up"][:] = 14.0                                   # no zero of an orbital near the walkers
    r = (0.5 + 0.2 * np.random.default_rng(0).random((64, 1, 3))).astype(np.float32)
    e_ref, _, _ = ansatz.local_energy(net, p.astype(np.float64), sysm.nuclei, sysm.charges, r.astype(np.float64))
    _, _, grad, lap = ansatz.log_psi_derivatives(net, p.astype(np.float64), sysm.nuclei, r.astype(np.float64))
    scale = np.maximum(np.maximum(1.0, np.abs(e_ref)), 0.5 * (np.sum(grad * grad, -1) + np.abs(lap)))
    scaled = p.copy()
    ansatz.unpack(net, scaled)["pi_up"][:] = p.dtype.type(1e-39) * d["pi_up"]
    e, lp, sg = gpu.local_energy(to_dev(scaled, torch.float32), to_dev(r, torch.float32))
    gpu.sync()
    assert np.all(np.abs(e.cpu().numpy() - e_ref) <= 1e-3 * scale)
    assert torch.isfinite(lp).all() and torch.all(sg == 1)

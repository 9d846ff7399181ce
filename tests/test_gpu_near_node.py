"""FP32 mode next to a node of one determinant: the determinant stage runs in FP64 there, so the
error of a local energy is that of its FP32 inputs and does not grow with the inverse of
the vanishing determinant.

He+ with two determinants, psi = phi_1 + phi_2: the walker is moved along a line to a zero of phi_1
(by bisection in FP64) while psi stays of order one, then displaced by 10^-k bohr.  E_L is a smooth
function there; FP32 products and sums of a few hundred terms with factors of order one leave at
most 1e-4 of the kinetic scale (the bound of the other FP32 tests), at every distance.  With the
cancelling terms 1/d^2 formed in FP32 the error would be 6e-8 / d^2 times the other terms: 6 at
d = 1e-4."""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import ansatz
from gpu_helpers import make_pair, need_gpu, oracle_params, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()
    yield
    torch.cuda.synchronize()


@pytest.mark.parametrize("h1", [32, 128])            # FMA-pipe and tensor-core stream layers
def test_local_energy_beside_a_zero_of_one_determinant(h1):
    sysm = W.atom(2, 1)
    ans = W.Ansatz(2, h1, 8, 2, "iso")
    net, gpu = make_pair(sysm, ans, 1)
    p = oracle_params(net, 3, 0.05).astype(np.float32)
    d = ansatz.unpack(net, p)                         # views of p

    def phi1(x):
        r = np.array([[[x, 0.3, -0.2]]])
        return ansatz.orbital_matrices(net, p.astype(np.float64), sysm.nuclei, r)[0][0, 0, 0, 0]

    # a bias that puts the zero of phi_1 between x = 0.5 and x = 1
    base = d["g_up"][0]
    lo, hi = 0.5, 1.0
    env = lambda x: np.exp(-abs(float(d["sigma_up"][0, 0])) * np.sqrt(x * x + 0.13)) * float(d["pi_up"][0, 0])
    mid = phi1(0.75) / env(0.75)
    d["g_up"][0] = np.float32(base - mid)
    assert phi1(lo) * phi1(hi) < 0
    for _ in range(60):
        m = 0.5 * (lo + hi)
        lo, hi = (m, hi) if phi1(lo) * phi1(m) > 0 else (lo, m)
    xs = lo + np.array([1e-1, 1e-2, 1e-3, 1e-4, 1e-5])
    r = np.stack([xs, np.full(5, 0.3), np.full(5, -0.2)], -1)[:, None, :].astype(np.float32)
    e, _, _ = gpu.local_energy(to_dev(p, torch.float32), to_dev(r, torch.float32))
    gpu.sync()
    r64, p64 = r.astype(np.float64), p.astype(np.float64)
    e_ref, _, _ = ansatz.local_energy(net, p64, sysm.nuclei, sysm.charges, r64)
    _, _, grad, lap = ansatz.log_psi_derivatives(net, p64, sysm.nuclei, r64)
    scale = np.maximum(np.maximum(1.0, np.abs(e_ref)), 0.5 * (np.sum(grad * grad, -1) + np.abs(lap)))
    err = np.abs(e.cpu().numpy() - e_ref) / scale
    assert np.all(err <= 1e-4), err

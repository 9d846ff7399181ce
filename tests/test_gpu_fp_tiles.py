"""FP32 and FP64 stream layers, orbitals and mean-field products at the edges of their tiles,
against the oracle.

The FMA-pipe kernels choose between a 128-row and a 32-row tile and between 16-byte and
single-element copies; the FP32 local-energy pass with h1 a multiple of 128 runs on the
tensor cores with every operand split into three BF16 parts.  The cases are a width that no
vector copy fits (33), a partial column tile (72), the large tile with a ragged last row tile,
one and two 128-column tiles, a spin with no electrons, and a contraction that is not a
multiple of 8.

Bounds: FP64 1e-8 of max(1, |E_L|) and 1e-10 in log|psi|.  FP32: 24-bit products and sums, so
relative to the terms that E_L is a difference of, max(1, |E_L|, (|grad log psi|^2 +
|lap log psi|) / 2), the rounding of a few hundred operations amplified by the conditioning of
the determinants: 1e-4, as the other FP32 tests; for log|psi| 1e-4 of max(1, |log|psi||).  A split
that lost its third part would be off by 2^-17 per product (7.6e-6, times the same
amplification); the median error over the walkers is therefore held to 5e-6 of the same
scale."""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import ansatz, mcmc
from gpu_helpers import make_pair, need_gpu, oracle_params, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()
    yield
    torch.cuda.synchronize()


CASES = [
    # system, ansatz, walkers
    (lambda: W.lih(0), W.Ansatz(3, 33, 7, 3, "aniso"), 45),
    (lambda: W.lih(0), W.Ansatz(3, 72, 16, 2, "iso"), 3301),
    (lambda: W.lih(1), W.Ansatz(3, 128, 9, 5, "aniso"), 301),
    (lambda: W.n2(), W.Ansatz(2, 256, 32, 3, "aniso"), 77),
    (W.hydrogen_atom, W.Ansatz(2, 128, 8, 2, "iso"), 131),
]


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("make,ans,B", CASES)
def test_tile_edges_against_oracle(make, ans, B, prec):
    sysm = make()
    net, gpu = make_pair(sysm, ans, prec)
    npdt, dt = (np.float64, torch.float64) if prec == 0 else (np.float32, torch.float32)
    p = oracle_params(net, 2, 0.05).astype(npdt)
    r, _ = mcmc.init_walkers(sysm.nuclei, sysm.charges, sysm.n_up, sysm.n_down, sysm.partial_charges, B, 3, 0.8,
                             dtype=npdt)
    e, lp, sg = (x.cpu().numpy() for x in gpu.local_energy(to_dev(p, dt), to_dev(r, dt)))
    lp2, sg2 = (x.cpu().numpy() for x in gpu.log_psi(to_dev(p, dt), to_dev(r, dt)))
    gpu.sync()
    # walkers are independent: the oracle takes the first and last ones and some between
    idx = np.unique(np.concatenate([np.arange(min(B, 12)), np.arange(max(0, B - 12), B), np.arange(0, B, 1 + B // 24)]))
    p64, r64 = p.astype(np.float64), r[idx].astype(np.float64)
    e_ref, lp_ref, sg_ref = ansatz.local_energy(net, p64, sysm.nuclei, sysm.charges, r64)
    np.testing.assert_array_equal(sg[idx], sg_ref)
    np.testing.assert_array_equal(sg2[idx], sg_ref)
    if prec == 0:
        for got in (lp, lp2):
            np.testing.assert_allclose(got[idx], lp_ref, rtol=0, atol=1e-10)
        assert np.all(np.abs(e[idx] - e_ref) <= 1e-8 * np.maximum(1.0, np.abs(e_ref)))
        return
    for got in (lp, lp2):
        assert np.all(np.abs(got[idx] - lp_ref) <= 1e-4 * np.maximum(1.0, np.abs(lp_ref)))
    _, _, grad, lap = ansatz.log_psi_derivatives(net, p64, sysm.nuclei, r64)
    scale = np.maximum(np.maximum(1.0, np.abs(e_ref)), 0.5 * (np.sum(grad * grad, -1) + np.abs(lap)))
    err = np.abs(e[idx] - e_ref) / scale
    assert np.median(err) <= 5e-6 and np.all(err <= 1e-4), (np.median(err), err.max())

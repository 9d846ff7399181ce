"""FP32 value pass: sums in two levels, and the energy gradient that rests on them.

A contraction of k terms is summed in stages of 16 whose results are added up.  One electron
with layer outputs that are exactly 1 (tanh 20 in FP32) shows it: a row of weights 1, 2^-25, 2^-25,
... sums to 1 + (k - 1) 2^-25, but in one FP32 chain each 2^-25 is below half a unit of the running
sum and is lost, 7.6e-6 for k = 256.  In two levels only the 15 of the first stage are, 4.5e-7, and the
ragged last stage rounds once, 6e-8.  FP32 log (of mantissa and exponent) adds 1.2e-7.
  orbitals:      log|psi| = log(sum), bound 8e-7;
  layer, mean field:  log|psi| = log(1 + tanh(sum)), where the sum's error enters times
                 sech^2(1) / (1 + tanh 1) = 0.24 and tanh, its sum with the residual and log add
                 2.3e-7: bound 6e-7, against 1.8e-6 of one chain.

Gradient: relative to FP64 mode on the same parameters and walkers.  The entries of the orbital
matrices carry about 3e-7 (two sums of 16 terms, tanh and exp of two units each, per layer); a
determinant multiplies that by the inverse of its normalised matrix, weighed with its share of psi.
Walkers are kept where that factor is at most 10 (the 7 x 7 blocks of N2: 100), so a walker's term
is off by 3e-6 (3e-5) of itself.  Walkers' errors are independent, as are their terms in a sum with
random energies: 3e-6 (3e-5) of the norm of the gradient, and 1e-6 times the factor's limit leaves a
factor of three."""
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


@pytest.mark.parametrize("B", [40, 30000])               # small and large row tiles
@pytest.mark.parametrize("h1", [256, 250])               # vector and single-element copies
@pytest.mark.parametrize("where", ["orbitals", "layer", "mean field"])
def test_small_terms_of_a_long_sum_are_kept(where, h1, B):
    sysm = W.hydrogen_atom()
    net, gpu = make_pair(sysm, W.Ansatz(1 if where == "orbitals" else 2, h1, 8, 1, "iso"), 1)
    p = np.zeros(ansatz.param_count(net))
    d = ansatz.unpack(net, p)                             # views of p
    d["b0"][:] = 20.0
    d["pi_up"][:] = 1.0
    row = np.full(h1, 2.0 ** -25)
    row[0] = 1.0
    if where == "orbitals":
        d["w_up"][0] = row
        bound = 8e-7
    else:
        lo = 0 if where == "layer" else h1                # columns of h, or of the spin-up mean of h
        d["V1"][:, lo:lo + h1] = row
        d["w_up"][0, 0] = 1.0
        bound = 6e-7
    r = np.random.default_rng(0).normal(size=(B, 1, 3))
    r = r.astype(np.float32)
    lp, sign = gpu.log_psi(to_dev(p, torch.float32), to_dev(r, torch.float32))
    gpu.sync()
    ref, _ = ansatz.log_psi(net, p, sysm.nuclei, r[:1].astype(np.float64))
    assert torch.all(sign == 1)
    assert float((lp - ref[0]).abs().max()) <= bound


@pytest.mark.parametrize("make,ans,B,limit", [
    (lambda: W.lih(1), W.Ansatz(4, 128, 16, 8, "aniso"), 4096, 10.0),
    (lambda: W.lih(-1), W.Ansatz(4, 128, 16, 8, "aniso"), 4096, 10.0),
    (W.n2, W.Ansatz(3, 256, 32, 4, "aniso"), 512, 100.0),
])
def test_fp32_gradient_off_the_nodes(make, ans, B, limit):
    sysm = make()
    net, g32 = make_pair(sysm, ans, 1)
    _, g64 = make_pair(sysm, ans, 0)
    p = oracle_params(net, 5, 0.02).astype(np.float32)
    r, _ = mcmc.init_walkers(sysm.nuclei, sysm.charges, sysm.n_up, sysm.n_down, sysm.partial_charges, B, 8, 0.8,
                             dtype=np.float32)
    mats = [m for m in ansatz.orbital_matrices(net, p.astype(np.float64), sysm.nuclei, r.astype(np.float64))
            if m.shape[-1]]
    det = np.prod([np.linalg.det(m) for m in mats], axis=0)
    share = np.abs(det) / np.abs(det.sum(-1, keepdims=True))
    factor = sum((share * np.sqrt((np.linalg.inv(m / np.linalg.norm(m, axis=-2, keepdims=True)) ** 2).sum((-1, -2)))).max(-1)
                 for m in mats)
    r = r[factor <= limit]
    assert r.shape[0] >= 64
    e = torch.as_tensor(np.random.default_rng(2).normal(-8.0, 1.0, r.shape[0])).cuda()
    a, _ = g32.energy_grad(to_dev(p, torch.float32), to_dev(r, torch.float32), e)
    b, _ = g64.energy_grad(to_dev(p, torch.float64), to_dev(r, torch.float64), e)
    g32.sync()
    g64.sync()
    assert float((a.double() - b).norm() / b.norm()) <= 1e-6 * limit

"""BF16 mode and the energy gradient where their tilings have edges.

Orbital row tiles hold the electrons of one spin, as many walker tiles together as fill them and
the chip; features and derivative terms put several walkers in a CTA; the pair kernels read odd
widths element by element.  None of it may depend on what else is in the batch: a walker's
log|psi| and sign have the same bits alone, in a small batch and in a large one (the roundings of
E_L's BF16 tangents are a function of the batch size), and E_L those of its copies in the same
batch.  Accuracy is held to the bounds of the BF16 tests (median 1e-2 of the kinetic scale and of
log|psi|).

Gradients: widths that no 16-byte copy fits (33, 7), against the FP64 oracle along a random
direction v.  Bounds relative to sum_w |c_w| |v . grad log|psi_w||-like term sums are those of the
other gradient tests: FP64 1e-5 of max(1, |d|); FP32 1e-3 and BF16 3e-2 of |g| (errors of
independent sign along a unit vector cannot exceed the norm of the error)."""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import ansatz, grad, mcmc
from gpu_helpers import make_pair, need_gpu, oracle_params, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()
    yield
    torch.cuda.synchronize()


def _walkers(net, p, sysm, B):
    r, _ = mcmc.init_walkers(sysm.nuclei, sysm.charges, sysm.n_up, sysm.n_down, sysm.partial_charges, B, 5, 0.8)
    lp0, _ = ansatz.log_psi(net, p, sysm.nuclei, r)
    r, _, _ = mcmc.metropolis(net, p, sysm.nuclei, r, lp0, 6, 60, 0.3)
    return r.astype(np.float32)


@pytest.mark.parametrize("make,ans", [
    (W.hydrogen_atom, W.Ansatz(2, 64, 9, 3, "iso")),            # one spin empty, no pairs
    (W.h2, W.Ansatz(2, 32, 7, 1, "aniso")),                     # 64 walkers to a tile, odd pair width
    (lambda: W.lih(-1), W.Ansatz(3, 64, 9, 5, "aniso")),        # 3 + 2 electrons, ragged column tile
    (lambda: W.atom(14, -1), W.Ansatz(2, 128, 16, 16, "aniso")),    # 9 + 6 electrons, two column tiles of one spin
    (W.n2, W.Ansatz(2, 64, 16, 3, "iso")),
])
def test_walkers_do_not_depend_on_the_batch(make, ans):
    sysm = make()
    net, gpu = make_pair(sysm, ans, 2)
    p = oracle_params(net, 0, 0.0).astype(np.float32).astype(np.float64)
    r = _walkers(net, p, sysm, 24)
    pd, n = to_dev(p, torch.float32), 2801
    big = to_dev(np.tile(r, (n // 24 + 1, 1, 1))[:n], torch.float32)

    def both(w):
        e, lp, sg = gpu.local_energy(pd, w)
        lv, sv = gpu.log_psi(pd, w)
        gpu.sync()
        assert torch.equal(sg, sv)
        return e.clone(), lp.clone(), lv.clone()

    whole = both(big)
    for lo, hi in ((0, 1), (3, 8), (0, 24), (13, 410)):
        for a, b in zip(both(big[lo:hi].contiguous())[1:], whole[1:]):
            assert torch.equal(a, b[lo:hi])
    for lo in (24, 1200, 2736):
        assert torch.equal(whole[0][:24], whole[0][lo:lo + 24])
    e, lp = (x[:24].cpu().numpy() for x in whole[:2])
    r64 = r.astype(np.float64)
    e_ref, lp_ref, _ = ansatz.local_energy(net, p, sysm.nuclei, sysm.charges, r64)
    _, _, g, lap = ansatz.log_psi_derivatives(net, p, sysm.nuclei, r64)
    scale = np.maximum(np.maximum(1.0, np.abs(e_ref)), 0.5 * (np.sum(g * g, -1) + np.abs(lap)))
    assert np.median(np.abs(e - e_ref) / scale) < 1e-2
    assert np.median(np.abs(lp - lp_ref)) < 1e-2


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("make,ans,B", [
    (lambda: W.lih(0), W.Ansatz(3, 33, 7, 3, "aniso"), 45),
    (lambda: W.lih(1), W.Ansatz(2, 96, 9, 2, "iso"), 131),
])
def test_gradient_at_odd_widths(make, ans, B, prec):
    if prec == 2 and ans.h1 % 32:
        pytest.skip("the BF16 mode takes widths that are multiples of 32")
    sysm = make()
    net, gpu = make_pair(sysm, ans, prec)
    p = oracle_params(net, 1, 0.02).astype(np.float32).astype(np.float64)
    r = _walkers(net, p, sysm, B).astype(np.float64)
    e = np.random.default_rng(7).normal(-8.0, 1.0, B)
    dt = torch.float64 if prec == 0 else torch.float32
    g, mean = gpu.energy_grad(to_dev(p, dt), to_dev(r, dt), torch.as_tensor(e).cuda())
    gpu.sync()
    g = g.cpu().numpy().astype(np.float64)
    assert abs(float(mean.item()) - e.mean()) < 1e-12
    for k in range(2):
        v = np.random.default_rng(20 + k).standard_normal(p.shape[0])
        v /= np.linalg.norm(v)
        d = grad.directional_richardson(net, p, sysm.nuclei, r, e, v, h=1e-5)
        bound = 1e-5 * max(1.0, abs(d)) if prec == 0 else (1e-3, 3e-2)[prec - 1] * np.linalg.norm(g)
        assert abs(g @ v - d) <= bound, (g @ v, d, bound)

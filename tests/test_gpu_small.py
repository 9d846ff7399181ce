"""FP64 value pass and Metropolis chain of small networks, which run in one kernel, against the
oracle over the forms that kernel takes: up to 8 electrons, 64 columns and 16 determinants, one
spin empty, unequal spins, a pair width below the 4 input features, one layer, both envelopes,
walker counts that do not fill the last CTA, an offset batch.

log|psi| within 1e-10 (the FP64 bound of the other tests).  A chain's proposals are the oracle's
bit for bit, so every walker that took the same decisions is equal to rounding of the sum r + s z
(none: 1e-14); decisions agree unless |log U - A| < 1e-9, which no step of these seeds meets."""
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


def _spin(sysm, up, dn):
    return W.System(sysm.name, sysm.nuclei, sysm.charges, up, dn, None)


CASES = [
    # system, ansatz, walkers
    (W.hydrogen_atom, W.Ansatz(1, 8, 1, 1, "iso"), 1),
    (W.h2, W.Ansatz(2, 32, 8, 1, "iso"), 257),
    (lambda: _spin(W.lih(0), 4, 0), W.Ansatz(3, 24, 2, 3, "aniso"), 33),
    (lambda: W.lih(-1), W.Ansatz(3, 64, 32, 16, "aniso"), 50),
    (lambda: _spin(W.atom(8, 0), 5, 3), W.Ansatz(2, 40, 5, 2, "aniso"), 19),
    (lambda: _spin(W.atom(8, 0), 8, 0), W.Ansatz(2, 16, 4, 2, "iso"), 9),
]


@pytest.mark.parametrize("make,ans,B", CASES)
def test_value_and_chain(make, ans, B):
    sysm = make()
    net, gpu = make_pair(sysm, ans, 0)
    p = oracle_params(net, 5, 0.05)
    r, _ = mcmc.init_walkers(sysm.nuclei, sysm.charges, sysm.n_up, sysm.n_down, None, B, 4, 0.8)
    pd, rd = to_dev(p, torch.float64), to_dev(r, torch.float64)
    lp, sg = gpu.log_psi(pd, rd)
    lp_ref, sg_ref = ansatz.log_psi(net, p, sysm.nuclei, r)
    np.testing.assert_allclose(lp.cpu().numpy(), lp_ref, rtol=0, atol=1e-10)
    np.testing.assert_array_equal(sg.cpu().numpy(), sg_ref)
    acc = torch.zeros(1, dtype=torch.int64, device="cuda")
    gpu.set_walker_offset(11)
    gpu.mcmc_steps(pd, rd, lp, 6, 0.15, 77, step_offset=2 ** 32 - 3, accept_count=acc)
    gpu.sync()
    r_ref, lp_end, taken = mcmc.metropolis(net, p, sysm.nuclei, r, lp_ref, 77, 6, 0.15, step_offset=2 ** 32 - 3,
                                           walker_offset=11)
    assert int(acc) == int(taken.sum())
    np.testing.assert_allclose(rd.cpu().numpy(), r_ref, rtol=0, atol=1e-14)
    np.testing.assert_allclose(lp.cpu().numpy(), lp_end, rtol=0, atol=1e-10)


def test_chain_split_over_launches_is_one_chain():
    """600 steps run as three launches; they equal 600 calls of one step, bit for bit."""
    sysm, ans = W.h2(), W.Ansatz(2, 16, 4, 1, "iso")
    net, gpu = make_pair(sysm, ans, 0)
    pd = to_dev(oracle_params(net, 5, 0.05), torch.float64)
    r0, _ = gpu.init_walkers(5, 3, 1.0)
    lp0, _ = gpu.log_psi(pd, r0)
    ra, la, rb, lb = r0.clone(), lp0.clone(), r0.clone(), lp0.clone()
    gpu.mcmc_steps(pd, ra, la, 600, 0.3, 9)
    for k in range(600):
        gpu.mcmc_steps(pd, rb, lb, 1, 0.3, 9, step_offset=k)
    gpu.sync()
    assert torch.equal(ra, rb) and torch.equal(la, lb)

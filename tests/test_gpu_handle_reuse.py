"""BF16 local energies do not depend on what a handle computed before, nor on the batch.

The slabs of a layer input lie at multiples of the padded row count, so a call with another batch
size finds earlier data in its place.  Every value that the layer products read has to be written by
the call itself: a handle that has served other batch sizes, value passes and gradients returns the
bits of a fresh handle, and walkers in a smaller batch the bits they have in a larger one.  The
widths are those where the low parts of the pair columns share a block of 64 columns with h: 32 and
96 in every layer, any in layer 0."""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import mcmc
from gpu_helpers import make_pair, need_gpu, oracle_params, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()
    yield
    torch.cuda.synchronize()


@pytest.mark.parametrize("make,ans", [
    (lambda: W.lih(-1), W.Ansatz(3, 32, 8, 2, "aniso")),
    (lambda: W.lih(-1), W.Ansatz(2, 64, 16, 3, "iso")),
    (lambda: W.atom(6), W.Ansatz(3, 96, 7, 2, "iso")),
    (W.h2, W.Ansatz(2, 128, 16, 2, "aniso")),
])
def test_energies_of_a_used_handle_are_those_of_a_fresh_one(make, ans):
    sysm = make()
    net, used = make_pair(sysm, ans, 2)
    p = to_dev(oracle_params(net, 0, 0.02), torch.float32)
    r, _ = mcmc.init_walkers(sysm.nuclei, sysm.charges, sysm.n_up, sysm.n_down, sysm.partial_charges, 2801, 5, 0.8,
                             dtype=np.float32)
    r = to_dev(r, torch.float32)
    whole = None
    for B in (2801, 397, 24, 1650, 2801, 1):
        w = r[:B].contiguous()
        e, lp, sg = used.local_energy(p, w)
        used.sync()
        fresh = make_pair(sysm, ans, 2)[1]
        ef, lpf, sgf = fresh.local_energy(p, w)
        fresh.sync()
        assert torch.equal(e, ef) and torch.equal(lp, lpf) and torch.equal(sg, sgf)
        whole = e if whole is None else whole
        assert torch.equal(e, whole[:B])
        v = r[:max(1, B // 2)].contiguous()               # other passes in between
        used.log_psi(p, v)
        used.energy_grad(p, v, e[:v.shape[0]].contiguous())

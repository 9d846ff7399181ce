"""Device memory of FP32 and FP64 calls: the projections that the derivative terms of the envelopes read
share the gradient's buffers, so a batch takes what it took without them (the bytes below), and FP32 with
h1 a multiple of 128 the three-part BF16 weights more.  Energies and gradients that alternate on one
handle, at several batch sizes, are those of handles that only do the one."""
import pytest
import torch

import workloads as W
from gpu_helpers import make_pair, need_gpu, oracle_params, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("make,ans,fp64,fp32", [
    (W.n2, W.Ansatz(4, 256, 32, 16, "aniso"), 32271938816, 16138058496),
    (lambda: W.lih(0), W.Ansatz(4, 128, 16, 8, "aniso"), 1779405568, 890231552),
    (W.h2, W.Ansatz(2, 32, 8, 1, "aniso"), 98646016, 49390080),
    (W.n2, W.Ansatz(3, 64, 16, 16, "aniso"), 9103694080, 4552045824),
])
def test_workspace_of_4096_walkers(make, ans, fp64, fp32):
    need_gpu()
    sysm = make()
    net, g64 = make_pair(sysm, ans, 0)
    assert g64.workspace_bytes(4096) <= fp64
    split = 0
    if ans.h1 % 128 == 0:
        up = lambda n: -(-n // 64) * 64
        for l in range(ans.n_layers):
            d_h, d_g = (4 * len(sysm.charges), 4) if l == 0 else (ans.h1, ans.h2)
            split += 2 * ans.h1 * 3 * (up(d_h + 2 * d_g) + up(2 * d_h))
        split += 2 * ans.n_dets * net.n_el * 3 * ans.h1 + 256
    assert make_pair(sysm, ans, 1)[1].workspace_bytes(4096) <= fp32 + split


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("make,ans", [
    (lambda: W.lih(-1), W.Ansatz(3, 128, 9, 3, "aniso")),
    (W.h2, W.Ansatz(2, 40, 8, 2, "iso")),
    (lambda: W.atom(6), W.Ansatz(1, 24, 4, 16, "iso")),          # projections larger than the gradient's buffers
])
def test_energies_and_gradients_alternate(make, ans, prec):
    need_gpu()
    sysm = make()
    net, both = make_pair(sysm, ans, prec)
    dt = torch.float64 if prec == 0 else torch.float32
    p = to_dev(oracle_params(net, 0, 0.02), dt)
    r, _ = both.init_walkers(300, 5, 0.8)
    eps = 2.0 ** -52 if prec == 0 else 2.0 ** -23
    for B in (300, 37, 111, 300):
        w = r[:B].contiguous()
        e, lp, _ = both.local_energy(p, w)
        g, _ = both.energy_grad(p, w, e)
        only_e, only_g = make_pair(sysm, ans, prec)[1], make_pair(sysm, ans, prec)[1]
        e1, lp1, _ = only_e.local_energy(p, w)
        g1, _ = only_g.energy_grad(p, w, e)
        torch.cuda.synchronize()
        assert torch.equal(e, e1) and torch.equal(lp, lp1)
        # the sums over walkers end in atomic additions of a few hundred partial sums
        assert float((g - g1).norm()) <= 300 * eps * float(g1.norm())

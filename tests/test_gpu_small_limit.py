"""Where FP64 passes of small networks leave the single-kernel path for the general one: by walkers, above
two electrons (four at 16 columns).  The path shows in the profile (only the general one has a feature kernel).
Across the limit log|psi| agrees within 1e-10, the FP64 bound of the other tests, and a Metropolis chain
takes the same decisions: proposals have the same bits, so walkers agree to rounding of r + s z, 1e-14."""
import pytest
import torch

import workloads as W
from gpu_helpers import make_pair, need_gpu, oracle_params, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("make,ans,limit", [
    (lambda: W.lih(0), W.Ansatz(2, 32, 8, 1, "iso"), 3072),
    (lambda: W.lih(1), W.Ansatz(3, 40, 8, 2, "aniso"), 4096),
    (lambda: W.atom(8), W.Ansatz(2, 16, 8, 1, "aniso"), 8192),
    (lambda: W.lih(0), W.Ansatz(2, 16, 8, 1, "aniso"), None),
    (W.h2, W.Ansatz(2, 32, 8, 1, "iso"), None),
])
def test_path_by_walkers(make, ans, limit):
    need_gpu()
    sysm = make()
    net, gpu = make_pair(sysm, ans, 0)
    p = to_dev(oracle_params(net, 5, 0.02), torch.float64)
    most = limit or 20000
    r, _ = gpu.init_walkers(most + 1, 3, 0.8)
    out = []
    for B in (most, most + 1):
        w = r[:B].clone()
        gpu.profile_enable(True)
        lp, sg = gpu.log_psi(p, w)
        first = lp.clone()
        gpu.mcmc_steps(p, w, lp, 3, 0.1, 9)
        gpu.sync()
        general = "features" in gpu.profile_read()
        gpu.profile_enable(False)
        assert general == (limit is not None and B > limit)
        out.append((first[:most], sg[:most], w[:most], lp[:most]))
    (l0, s0, w0, e0), (l1, s1, w1, e1) = out
    assert torch.equal(s0, s1)
    assert float((l0 - l1).abs().max()) <= 1e-10 and float((e0 - e1).abs().max()) <= 1e-10
    assert float((w0 - w1).abs().max()) <= 1e-14

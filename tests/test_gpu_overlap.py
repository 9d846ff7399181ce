"""Overlapped launches change no bits: the same calls in two fresh processes, one as usual and one
with CUDA_LAUNCH_BLOCKING=1 (each kernel ends before the next is launched).  The sizes are those whose
launches overlap: value passes and Metropolis chains, and energies of few rows.  None of these calls
adds with float atomics, so walkers, log|psi| and E_L have to agree bit for bit."""
import os
import subprocess
import sys

import pytest

from gpu_helpers import need_gpu

pytestmark = pytest.mark.gpu
ROOT = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..")

CHILD = r"""
import hashlib, sys
import torch
import workloads as W
import paper_2401_10287_gb300 as P

def digest(*xs):
    return hashlib.sha256(b"".join(x.cpu().numpy().tobytes() for x in xs)).hexdigest()

for sysm, ans, prec, B, steps in [
        (W.lih(0), W.Ansatz(4, 128, 16, 8, "aniso"), P.BF16_MIXED, 4096, 400),
        (W.lih(0), W.Ansatz(4, 128, 16, 8, "aniso"), P.FP32, 1024, 100),
        (W.atom(6), W.Ansatz(4, 256, 32, 16, "aniso"), P.BF16_MIXED, 256, 200),
        (W.h2(), W.Ansatz(2, 32, 8, 1, "iso"), P.BF16_MIXED, 700, 200)]:
    s = P.System(sysm.nuclei, sysm.charges, sysm.n_up, sysm.n_down, P.NetConfig.from_ansatz(ans, prec))
    p = s.init_params(3)
    r, _ = s.init_walkers(B, 5, 0.8)
    lp, _ = s.log_psi(p, r)
    n = torch.zeros(1, dtype=torch.int64, device="cuda")
    s.mcmc_steps(p, r, lp, steps, 0.1, 7, accept_count=n)
    e, lpe, sg = s.local_energy(p, r)
    s.sync()
    assert 0 < int(n) < steps * B
    print(digest(r, lp, n, e, lpe, sg))
"""


def test_overlapped_and_blocking_launches_agree_bit_for_bit():
    need_gpu()
    out = []
    for blocking in ("0", "1"):
        env = dict(os.environ, CUDA_LAUNCH_BLOCKING=blocking)
        res = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=env, capture_output=True, text=True,
                             timeout=300)
        assert res.returncode == 0, res.stderr[-2000:]
        out.append(res.stdout.split())
    assert len(out[0]) == 4 and out[0] == out[1]

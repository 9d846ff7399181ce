"""The calls whose speed matters to a program that uses this package, as measurable cases.

The package is the hot path of variational Monte Carlo with a FermiNet-style wavefunction:
sample walkers, evaluate log|psi| and exact local energies, form the energy gradient, update
the parameters.  The cases are these calls on the systems and network sizes of the
repository's own workloads, in the three precision modes, from one optimiser update to the
largest local-energy call.

Values come back from the library in double in every mode.  A case returns them in the type
of the mode's parameters (as ``EnergyGrad`` does with the mean energy): double in FP64 mode,
single in FP32 and BF16-mixed mode, which is what a program in that mode keeps.

Inputs are made with torch alone from the seed: parameters with the library's initial
distribution plus a perturbation (so that no two envelopes are alike), and walkers moved by
an FP32 Metropolis chain on |psi|^2 of those parameters, written here, so that they lie
where a sampler's walkers lie; the few nearest to a node, of the sum or of one determinant
in it, are left out, because there rounding alone decides the leading digits of an FP32
energy.  ``exact`` computes the same quantities in FP64 with torch.
"""
import math

import torch

import paper_2401_10287_gb300 as fn

SYMBOLS = ("", "H", "He", "Li", "Be", "B", "C", "N", "O", "F", "Ne", "Na", "Mg", "Al", "Si")
DIATOMICS = {  # Z, Z, bond length (bohr), centred on the origin
    "H2": (1, 1, 1.4, True), "N2": (7, 7, 2.068, True), "CO": (6, 8, 2.132, True), "LiH": (3, 1, 3.015, False),
}
CION = {"LiH+": (2, 1), "LiH-": (4, 1)}      # electrons per nucleus of the diatomic ions
MODES = {"fp64": fn.FP64, "fp32": fn.FP32, "bf16": fn.BF16_MIXED}


def listed():
    big = dict(layers=4, h1=256, h2=32, dets=16, aniso=True)      # N2 workload and serving network
    ion = dict(layers=4, h1=128, h2=16, dets=8, aniso=True)       # LiH ions and the ionisation workload
    small = dict(layers=2, h1=32, h2=8, dets=1, aniso=False)      # H2 workloads
    return [
        # end of a training iteration: clipping and the Adam update (the smallest work of the list)
        dict(name="update_n2_fp32", op="update", mode="fp32", mol="N2", walkers=4096, **big),
        # one Metropolis evaluation of the smallest serving job: launches and latency count
        dict(name="log_psi_c_bf16", op="log_psi", mode="bf16", mol="C", walkers=256, **big),
        # the H2 precision reference: start, 20 Metropolis steps and E_L of few walkers, a whole FP64 call chain
        dict(name="pass_h2_fp64", op="pass", mode="fp64", mol="H2", walkers=256, steps=20, **small),
        # one training iteration of the ionisation-potential workload (10 Metropolis steps, E_L, gradient, Adam)
        dict(name="train_lih_bf16", op="train", mode="bf16", mol="LiH", walkers=4096, steps=10, **ion),
        # what a Metropolis step of the large workload costs
        dict(name="log_psi_n2_bf16", op="log_psi", mode="bf16", mol="N2", walkers=4096, **big),
        # the headline call: exact local energies of the large workload in the mixed mode
        dict(name="energy_n2_bf16", op="energy", mode="bf16", mol="N2", walkers=4096, **big),
        # the same call in FP32, the largest work of the list
        dict(name="energy_n2_fp32", op="energy", mode="fp32", mol="N2", walkers=4096, **big),
        # a serving job's energy: the largest atom of the stream, an odd number of walkers and unequal spins
        dict(name="energy_si_anion_bf16", op="energy", mode="bf16", mol="Si-", walkers=1031, **big),
        # the ion workload, an open shell in FP32
        dict(name="energy_lih_anion_fp32", op="energy", mode="fp32", mol="LiH-", walkers=4096, **ion),
        # the narrow network at its largest batch
        dict(name="energy_h2_bf16", op="energy", mode="bf16", mol="H2", walkers=16384, **small),
        # the gradient (value pass and reverse pass) of the large workload and of the ion workload
        dict(name="grad_n2_bf16", op="grad", mode="bf16", mol="N2", walkers=4096, **big),
        dict(name="grad_lih_cation_fp32", op="grad", mode="fp32", mol="LiH+", walkers=4096, **ion),
    ]


def draw(rng):
    op = rng.choice(["update", "log_psi", "log_psi", "pass", "train", "energy", "energy", "energy", "grad", "grad"])

    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    if op == "pass":
        mol = rng.choice(["H", "H2", "He", "LiH"])
        net = dict(layers=rng.choice([2, 3]), h1=rng.choice([16, 32, 64]), h2=rng.choice([8, 16]),
                   dets=rng.choice([1, 2, 4]), aniso=rng.random() < 0.5)
        return dict(op=op, mode="fp64", mol=mol, walkers=spread(64, 1024), steps=rng.randint(5, 20), **net)
    if op == "train":
        net = dict(layers=4, h1=rng.choice([64, 128]), h2=16, dets=rng.choice([4, 8]), aniso=True)
        return dict(op=op, mode="bf16", mol=rng.choice(["H2", "LiH", "LiH+", "LiH-"]), walkers=spread(256, 4096),
                    steps=rng.randint(2, 10), **net)
    mode = "fp32" if op == "update" else rng.choice(["bf16", "bf16", "fp32"])
    if rng.random() < 0.5:
        mol = rng.choice(["H2", "LiH", "N2", "CO", "LiH+", "LiH-"])
    else:
        mol = SYMBOLS[rng.randint(2, 14)] + rng.choice(["", "+", "-"])
    net = rng.choice([dict(layers=4, h1=256, h2=32, dets=16, aniso=True),
                      dict(layers=4, h1=128, h2=16, dets=8, aniso=True),
                      dict(layers=3, h1=64, h2=16, dets=4, aniso=False),
                      dict(layers=2, h1=32, h2=8, dets=1, aniso=False)])
    most = 4096 if net["h1"] > 64 else 16384
    # at most the cost of 4096 walkers of the 14-electron workload (one row for each electron, coordinate and electron)
    n = sum(_counts(mol))
    if op == "energy":
        most = min(most, int(4096 * 14 * 44 / (n * (3 * n + 2))))
    return dict(op=op, mode=mode, mol=mol, walkers=spread(256, most), **net)


# --- systems and networks ---------------------------------------------------------------


def _atoms(mol):
    """(nuclei, charges) of a molecule or atom."""
    name = mol.rstrip("+-")
    if name in DIATOMICS:
        a, b, bond, centred = DIATOMICS[name]
        lo = -bond / 2 if centred else 0.0
        return [[0.0, 0.0, lo], [0.0, 0.0, lo + bond]], [a, b]
    return [[0.0, 0.0, 0.0]], [SYMBOLS.index(name)]


def _counts(mol):
    """Electrons per nucleus."""
    if mol in CION:
        return CION[mol]
    z = list(_atoms(mol)[1])
    z[0] += {"+": -1, "-": 1}.get(mol[-1], 0)
    return tuple(z)


def _spins(mol):
    n = sum(_counts(mol))
    return (n + 1) // 2, n // 2


def _electron_atoms(mol):
    """The nucleus of each electron: halves up and down per atom, flipped until the totals fit."""
    up = [(c + 1) // 2 for c in _counts(mol)]
    dn = [c // 2 for c in _counts(mol)]
    n_up = _spins(mol)[0]
    while sum(up) > n_up:
        a = max(range(len(up)), key=lambda q: (up[q] - dn[q], -q))
        up[a], dn[a] = up[a] - 1, dn[a] + 1
    return [a for a, c in enumerate(up) for _ in range(c)] + [a for a, c in enumerate(dn) for _ in range(c)]


def _layout(c):
    """(key, shape, fan-in or None) of every parameter in blob order."""
    m, h1, h2 = len(_atoms(c["mol"])[1]), c["h1"], c["h2"]
    out = []
    for l in range(c["layers"]):
        dh, dg = (4 * m, 4) if l == 0 else (h1, h2)
        out += [(("V", l), (h1, 3 * dh + 2 * dg), 3 * dh + 2 * dg), (("b", l), (h1,), 3 * dh + 2 * dg)]
        if l < c["layers"] - 1:
            out += [(("W", l), (h2, dg), dg), (("c", l), (h2,), dg)]
    rows = [c["dets"] * n for n in _spins(c["mol"])]
    for s in (0, 1):
        if rows[s]:
            out += [(("w", s), (rows[s], h1), h1), (("g", s), (rows[s],), h1)]
    for s in (0, 1):
        if rows[s]:
            out += [(("pi", s), (rows[s], m), None), (("sig", s), (rows[s], m, 3, 3) if c["aniso"] else (rows[s], m), None)]
    return out


def _unpack(c, blob):
    p, off = {}, 0
    for key, shape, _ in _layout(c):
        n = math.prod(shape)
        p[key] = blob[off:off + n].view(shape)
        off += n
    return p


def _generator(seed, stream):
    return torch.Generator(device="cuda").manual_seed(1000003 * (seed + 1) + stream)


def _dtype(c):
    return torch.float64 if c["mode"] == "fp64" else torch.float32


def _params(c, seed):
    gen, parts = _generator(seed, 1), []
    for key, shape, fan_in in _layout(c):
        z = torch.randn(math.prod(shape), generator=gen, device="cuda", dtype=torch.float64)
        if fan_in is None:
            one = torch.eye(3, dtype=torch.float64, device="cuda").expand(shape).reshape(-1) \
                if key[0] == "sig" and c["aniso"] else 1.0
            parts.append(one + 0.05 * z)
        else:
            parts.append(z / math.sqrt(fan_in))
    return torch.cat(parts).to(_dtype(c))


def _walkers(c, seed, params):
    """Walkers around their nuclei, moved by 40 Metropolis steps on |psi|^2 in single precision;
    of 1/16 more than are wanted, those with the best conditioned determinants are kept."""
    gen, b = _generator(seed, 2), c["walkers"] + c["walkers"] // 16 + 8
    nuclei, _ = _atoms(c["mol"])
    centre = torch.tensor([nuclei[a] for a in _electron_atoms(c["mol"])], dtype=torch.float32, device="cuda")
    r = centre + 0.8 * torch.randn((b,) + centre.shape, generator=gen, device="cuda")
    step = 0.5 / math.sqrt(centre.shape[0])
    p32 = params.float()
    with torch.no_grad():
        lp = _log_psi(c, p32, r)[0]
        for _ in range(40):
            new = r + step * torch.randn(r.shape, generator=gen, device="cuda")
            lp_new = _log_psi(c, p32, new)[0]
            take = torch.rand(b, generator=gen, device="cuda").log() <= 2 * (lp_new - lp)
            r = torch.where(take[:, None, None], new, r)
            lp = torch.where(take, lp_new, lp)
        mats = _orbitals(c, p32, r)
        dets = [torch.linalg.slogdet(a) for a in mats]
        log_d = sum(x[1] for x in dets)
        weight = torch.exp(log_d - lp[:, None])                             # |D_k| / |psi|
        score = 0.0
        for a in mats:
            a = a / a.norm(dim=-2, keepdim=True)
            score = score + (weight * torch.linalg.inv(a).square().sum((-1, -2))).sum(-1)
    return r[score.sort(stable=True)[1][:c["walkers"]].sort()[0]].to(_dtype(c)).contiguous()


def _energies(c, seed):
    """Local energies of an iteration under way: around the molecule's scale, with a few outliers."""
    gen = _generator(seed, 3)
    z = sum(x * x for x in _atoms(c["mol"])[1])
    e = torch.randn(c["walkers"], generator=gen, device="cuda", dtype=torch.float64)
    far = torch.rand(c["walkers"], generator=gen, device="cuda") < 0.01
    return -0.5 * z + 0.05 * z * torch.where(far, 8 * e, e)


def _moments(c, seed, n):
    """Adam's running moments of a training under way."""
    gen = _generator(seed, 4)
    m = 1e-2 * torch.randn(n, generator=gen, device="cuda", dtype=torch.float64)
    v = 1e-4 * (0.1 + torch.rand(n, generator=gen, device="cuda", dtype=torch.float64))
    return m.to(_dtype(c)), v.to(_dtype(c))


TRAIN = dict(step_size=0.1, clip_width=5.0, lr=3e-3)
ITERATION = 100      # of the training whose iteration is measured


def prepare(case, seed):
    c = case
    nuclei, charges = _atoms(c["mol"])
    up, dn = _spins(c["mol"])
    cfg = fn.NetConfig(c["layers"], c["h1"], c["h2"], c["dets"], fn.ANISO if c["aniso"] else fn.ISO, MODES[c["mode"]])
    s = dict(case=c, seed=seed, system=fn.System(nuclei, charges, up, dn, cfg), params=_params(c, seed))
    if c["op"] in ("update", "train"):
        s["m"], s["v"] = _moments(c, seed, s["params"].numel())
    if c["op"] in ("update", "grad"):
        s["e"] = _energies(c, seed)
    if c["op"] == "update":
        s["grad"] = 1e-2 * torch.randn(s["params"].numel(), generator=_generator(seed, 5), device="cuda")
    elif c["op"] != "pass":
        s["walkers"] = _walkers(c, seed, s["params"])
    if c["op"] == "train":
        s["cfg"] = fn.TrainConfig(n_mcmc_steps=c["steps"], seed=seed, **TRAIN)
        s["opt"] = torch.cat([s["m"], s["v"]])
    torch.cuda.synchronize()
    return s


def run(state):
    s, c, system = state, state["case"], state["system"]
    p, dt = s["params"], s["params"].dtype
    if c["op"] == "update":
        clipped, stats = system.clip_local_energy(s["e"], 5.0)
        system.adam_step(p, s["grad"], s["m"], s["v"], ITERATION, 3e-3)
        return clipped, stats, p, s["m"], s["v"]
    if c["op"] == "log_psi":
        lp, sign = system.log_psi(p, s["walkers"])
        return lp.to(dt), sign
    if c["op"] == "energy":
        e, lp, sign = system.local_energy(p, s["walkers"])
        return e.to(dt), lp.to(dt), sign
    if c["op"] == "grad":
        grad, mean = system.energy_grad(p, s["walkers"], s["e"])
        return grad, mean
    if c["op"] == "pass":
        walkers, _ = system.init_walkers(c["walkers"], s["seed"], 1.0)
        lp, _ = system.log_psi(p, walkers)
        accepted = torch.zeros(1, dtype=torch.int64, device="cuda")
        system.mcmc_steps(p, walkers, lp, c["steps"], 0.02, s["seed"], accept_count=accepted)
        e, lp_e, sign = system.local_energy(p, walkers)
        return walkers, lp, accepted, e, lp_e, sign
    # train: on copies, as a program that keeps its last good state does (and so that a pass can be repeated)
    p, walkers, opt = p.clone(), s["walkers"].clone(), s["opt"].clone()
    b = c["walkers"]
    grad = torch.empty_like(p)
    lp, e = (torch.empty(b, dtype=torch.float64, device="cuda") for _ in range(2))
    mean = torch.empty(1, dtype=torch.float64, device="cuda")
    accepted = torch.zeros(1, dtype=torch.int64, device="cuda")
    system.vmc_iteration(s["cfg"], p, walkers, ITERATION, opt, grad, lp, e, mean, accepted)
    return p, walkers, opt, grad, lp.to(dt), e.to(dt), mean.to(dt), accepted


def work(case):
    c = case
    n_par = sum(math.prod(shape) for _, shape, _ in _layout(c))
    b, size = c["walkers"], 8 if c["mode"] == "fp64" else 4
    up, dn = _spins(c["mol"])
    n, k, h1, h2, m = up + dn, c["dets"], c["h1"], c["h2"], len(_atoms(c["mol"])[1])
    value = dets = 0.0
    for l in range(c["layers"]):
        dh, dg = (4 * m, 4) if l == 0 else (h1, h2)
        value += 2.0 * n * h1 * (dh + 2 * dg) + 2.0 * h1 * 2 * dh          # rows, and the spin means once per walker
        if l < c["layers"] - 1:
            value += 2.0 * n * (n - 1) * h2 * dg
    value += 2.0 * k * (up * up + dn * dn) * h1
    lu = k * 2.0 / 3.0 * (up ** 3 + dn ** 3)
    dets = lu + k * (2.0 * (up ** 3 + dn ** 3) + 3 * n * 2.0 * (up ** 3 + dn ** 3))   # inverse and tangent products
    full = value * (3 * n + 2) + dets
    walk = 3.0 * n * b * size
    flops, data = {
        "update": (12.0 * n_par + 10.0 * b, size * 7.0 * n_par + 16.0 * b),
        "log_psi": ((value + lu) * b, size * n_par + walk + 9.0 * b),
        "energy": (full * b, size * n_par + walk + 17.0 * b),
        "grad": ((3 * value + lu) * b, size * 2.0 * n_par + walk + 8.0 * b),
        "pass": (((c.get("steps", 0) + 1) * (value + lu) + full) * b, size * n_par + walk + 25.0 * b),
        "train": (((c.get("steps", 0) + 4) * (value + lu) + full) * b, size * 8.0 * n_par + 2 * walk + 16.0 * b),
    }[c["op"]]
    return {"bytes": data, "flops": flops}


# --- the same quantities in plain torch ---------------------------------------------------


def _mean(x, dim, lo, hi):
    return x.narrow(dim, lo, hi - lo).mean(dim) if hi > lo else torch.zeros_like(x.select(dim, 0))


def _stream(c, p, r):
    """The one-electron stream's last layer [B, N, h1], value only."""
    dt, (up, _) = r.dtype, _spins(c["mol"])
    n = r.shape[1]
    nuc = torch.tensor(_atoms(c["mol"])[0], dtype=dt, device=r.device)
    d = r[:, :, None] - nuc
    h = torch.cat([d, d.norm(dim=-1, keepdim=True)], -1).flatten(2)
    d2 = r[:, :, None] - r[:, None, :]
    # the pair of an electron with itself is zero; its norm is kept off the derivative
    eye = torch.eye(n, dtype=torch.bool, device=r.device)[None, :, :, None]
    g = torch.cat([d2, torch.where(eye, 0.0, torch.where(eye, 1.0, d2).norm(dim=-1, keepdim=True))], -1)
    for l in range(c["layers"]):
        v, dh = p["V", l], h.shape[2]
        z = h @ v[:, :dh].T + p["b", l]
        z = z + (_mean(h, 1, 0, up) @ v[:, dh:2 * dh].T + _mean(h, 1, up, n) @ v[:, 2 * dh:3 * dh].T)[:, None]
        gm = torch.cat([_mean(g, 2, 0, up), _mean(g, 2, up, n)], -1)
        z = z + gm @ v[:, 3 * dh:].T
        h = torch.tanh(z) + (h if l else 0.0)
        if l < c["layers"] - 1:
            g = torch.tanh(g @ p["W", l].T + p["c", l]) + (g if l else 0.0)
    return h


def _orbitals(c, blob, r):
    """The orbital matrices [B, K, n, n] (orbital, electron) of each spin that has electrons."""
    p, (up, dn), k, mats = _unpack(c, blob), _spins(c["mol"]), c["dets"], []
    h = _stream(c, p, r)
    nuc = torch.tensor(_atoms(c["mol"])[0], dtype=r.dtype, device=r.device)
    for s, lo, n in ((0, 0, up), (1, up, dn)):
        if not n:
            continue
        d = r[:, lo:lo + n, None, :] - nuc
        if c["aniso"]:
            dist = torch.einsum("omxy,bjmy->bjomx", p["sig", s], d).norm(dim=-1)
        else:
            dist = p["sig", s] * d.norm(dim=-1)[:, :, None]
        env = (p["pi", s] * torch.exp(-dist)).sum(-1)
        phi = (h[:, lo:lo + n] @ p["w", s].T + p["g", s]) * env
        mats.append(phi.view(-1, n, k, n).permute(0, 2, 3, 1).contiguous())
    return mats


def _log_psi(c, blob, r):
    """(log|psi|, sign) of the walkers r [B, N, 3]."""
    dets = [torch.linalg.slogdet(a) for a in _orbitals(c, blob, r)]
    total, sign = sum(x[1] for x in dets), math.prod(x[0] for x in dets)
    top = total.max(-1, keepdim=True)[0]
    psi = (sign * torch.exp(total - top)).sum(-1)
    return top[:, 0] + psi.abs().log(), torch.sign(psi)


def _energy(c, blob, r):
    """(E_L, log|psi|, sign) with the Laplacian carried forward: slab 0 the value, one slab for each of the
    3N derivatives, the last the Laplacian; r is FP64."""
    p, (up, dn), k = _unpack(c, blob), _spins(c["mol"]), c["dets"]
    dt, dev = r.dtype, r.device
    b, n = r.shape[:2]
    t = 3 * n + 2
    nuclei, charges = _atoms(c["mol"])
    nuc = torch.tensor(nuclei, dtype=dt, device=dev)
    m, unit = nuc.shape[0], torch.eye(3, dtype=dt, device=dev)
    d = r[:, :, None] - nuc
    dist = d.norm(dim=-1)
    h = torch.zeros(t, b, n, m, 4, dtype=dt, device=dev)
    h[0, ..., :3], h[0, ..., 3], h[-1, ..., 3] = d, dist, 2.0 / dist
    for e in range(n):
        for x in range(3):
            h[1 + 3 * e + x, :, e, :, :3] = unit[x]
            h[1 + 3 * e + x, :, e, :, 3] = d[:, e, :, x] / dist[:, e]
    h = h.flatten(3)
    # a pair's jet: value, the derivatives along the first electron (the second's are minus these), Laplacian
    d2 = r[:, :, None] - r[:, None, :]
    eye = torch.eye(n, dtype=torch.bool, device=dev)
    dist2 = torch.where(eye, 1.0, d2.norm(dim=-1))
    off = (~eye).to(dt)
    g = torch.zeros(5, b, n, n, 4, dtype=dt, device=dev)
    g[0, ..., :3], g[0, ..., 3], g[4, ..., 3] = d2, dist2 * off, 4.0 / dist2 * off
    for x in range(3):
        g[1 + x, ..., :3] = unit[x] * off[:, :, None]
        g[1 + x, ..., 3] = d2[..., x] / dist2 * off
    for l in range(c["layers"]):
        v, dh, dg = p["V", l], h.shape[3], g.shape[4]
        z = h @ v[:, :dh].T
        z += (_mean(h, 2, 0, up) @ v[:, dh:2 * dh].T + _mean(h, 2, up, n) @ v[:, 2 * dh:3 * dh].T)[:, :, None]
        z[0] += p["b", l]
        gm = torch.zeros(t, b, n, 2, dg, dtype=dt, device=dev)
        for s, lo, hi in ((0, 0, up), (1, up, n)):
            if hi == lo:
                continue
            gs = _mean(g, 3, lo, hi)
            gm[0, :, :, s], gm[-1, :, :, s] = gs[0], gs[4]
            gm[1 + 3 * lo:1 + 3 * hi, :, :, s] = -g[1:4, :, :, lo:hi].permute(3, 0, 1, 2, 4).reshape(
                3 * (hi - lo), b, n, dg) / (hi - lo)
            for e in range(n):
                gm[1 + 3 * e:4 + 3 * e, :, e, s] += gs[1:4, :, e]
        z += gm.flatten(3) @ v[:, 3 * dh:].T
        z = _tanh_jet(z, 1.0)
        h = z + h if l else z
        if l < c["layers"] - 1:
            y = g @ p["W", l].T
            y[0] += p["c", l]
            y = _tanh_jet(y, 2.0)
            g = y + g if l else y
    logs, signs, grads, laps = 0.0, 1.0, 0.0, 0.0
    for s, lo, n_s in ((0, 0, up), (1, up, dn)):
        if not n_s:
            continue
        proj = h[:, :, lo:lo + n_s] @ p["w", s].T
        proj[0] += p["g", s]
        ds = d[:, lo:lo + n_s, None]                                        # [b, j, 1, m, 3]
        sig = p["sig", s] if c["aniso"] else p["sig", s][..., None, None] * unit
        u = torch.einsum("omxy,bjomy->bjomx", sig, ds.expand(b, n_s, sig.shape[0], m, 3))
        q = u.norm(dim=-1)
        su = torch.einsum("omxy,bjomx->bjomy", sig, u)
        dq = su / q[..., None]
        lq = ((sig * sig).sum((-1, -2)) - (dq * dq).sum(-1)) / q
        w = p["pi", s] * torch.exp(-q)
        env, denv = w.sum(-1), -(w[..., None] * dq).sum(-2)
        lenv = (w * ((dq * dq).sum(-1) - lq)).sum(-1)
        phi = proj * env
        for j in range(n_s):
            e = lo + j
            for x in range(3):
                phi[1 + 3 * e + x, :, j] += proj[0, :, j] * denv[:, j, :, x]
                phi[-1, :, j] += 2.0 * proj[1 + 3 * e + x, :, j] * denv[:, j, :, x]
            phi[-1, :, j] += proj[0, :, j] * lenv[:, j]
        a = phi.view(t, b, n_s, k, n_s).permute(0, 1, 3, 4, 2)
        sg, ld = torch.linalg.slogdet(a[0].contiguous())
        inv = torch.linalg.inv(a[0].contiguous())
        da = inv @ a[1:-1]
        tr = da.diagonal(dim1=-2, dim2=-1).sum(-1)                          # [3N, b, k]
        lap = (inv.transpose(-1, -2) * a[-1]).sum((-1, -2)) - (da * da.transpose(-1, -2)).sum((-1, -2)).sum(0)
        logs, signs, grads, laps = logs + ld, signs * sg, grads + tr, laps + lap
    top = logs.max(-1, keepdim=True)[0]
    terms = signs * torch.exp(logs - top)
    psi = terms.sum(-1)
    rho = terms / psi[:, None]
    grad = (rho * grads).sum(-1)                                            # [3N, b]
    lap = (rho * (laps + (grads * grads).sum(0))).sum(-1) - (grad * grad).sum(0)
    e = -0.5 * (lap + (grad * grad).sum(0))
    zs = torch.tensor(charges, dtype=dt, device=dev)
    e = e - (zs / dist).sum((1, 2)) + (off / dist2).sum((1, 2)) / 2
    for i in range(m):
        for j in range(i):
            e = e + float(charges[i] * charges[j]) / (nuc[i] - nuc[j]).norm()
    return e, top[:, 0] + psi.abs().log(), torch.sign(psi)


def _tanh_jet(z, twice):
    """tanh of a jet; `twice`: how often each squared derivative enters the Laplacian."""
    t = torch.tanh(z[0])
    d = 1.0 - t * t
    out = d * z
    out[-1] -= 2.0 * twice * t * d * (z[1:-1] * z[1:-1]).sum(0)
    out[0] = t
    return out


def _chunks(c, f, r, size):
    got = [f(x) for x in r.split(size)]
    return tuple(torch.cat(x) for x in zip(*got))


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 (Salmon et al. 2011): four 32-bit words, as int64 tensors."""
    mask = 0xFFFFFFFF
    x = [torch.as_tensor(v, dtype=torch.int64, device="cuda") & mask for v in (c0, c1, c2, c3)]
    x = list(torch.broadcast_tensors(*x))
    k0, k1 = seed & mask, (seed >> 32) & mask

    def mul(a, w):       # (high, low) words of a 32 x 32 bit product, by the 16-bit halves of a
        lo, hi = (a & 0xFFFF) * w, (a >> 16) * w
        return (hi + (lo >> 16)) >> 16, ((hi << 16) + lo) & mask

    for _ in range(10):
        h0, l0 = mul(x[0], 0xD2511F53)
        h1, l1 = mul(x[2], 0xCD9E8D57)
        x = [h1 ^ x[1] ^ k0, l1, h0 ^ x[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return x


def _uniform(hi, lo):
    return (hi << 21 | lo >> 11).double() * 2.0 ** -53


def _normals(b, coords, step, stream, seed):
    w = torch.arange(b, device="cuda")[:, None]
    j = torch.arange(coords, device="cuda")[None]
    x = _philox(j >> 1, w, step, stream, seed)
    rad = torch.sqrt(-2.0 * torch.log(_uniform(x[0], x[1]) + 2.0 ** -53))
    ang = 2.0 * math.pi * _uniform(x[2], x[3])
    return torch.where(j & 1 == 0, rad * torch.cos(ang), rad * torch.sin(ang))


def exact(case, seed):
    c = case
    if c["op"] == "train":      # its accept decisions are the precision's own: no value in 64 bits belongs to them
        return None
    params = _params(c, seed)
    blob = params.double()
    n = sum(_counts(c["mol"]))
    size = max(1, int(2.0e9 / (8 * (3 * n + 2) * n * max(c["h1"], c["dets"] * n))))
    if c["op"] == "update":
        e = _energies(c, seed)
        centre = e.sort()[0][(e.numel() - 1) // 2]
        spread = (e - centre).abs().mean()
        m, v = (x.double() for x in _moments(c, seed, blob.numel()))
        g = (1e-2 * torch.randn(blob.numel(), generator=_generator(seed, 5), device="cuda")).double()
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        p = blob - 3e-3 * (m / (1 - 0.9 ** ITERATION)) / (torch.sqrt(v / (1 - 0.999 ** ITERATION)) + 1e-8)
        return e.clamp(centre - 5 * spread, centre + 5 * spread), torch.stack([centre, spread]), p, m, v
    if c["op"] == "pass":
        nuclei = torch.tensor(_atoms(c["mol"])[0], dtype=torch.float64, device="cuda")
        b = c["walkers"]
        r = nuclei[_electron_atoms(c["mol"])] + _normals(b, 3 * n, 0, 0, seed).view(b, n, 3)
        lp, taken = _log_psi(c, blob, r)[0], 0
        for k in range(c["steps"]):
            new = r + 0.02 * _normals(b, 3 * n, k, 1, seed).view(b, n, 3)
            lp_new = _log_psi(c, blob, new)[0]
            x = _philox(0, torch.arange(b, device="cuda"), k, 2, seed)
            take = torch.log(_uniform(x[0], x[1]) + 2.0 ** -53) <= 2 * (lp_new - lp)
            r, lp = torch.where(take[:, None, None], new, r), torch.where(take, lp_new, lp)
            taken = taken + take.sum()
        e, lp_e, sign = _energy(c, blob, r)
        return r, lp, taken.view(1), e, lp_e, sign.to(torch.int8)
    r = _walkers(c, seed, params).double()
    if c["op"] == "log_psi":
        with torch.no_grad():
            lp, sign = _chunks(c, lambda x: _log_psi(c, blob, x), r, 4096)
        return lp, sign.to(torch.int8)
    if c["op"] == "energy":
        with torch.no_grad():
            e, lp, sign = _chunks(c, lambda x: _energy(c, blob, x), r, size)
        return e, lp, sign.to(torch.int8)
    e = _energies(c, seed)
    weights = 2.0 * (e - e.mean()) / e.numel()
    blob.requires_grad_()
    for x, w in zip(r.split(2048), weights.split(2048)):
        (w * _log_psi(c, blob, x)[0]).sum().backward()
    return blob.grad, e.mean().view(1)

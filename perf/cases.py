"""What the speed of this library is measured on.

Every case is work a user has the library do through its Python entry points
(fdtd.Sim, fdtd.adjoint_gradient, fdtd.learned_record, fdtd.mlp_train): one
pass writes a starting state, advances it and reads the result, or runs one
gradient, one recording or one training call.  Kinds of case:

  box      a domain stepped from given fields: PEC or graded-absorber walls,
           either schedule, any field storage;
  learned  a domain with the learned boundary (naive schedule);
  adjoint  dL/deps of a design box for the mode-overlap objective;
  record   training pairs of the learned boundary from a reference run;
  train    Adam on such pairs.

exact() states the same results in 64 bits with plain torch and numpy.
"""
import math

import numpy as np
import torch

from paper_2502_20610_gb300 import fdtd

DT = 0.99 / math.sqrt(3.0)  # Courant number 0.99, dx = c = 1
EPS_SIO2, EPS_SI = 2.1, 12.1
N_IN, N_HID, N_OUT = 324, 64, 6  # the learned boundary's network


def listed():
    return [
        # a unit-test sized cavity: one CTA holds the domain (the left end of the size sweep)
        box("tiny_naive_8", 8, 8, 8, steps=100, scheme="naive", start="pulse"),
        # the smallest benchmark workload: a Gaussian pulse in a 64^3 cavity for 200 steps
        box("cavity_64", 64, 64, 64, steps=200, start="pulse"),
        # the 16-bit storage workload
        box("f16_128", 128, 128, 128, steps=300, storage="f16", start="pulse", source=True, eps="slabs"),
        # the same option on a ragged domain (no extent a multiple of a tile's)
        box("bf16_ragged", 203, 149, 101, steps=300, storage="bf16", start="noise", source=True, eps="slabs"),
        # the headline workload: Si slabs in SiO2, a point dipole, one call of many steps
        box("slabs_256", 256, 256, 256, steps=1000, start="zero", source=True, eps="slabs"),
        # a large domain, far beyond L2
        box("slabs_512", 512, 512, 512, steps=150, start="pulse", source=True, eps="slabs"),
        # an open domain: the 32-cell graded absorber
        box("absorber_224", 224, 224, 224, steps=200, boundary="graded", thickness=32, start="pulse", source=True),
        # the streaming schedule (yardsticks and comparisons are run on it)
        box("naive_160", 160, 160, 160, steps=40, scheme="naive", start="noise", eps="slabs"),
        # an open domain with the 4-cell learned boundary
        dict(name="learned_160", kind="learned", n=160, steps=20, thickness=4, sigma=0.3),
        # inverse design: one gradient of the overlap objective on the 200 x 200 x 100 problem
        dict(name="adjoint_200", kind="adjoint", nx=200, ny=200, nz=100, steps=400, window=60, every=100, bx=64, by=64,
             bz=20),
        # training data of the learned boundary: a 48^3 box in its thick-absorber reference
        dict(name="record_48", kind="record", n=48, pad=32, thickness=4, steps=40, per_step=1000),
        # training of the learned boundary: two passes over shuffled minibatches
        dict(name="train_32k", kind="train", samples=32768, batch=4096, epochs=2),
    ]


def box(name, nx, ny, nz, steps, scheme="systolic", storage="f32", boundary="pec", thickness=0, start="pulse",
        source=False, eps="uniform", scaled=False):
    c = dict(kind="box", nx=nx, ny=ny, nz=nz, steps=steps, scheme=scheme, storage=storage, boundary=boundary,
             thickness=thickness, start=start, source=source, eps=eps, scaled=scaled)
    return dict(c, name=name) if name else c


def log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))))


def draw(rng):
    kind = rng.choice(["box", "box", "box", "box", "box", "tiny", "learned", "adjoint", "record", "train"])
    if kind == "tiny":
        n = [rng.randint(2, 10) for _ in range(3)]
        return box(None, *n, steps=log_int(rng, 1, 400), scheme="naive",
                   storage=rng.choice(["f32", "f32", "f16", "bf16"]), start="noise")
    if kind == "box":
        n = [log_int(rng, 24, 420) for _ in range(3)]
        cells = n[0] * n[1] * n[2]
        scheme = rng.choice(["systolic"] * 4 + ["naive"])
        storage = rng.choice(["f32", "f32", "f16", "bf16"])
        graded = rng.random() < 0.25 and min(n) >= 40
        steps = log_int(rng, 1, int(max(8, min(1000, (6e9 if scheme == "systolic" else 1.5e9) / cells))))
        return box(None, *n, steps=steps, scheme=scheme, storage=storage, boundary="graded" if graded else "pec",
                   thickness=rng.randint(8, min(32, min(n) // 3)) if graded else 0, start=rng.choice(["pulse", "noise"]),
                   source=rng.random() < 0.6, eps=rng.choice(["uniform", "slabs"]),
                   scaled=storage == "f16" and rng.random() < 0.3)
    if kind == "learned":
        return dict(kind="learned", n=log_int(rng, 24, 240), steps=rng.randint(2, 24), thickness=4,
                    sigma=rng.choice([0.0, 0.3]))
    if kind == "adjoint":
        nx, ny, nz = log_int(rng, 32, 220), log_int(rng, 32, 220), log_int(rng, 32, 110)
        steps = log_int(rng, 40, 400)
        return dict(kind="adjoint", nx=nx, ny=ny, nz=nz, steps=steps, window=rng.randint(1, max(1, steps // 4)),
                    every=rng.choice([25, 50, 100, 128]), bx=rng.randint(4, nx // 2), by=rng.randint(4, ny // 2),
                    bz=rng.randint(2, nz // 3))
    if kind == "record":
        return dict(kind="record", n=rng.randint(20, 64), pad=rng.randint(20, 34), thickness=4,
                    steps=rng.randint(4, 40), per_step=log_int(rng, 50, 4000))
    batch = log_int(rng, 64, 8192)
    return dict(kind="train", samples=batch * rng.randint(1, 6) + rng.randint(0, batch - 1), batch=batch,
                epochs=rng.randint(1, 3))


# ---------------------------------------------------------------- inputs

def generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def uniform(g, *shape, scale=1.0, dtype=torch.float32):
    return (torch.rand(shape, generator=g, device="cuda", dtype=dtype) * 2 - 1) * scale


def permittivity(c, seed):
    """Host doubles: uniform SiO2, or 8 to 20 Si slabs of 10 x 10 cells in it."""
    shape = (c["nz"], c["ny"], c["nx"])
    eps = np.full(shape, EPS_SIO2)
    if c.get("eps") == "slabs":
        r = np.random.default_rng(seed)
        for _ in range(int(r.integers(8, 21))):
            along = int(r.integers(0, 3))
            at = []
            for a in range(3):
                w = min(shape[a], int(r.integers(shape[a] // 2, shape[a] - 1)) if a == along else 10)
                lo = int(r.integers(0, shape[a] - w + 1))
                at.append(slice(lo, lo + w))
            eps[tuple(at)] = EPS_SI
    return eps


def fields(c, seed):
    """The starting state, float32 (6, nz, ny, nx) on the GPU: nothing, a Gaussian Ez, or noise in every component."""
    nz, ny, nx = c["nz"], c["ny"], c["nx"]
    f = torch.zeros((6, nz, ny, nx), device="cuda")
    g = generator(seed)
    if c["start"] == "noise":
        f = uniform(g, 6, nz, ny, nx)
        f[0][:, 0, :] = 0  # tangential E on the low walls
        f[0][0] = 0
        f[1][:, :, 0] = 0
        f[1][0] = 0
        f[2][:, :, 0] = 0
        f[2][:, 0, :] = 0
    elif c["start"] == "pulse":
        at = [n * (0.5 + 0.1 * float(u)) for n, u in zip((nz, ny, nx), uniform(g, 3).tolist())]
        z, y, x = (torch.arange(n, device="cuda", dtype=torch.float64) for n in (nz, ny, nx))
        width = max(1.0, min(nz, ny, nx) / 16.0)
        e = [torch.exp(-((p - m) ** 2) / (2 * width * width)) for p, m in zip((z, y, x), at)]
        f[2] = (e[0][:, None, None] * e[1][None, :, None] * e[2][None, None, :]).float()
        f[2][:, :, 0] = 0
        f[2][:, 0, :] = 0
    return f


def dipole(c, seed):
    """(component, x, y, z, waveform): a sinusoid of 20 cells' wavelength near the middle."""
    r = np.random.default_rng(seed + 77)
    at = [int(n * (0.4 + 0.2 * r.random())) for n in (c["nx"], c["ny"], c["nz"])]
    t = (np.arange(c["steps"]) + 0.5) * DT
    return (int(r.integers(0, 3)), *at, (0.5 + r.random()) * np.sin(2 * math.pi / 20.0 * t))


def graded_sigma(shape, thickness, peak, order):
    """peak * sum over the axes of (depth / thickness)^order, as the library's graded layer."""
    out = np.zeros(shape)
    for a, n in enumerate(shape):
        i = np.arange(n)
        d = np.where(i < thickness, thickness - i, np.where(i >= n - thickness, i - (n - 1 - thickness), 0))
        out += ((np.maximum(d, 0) / thickness) ** order).reshape([-1 if b == a else 1 for b in range(3)])
    return peak * out


def network(seed):
    """A small seeded network: W1 [64][324], b1, W2 [64][64], b2, W3 [6][64], b3."""
    r = np.random.default_rng(seed + 5)
    parts = []
    for rows, cols, gain in ((N_HID, N_IN, 1.0), (N_HID, N_HID, 1.0), (N_OUT, N_HID, 0.1)):
        parts += [r.uniform(-1, 1, rows * cols) * gain / math.sqrt(cols), r.uniform(-1, 1, rows) * 0.02 * gain]
    return np.concatenate(parts).astype(np.float32)


def mode_profile(c, seed):
    g = generator(seed + 9)
    y = torch.linspace(-2, 2, c["ny"], device="cuda")[:, None]
    x = torch.linspace(-2, 2, c["nx"], device="cuda")[None, :]
    return (torch.exp(-x * x - y * y) * (1 + 0.2 * uniform(g, c["ny"], c["nx"]))).contiguous()


def design(c, seed):
    """eps of the adjoint problem (a random design box in SiO2), the box's corners (x, y, z), its output plane."""
    r = np.random.default_rng(seed + 3)
    eps = np.full((c["nz"], c["ny"], c["nx"]), EPS_SIO2)
    size = (c["bx"], c["by"], c["bz"])
    lo = [(c[n] - s) // 2 for n, s in zip(("nx", "ny", "nz"), size)]
    hi = [p + s for p, s in zip(lo, size)]
    eps[lo[2]:hi[2], lo[1]:hi[1], lo[0]:hi[0]] = r.uniform(EPS_SIO2, EPS_SI, (size[2], size[1], size[0]))
    return eps, lo, hi, min(c["nz"] - 1, hi[2] + max(1, c["nz"] // 10))


def design_source(c, seed, lo):
    r = np.random.default_rng(seed + 4)
    t = (np.arange(c["steps"]) + 0.5) * DT
    return (2, c["nx"] // 2, c["ny"] // 2, max(1, lo[2] // 2), (1 + 0.2 * r.random()) * np.sin(2 * math.pi / 20.0 * t))


def reference(c, seed):
    """The recording's reference domain: (box case, conductivity, corners of the box, host seed)."""
    n = c["n"] + 2 * c["pad"]
    b = box(None, n, n, n, steps=c["steps"] + 1, start="noise", source=True)
    p, q = c["pad"], c["pad"] + c["n"]
    sigma = graded_sigma((n, n, n), c["pad"], 0.5, 3)
    sigma[p:q, p:q, p:q] += graded_sigma((c["n"],) * 3, c["thickness"], 0.3, 3)
    return b, sigma, (p,) * 3, (q,) * 3


def samples(c, seed):
    """Normalised stencils and the corrections of a teacher: two of the six components are corrected in a sample."""
    g = generator(seed + 21)
    x = torch.randn((c["samples"], N_IN), generator=g, device="cuda")
    x /= x.square().mean(1, keepdim=True).sqrt()
    w = torch.randn((N_IN, N_OUT), generator=g, device="cuda") * (0.3 / math.sqrt(N_IN))
    y = torch.tanh(x.double() @ w.double()).float()
    keep = torch.rand((c["samples"], N_OUT), generator=g, device="cuda").argsort(1) < 2
    return x.contiguous(), (y * keep).contiguous()


# ------------------------------------------------------------------ passes

def prepare(case, seed):
    c = dict(case)
    if c["kind"] == "box":
        f = fields(c, seed)
        kw = {}
        if c["scaled"]:
            kw["field_scale"] = fdtd.field_scales(f.cpu().numpy(), c["storage"])
        if c["boundary"] == "graded":
            kw.update(boundary="graded", absorber=(c["thickness"], 0.5, 3))
        sim = fdtd.Sim((c["nz"], c["ny"], c["nx"]), permittivity(c, seed), DT, scheme=c["scheme"], storage=c["storage"],
                       max_source_steps=c["steps"], **kw)
        if c["source"]:
            sim.add_source(*dipole(c, seed))
        return dict(case=c, sim=sim, fields=f)
    if c["kind"] == "learned":
        b = box(None, c["n"], c["n"], c["n"], steps=c["steps"], start="noise")
        learned = (c["thickness"], network(seed)) + ((c["sigma"], 3) if c["sigma"] else ())
        sim = fdtd.Sim((c["n"],) * 3, permittivity(b, seed), DT, scheme="naive", boundary="learned", learned=learned,
                       max_source_steps=c["steps"])
        return dict(case=c, sim=sim, fields=fields(b, seed))
    if c["kind"] == "adjoint":
        eps, lo, hi, k0 = design(c, seed)
        sim = fdtd.Sim(eps.shape, eps, DT, max_source_steps=c["steps"])
        sim.add_source(*design_source(c, seed, lo))
        return dict(case=c, sim=sim, fields=torch.zeros((6,) + eps.shape, device="cuda"), lo=lo, hi=hi, k0=k0,
                    mode=mode_profile(c, seed))
    if c["kind"] == "record":
        b, sigma, lo, hi = reference(c, seed)
        sim = fdtd.Sim(sigma.shape, EPS_SIO2, DT, boundary="graded", absorber=sigma, max_source_steps=b["steps"])
        sim.add_source(*dipole(b, seed))
        return dict(case=c, sim=sim, fields=0.1 * fields(b, seed), lo=lo, hi=hi, seed=seed)
    x, y = samples(c, seed)
    return dict(case=c, x=x, y=y, params=torch.from_numpy(network(seed)).cuda(), seed=seed)


def run(state):
    c = state["case"]
    if c["kind"] == "train":
        params = state["params"].clone()
        loss = fdtd.mlp_train(params, state["x"], state["y"], c["epochs"], batch=c["batch"], lr=1e-3, seed=state["seed"])
        return dict(loss=loss, params=params)
    sim = state["sim"]
    sim.write_fields(state["fields"])
    sim.set_current_step(0)
    if c["kind"] == "adjoint":
        loss, grad = fdtd.adjoint_gradient(sim, state["k0"], state["mode"], c["window"], c["steps"], state["lo"],
                                           state["hi"], checkpoint_every=c["every"])
        return dict(loss=loss, grad=grad)
    if c["kind"] == "record":
        x, y = fdtd.learned_record(sim, state["lo"], state["hi"], c["thickness"], c["steps"], c["per_step"],
                                   seed=state["seed"])
        return dict(x=x, y=y)
    sim.step(c["steps"])
    return sim.read_fields()


def work(case):
    """Each input read once, each output written once; a Yee update is 18 subtractions and 6 multiply-adds a cell (and 3
    multiplications where cells conduct)."""
    c = case
    if c["kind"] == "box":
        cells, lossy = c["nx"] * c["ny"] * c["nz"], c["boundary"] == "graded"
        return dict(bytes=cells * (48 + (8 if lossy else 4)), flops=cells * c["steps"] * (33 if lossy else 30))
    if c["kind"] == "learned":
        cells, faces = c["n"] ** 3, c["n"] ** 3 - (c["n"] - 2) ** 3
        net = 2 * (N_IN * N_HID + N_HID * N_HID + N_HID * N_OUT)
        return dict(bytes=cells * (48 + (8 if c["sigma"] else 4)), flops=c["steps"] * (cells * 30 + faces * net))
    if c["kind"] == "adjoint":
        cells, inner = c["nx"] * c["ny"] * c["nz"], c["bx"] * c["by"] * c["bz"]
        return dict(bytes=cells * 28 + c["nx"] * c["ny"] * 4 + inner * 8, flops=2 * c["steps"] * cells * 30)
    if c["kind"] == "record":
        cells = (c["n"] + 2 * c["pad"]) ** 3
        return dict(bytes=cells * 32 + c["steps"] * c["per_step"] * 4 * (N_IN + N_OUT), flops=(c["steps"] + 1) * cells * 33)
    seen = c["epochs"] * (c["samples"] // c["batch"]) * c["batch"]
    net = 2 * (N_IN * N_HID + N_HID * N_HID + N_HID * N_OUT)
    return dict(bytes=c["samples"] * 4 * (N_IN + N_OUT), flops=seen * (3 * net - 2 * N_IN * N_HID))


# ------------------------------------------------------------------ 64 bits

def forward_difference(a, axis):
    d = -a  # the value past the last one reads 0
    n = a.shape[axis]
    d.narrow(axis, 0, n - 1).add_(a.narrow(axis, 1, n - 1))
    return d


def backward_difference(a, axis):
    d = a.clone()
    n = a.shape[axis]
    d.narrow(axis, 1, n - 1).sub_(a.narrow(axis, 0, n - 1))
    return d


def yee_step(f, cb, ca=None):
    """One step of f (6, nz, ny, nx) in place: H, then E, on the box with PEC walls."""
    ex, ey, ez, hx, hy, hz = f
    fwd, bwd, Z, Y, X = forward_difference, backward_difference, 0, 1, 2
    hx.sub_((fwd(ez, Y).sub_(fwd(ey, Z))), alpha=DT)
    hy.sub_((fwd(ex, Z).sub_(fwd(ez, X))), alpha=DT)
    hz.sub_((fwd(ey, X).sub_(fwd(ex, Y))), alpha=DT)
    for e, curl, inner in ((ex, lambda: bwd(hz, Y).sub_(bwd(hy, Z)), np.s_[1:, 1:, :]),
                           (ey, lambda: bwd(hx, Z).sub_(bwd(hz, X)), np.s_[1:, :, 1:]),
                           (ez, lambda: bwd(hy, X).sub_(bwd(hx, Y)), np.s_[:, 1:, 1:])):
        d = curl().mul_(cb)
        if ca is not None:
            e[inner].mul_(ca[inner])
        e[inner].add_(d[inner])


def coefficients(eps, sigma=None):
    eps = torch.from_numpy(np.ascontiguousarray(eps)).cuda()
    if sigma is None:
        return DT / eps, None
    g = torch.from_numpy(sigma).cuda() * DT / (2 * eps)
    return (DT / eps) / (1 + g), (1 - g) / (1 + g)


def add_dipole(f, cb, source, n):
    comp, x, y, z, wave = source
    f[comp, z, y, x] -= cb[z, y, x] * float(wave[n])


def twister(seed):
    """The 64-bit Mersenne Twister's outputs (Nishimura 2000)."""
    mask, low = (1 << 64) - 1, (1 << 31) - 1
    s = [seed & mask]
    for i in range(1, 312):
        s.append((6364136223846793005 * (s[-1] ^ (s[-1] >> 62)) + i) & mask)
    while True:
        for i in range(312):
            x = (s[i] & ~low & mask) | (s[(i + 1) % 312] & low)
            s[i] = s[(i + 156) % 312] ^ (x >> 1) ^ (0xB5026F5AA96619E9 if x & 1 else 0)
        for x in list(s):
            x ^= (x >> 29) & 0x5555555555555555
            x ^= (x << 17) & 0x71D67FFFEDA60000
            x ^= (x << 37) & 0xFFF7EEE000000000
            yield x ^ (x >> 43)


def below(bits, n):
    """A uniform integer below n from 64-bit outputs (Lemire 2019)."""
    p = next(bits) * n
    if p & ((1 << 64) - 1) < n:
        floor = (1 << 64) % n
        while p & ((1 << 64) - 1) < floor:
            p = next(bits) * n
    return p >> 64


def shuffle(order, bits):
    """The GNU C++ library's std::shuffle: two places from each draw."""
    i, n = 1, len(order)
    if n and n % 2 == 0:
        k = below(bits, 2)
        order[i], order[k] = order[k], order[i]
        i += 1
    while i < n:
        k, l = divmod(below(bits, (i + 1) * (i + 2)), i + 2)
        order[i], order[k] = order[k], order[i]
        order[i + 1], order[l] = order[l], order[i + 1]
        i += 2


def layers(theta):
    out, at = [], 0
    for rows, cols in ((N_HID, N_IN), (N_HID, N_HID), (N_OUT, N_HID)):
        out.append((theta[at:at + rows * cols].reshape(rows, cols), theta[at + rows * cols:at + rows * cols + rows]))
        at += rows * cols + rows
    return out


def evaluate(theta, x):
    (w1, b1), (w2, b2), (w3, b3) = layers(theta)
    return torch.tanh(torch.tanh(x @ w1.T + b1) @ w2.T + b2) @ w3.T + b3


def stencils(states, x, y, z):
    """[cells, 324]: the 3 x 3 x 3 neighbours of every component in each state, 0 outside."""
    out = []
    for f in states:
        p = torch.nn.functional.pad(f, (1, 1, 1, 1, 1, 1))
        out += [p[:, z + dz, y + dy, x + dx] for dz in range(3) for dy in range(3) for dx in range(3)]
    s = torch.stack(out).reshape(len(states), 27, 6, -1)
    return s.permute(3, 0, 2, 1).reshape(x.numel(), -1)


def corrected(x, y, z, n):
    """[cells, 6]: tangential E on a low face, tangential H on a high face."""
    m = torch.zeros((x.numel(), 6), dtype=torch.bool, device="cuda")
    for p, (a, b) in ((x, (1, 2)), (y, (0, 2)), (z, (0, 1))):
        for comp in (a, b):
            m[:, comp] |= p == 0
            m[:, 3 + comp] |= p == n - 1
    return m


def exact(case, seed):
    c = dict(case)
    return dict(box=exact_box, learned=exact_learned, adjoint=exact_adjoint, record=exact_record,
                train=exact_train)[c["kind"]](c, seed)


def exact_box(c, seed):
    shape = (c["nz"], c["ny"], c["nx"])
    sigma = graded_sigma(shape, c["thickness"], 0.5, 3) if c["boundary"] == "graded" else None
    cb, ca = coefficients(permittivity(c, seed), sigma)
    f = fields(c, seed).double()
    source = dipole(c, seed) if c["source"] else None
    for n in range(c["steps"]):
        yee_step(f, cb, ca)
        if source:
            add_dipole(f, cb, source, n)
    return f


def exact_learned(c, seed):
    n = c["n"]
    b = box(None, n, n, n, steps=c["steps"], start="noise")
    sigma = graded_sigma((n,) * 3, c["thickness"], c["sigma"], 3) if c["sigma"] else None
    cb, ca = coefficients(permittivity(b, seed), sigma)
    theta = torch.from_numpy(network(seed)).cuda().double()
    f = fields(b, seed).double()
    before = torch.zeros_like(f)
    inner = torch.zeros((n,) * 3, dtype=torch.bool, device="cuda")
    inner[1:-1, 1:-1, 1:-1] = True
    z, y, x = (~inner).nonzero(as_tuple=True)
    mask = corrected(x, y, z, n)
    for _ in range(c["steps"]):
        s = stencils((f, before), x, y, z)
        r = s.square().mean(1, keepdim=True).sqrt()
        add = torch.where(r >= 1e-30, r * evaluate(theta, s / r.clamp_min(1e-300)), torch.zeros_like(r)) * mask
        before = f.clone()
        yee_step(f, cb, ca)
        f[:, z, y, x] += add.T
    return f


def exact_adjoint(c, seed):
    eps, lo, hi, k0 = design(c, seed)
    cb, _ = coefficients(eps)
    source, mode = design_source(c, seed, lo), mode_profile(c, seed).double()
    inner = np.s_[:3, lo[2]:hi[2], lo[1]:hi[1], lo[0]:hi[0]]
    f = torch.zeros((6,) + eps.shape, dtype=torch.float64, device="cuda")
    seen, overlap = [f[inner].clone()], [0.0]
    for n in range(c["steps"]):
        yee_step(f, cb)
        add_dipole(f, cb, source, n)
        seen.append(f[inner].clone())
        overlap.append((mode * f[2, k0]).sum())
    counted = range(c["steps"] - c["window"] + 1, c["steps"] + 1)
    loss = sum(float(overlap[n]) ** 2 for n in counted)
    # the transposed step in (c lambda_E, -dt lambda_H) is the step itself
    adj = torch.zeros_like(f)
    grad = torch.zeros_like(seen[0][0])
    drive = 2 * (cb[k0] * mode)
    drive[0, :] = 0
    drive[:, 0] = 0
    adj[2, k0] += drive * overlap[-1]
    for n in range(c["steps"] - 1, -1, -1):
        grad -= (adj[inner] * (seen[n + 1] - seen[n])).sum(0) / DT
        yee_step(adj, cb)
        if n in counted:
            adj[2, k0] += drive * overlap[n]
    return dict(loss=loss, grad=grad)


def exact_record(c, seed):
    b, sigma, lo, hi = reference(c, seed)
    cb, ca = coefficients(permittivity(b, seed), sigma)
    f, source = 0.1 * fields(b, seed).double(), dipole(b, seed)
    n, p, q = c["n"], lo[0], hi[0]
    at = np.s_[..., p:q, p:q, p:q]
    bits = twister(seed)
    states = [f[at].clone()]
    yee_step(f, cb, ca)
    add_dipole(f, cb, source, 0)
    states.append(f[at].clone())
    xs, ys = [], []
    for s in range(c["steps"]):
        yee_step(f, cb, ca)
        add_dipole(f, cb, source, s + 1)
        cells = []
        while len(cells) < c["per_step"]:
            cell = [next(bits) % n for _ in range(3)]
            if min(min(v, n - 1 - v) for v in cell) < c["thickness"]:
                cells.append(cell)
        x, y, z = torch.tensor(cells, device="cuda").T
        own = states[1].clone()
        yee_step(own, cb[at].contiguous(), ca[at].contiguous())
        v = stencils((states[1], states[0]), x, y, z)
        r = v.square().mean(1, keepdim=True).sqrt()
        live = r >= 1e-30
        xs.append(torch.where(live, v / r, 0.0))
        ys.append(torch.where(live & corrected(x, y, z, n), (f[at][:, z, y, x] - own[:, z, y, x]).T / r, 0.0))
        states = [states[1], f[at].clone()]
    return dict(x=torch.cat(xs), y=torch.cat(ys))


def exact_train(c, seed):
    x, y = (v.double() for v in samples(c, seed))
    theta = torch.from_numpy(network(seed)).cuda().double().requires_grad_()
    m, v = torch.zeros_like(theta), torch.zeros_like(theta)
    bits, order, t, loss = twister(seed), list(range(c["samples"])), 0, 0.0
    batches = c["samples"] // c["batch"]
    for _ in range(c["epochs"]):
        shuffle(order, bits)
        rows, loss = torch.tensor(order, device="cuda"), 0.0
        for k in range(batches):
            at = rows[k * c["batch"]:(k + 1) * c["batch"]]
            here = (evaluate(theta, x[at]) - y[at]).square().mean()
            g, = torch.autograd.grad(here, theta)
            t += 1
            m = 0.9 * m + 0.1 * g
            v = 0.999 * v + 0.001 * g * g
            with torch.no_grad():
                theta -= 1e-3 * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8)
            loss += float(here) / batches
    return dict(loss=loss, params=theta.detach())

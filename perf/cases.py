"""The calls whose speed matters to a user of this library, as runnable cases.

A case is one pass through the public entry points of
``paper_2607_24908_gb300.tl`` (the ctypes binding of include/tl.h), over the
kinds of work a simulation program has the library do:

* ``evolve``: advance one lattice by some steps and read its energies (the
  simulation loop between two measurements), scalar fields in torch buffers
  that the program owns;
* ``ensemble``: advance many small lattices of uneven size together
  (``tl_batch_step``) and read every job's energies;
* ``spectrum``: the binned power spectra measured along a run;
* ``init``: draw a job's initial Gaussian random fields;
* ``langevin``: Langevin steps of a phi^4 field;
* ``su2``: SU(2) Yang-Mills steps, then the energies and Gauss's law and the
  links and electric fields copied out to page-locked host memory.

``exact`` restates each pass in plain torch, FP64.
"""
import math
import random

import torch

from paper_2607_24908_gb300 import tl as T

TORCH_DTYPE = {"f32": torch.float32, "f64": torch.float64}
# a drawn case's cost in FP32 site-updates is at most this (the largest listed
# case: 1024^3 sites, two fields, seven passes)
MAX_SITE_UPDATES = 7 * 2 * 1024 ** 3


def _evolve(name, N, nf, dtype, expanding, kIR, q, dt, steps, integrator):
    return {"name": name, "kind": "evolve", "N": N, "nf": nf, "dtype": dtype, "expanding": expanding, "kIR": kIR,
            "q": q, "dt": dt, "steps": steps, "integrator": integrator}


def listed():
    return [
        # phi^4 in a static box, the smallest production lattice: 100 steps between two measurements
        _evolve("static-32-f64-leapfrog", 32, 1, "f64", False, 0.5, 0.0, 0.05, 100, "leapfrog"),
        # the smallest call: one step of a small coupled lattice driven step by step from a host loop
        _evolve("onestep-48-f32-2f", 48, 2, "f32", True, 0.5, 10.0, 0.01, 1, "verlet"),
        # parametric resonance of phi^4 in an expanding box, the FP64 production run
        _evolve("expanding-256-f64", 256, 1, "f64", True, 0.1, 0.0, 0.01, 25, "verlet"),
        # the same run with FP32 fields: the 100 steps between two spectra
        _evolve("expanding-256-f32", 256, 1, "f32", True, 0.1, 0.0, 0.01, 100, "verlet"),
        # a served job near the largest size, three coupled fields, a size that no tile divides
        _evolve("served-380-f32-3f", 380, 3, "f32", True, 0.1, 100.0, 0.01, 20, "verlet"),
        # the headline workload: 1024^3, two fields, fourth-order Yoshida
        _evolve("twofield-1024-f32-yoshida", 1024, 2, "f32", True, 0.05, 100.0, 0.005, 2, "yoshida4"),
        # an ensemble of 96 uneven jobs advanced together
        {"name": "ensemble-96-f32", "kind": "ensemble", "jobs": 96, "dtype": "f32", "min_N": 32, "max_N": 128,
         "mix": 1, "dt": 0.01, "steps": 50},
        # the spectra of both fields of a coupled run, every 100 steps
        {"name": "spectrum-256-f32-2f", "kind": "spectrum", "N": 256, "nf": 2, "dtype": "f32", "kIR": 0.1},
        # the initial state of a two-field job
        {"name": "init-256-f32-2f", "kind": "init", "N": 256, "nf": 2, "dtype": "f32", "kIR": 0.1,
         "fluct_pi": False},
        # Langevin phi^4 at a production size
        {"name": "langevin-384-f32", "kind": "langevin", "N": 384, "dtype": "f32", "steps": 10},
        # SU(2) Yang-Mills with FP32 links: a measurement every 50 steps
        {"name": "su2-128-f32", "kind": "su2", "N": 128, "dtype": "f32", "steps": 50},
        # and in FP64, at a size that no tile divides
        {"name": "su2-100-f64", "kind": "su2", "N": 100, "dtype": "f64", "steps": 20},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _log_N(rng, lo, hi, multiple):
    return max(lo, min(hi, _log_int(rng, lo, hi) // multiple * multiple))


def draw(rng):
    kind = rng.choice(["evolve"] * 5 + ["ensemble", "spectrum", "init", "langevin", "su2"])
    dtype = rng.choice(["f32", "f64"])
    cost = 8.0 if dtype == "f64" else 1.0  # FP64 arithmetic is this much dearer a site
    if kind == "evolve":
        N, nf = _log_N(rng, 16, 640, 4), rng.choice([1, 1, 2, 2, 3])
        integrator = rng.choice(["leapfrog", "verlet", "yoshida4"])
        per_step = N ** 3 * nf * cost * (3 if integrator == "yoshida4" else 1)
        steps = _log_int(rng, 1, max(1, min(100, MAX_SITE_UPDATES / per_step - 1)))
        return {"kind": kind, "N": N, "nf": nf, "dtype": dtype, "expanding": rng.random() < 0.75,
                "kIR": rng.choice([0.5, 0.1]) if N < 192 else rng.choice([0.1, 0.05]),
                "q": rng.choice([0.0, 1.0, 10.0, 100.0]) if nf > 1 else 0.0,
                "dt": 0.005 if integrator == "yoshida4" else 0.01, "steps": steps, "integrator": integrator}
    if kind == "ensemble":
        return {"kind": kind, "jobs": _log_int(rng, 8, 96), "dtype": dtype, "min_N": rng.choice([16, 32]),
                "max_N": rng.choice([96, 128, 144]), "mix": rng.randrange(1, 1 << 20), "dt": 0.01,
                "steps": _log_int(rng, 5, 20 if dtype == "f64" else 50)}
    if kind == "spectrum":
        return {"kind": kind, "N": _log_N(rng, 32, 384, 4), "nf": rng.choice([1, 2]), "dtype": dtype,
                "kIR": rng.choice([0.5, 0.1])}
    if kind == "init":
        return {"kind": kind, "N": _log_N(rng, 32, 320, 4), "nf": rng.choice([1, 2]), "dtype": dtype,
                "kIR": rng.choice([0.5, 0.1]), "fluct_pi": rng.random() < 0.5}
    if kind == "langevin":
        return {"kind": kind, "N": _log_N(rng, 32, 384 if dtype == "f32" else 256, 4), "dtype": dtype,
                "steps": _log_int(rng, 2, 20)}
    return {"kind": kind, "N": _log_N(rng, 12, 160 if dtype == "f32" else 112, 1), "dtype": dtype,
            "steps": _log_int(rng, 5, 50 if dtype == "f32" else 20)}


# --- inputs ------------------------------------------------------------------


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _white_noise(N, nf, dtype, gen):
    """phi_0 = 1 and phi_f = 0 plus white noise, momenta white noise (the start
    of the phi^4 benchmarks): yields (field, which, dense array)."""
    for f in range(nf):
        for which in range(2):
            x = torch.randn((N, N, N), generator=gen, device="cuda", dtype=TORCH_DTYPE[dtype]).mul_(1e-2)
            yield f, which, x.add_(1.0) if (f, which) == (0, 0) else x


def _ensemble_members(case):
    """(N, fields, q) of every job: the composition is the case's own."""
    rng = random.Random(case["mix"])
    sizes = [n for n in (16, 32, 48, 64, 96, 128, 144) if case["min_N"] <= n <= case["max_N"]]
    return [(rng.choice(sizes), rng.choice([1, 2]), rng.choice([0.0, 10.0, 100.0])) for _ in range(case["jobs"])]


def _su2_start(N, gen):
    q = torch.randn((3, 4, N, N, N), generator=gen, device="cuda", dtype=torch.float64).mul_(0.6)
    q[:, 0] = 1.0
    q /= q.square().sum(1, keepdim=True).sqrt()
    return q, torch.randn((3, 3, N, N, N), generator=gen, device="cuda", dtype=torch.float64).mul_(0.2)


# --- what a program keeps between calls ---------------------------------------


class Sim:
    """A lattice over torch memory: the handle, the buffers and a view of every
    array's interior sites by device address."""

    def __init__(self, N, nf, dtype, kIR, expanding, q, storage=None):
        elems, pitch, _, origin = T.tl_array_layout(N, T.DTYPES[dtype])
        self.N, self.nf = N, nf
        self.storage = storage if storage is not None else torch.zeros((4 * nf, elems), dtype=TORCH_DTYPE[dtype],
                                                                       device="cuda")
        ex = T.tl_expansion(int(expanding), 1.0, 1.0, 1.0)
        self.h = T.tl_lattice_create_with_buffers(N, kIR, nf, T.DTYPES[dtype], ex, 0,
                                                  [a.data_ptr() for a in self.storage])
        T.tl_set_potential(self.h, 1.0, q, (0.0, 0.0, 0.0))
        esz, lpad = self.storage.element_size(), origin - pitch
        self.views = {a.data_ptr() + origin * esz: a.view(N, N + 2, pitch)[:, 1:N + 1, lpad:lpad + N]
                      for a in self.storage}

    def array(self, f, which):
        return self.views[T.tl_state_device_ptr(self.h, f, which)]

    def state(self):
        return [self.array(f, which) for f in range(self.nf) for which in range(2)]

    def start(self, gen, dtype, expanding):
        for f, which, x in _white_noise(self.N, self.nf, dtype, gen):
            self.array(f, which).copy_(x)
        T.tl_commit_state(self.h)
        if expanding:
            T.tl_set_background(self.h, 1.0, 0.0, True)

    def energies(self):
        e = T.tl_energies(self.h)
        return list(e.K[:self.nf]) + list(e.G[:self.nf]) + [e.V, e.a, e.b]

    def __del__(self):
        if getattr(self, "h", None):
            T.tl_lattice_destroy(self.h)
            self.h = None


class Ensemble:
    """Jobs of one batch; the arrays of all jobs of a size share one torch
    tensor [array][parity][field of a job], so a size's state is one view."""

    def __init__(self, case, seed):
        members, dtype = _ensemble_members(case), case["dtype"]
        self.sizes = {}
        for N in sorted({m[0] for m in members}):
            elems, pitch, _, origin = T.tl_array_layout(N, T.DTYPES[dtype])
            slots = sum(nf for n, nf, _ in members if n == N)
            self.sizes[N] = (torch.zeros((2, 2, slots, elems), dtype=TORCH_DTYPE[dtype], device="cuda"), pitch,
                             origin - pitch)
        used = dict.fromkeys(self.sizes, 0)
        self.sims = []
        gen = _generator(seed)
        for N, nf, q in members:
            block, at = self.sizes[N][0], used[N]
            used[N] += nf
            arrays = [block[which, parity, at + f] for f in range(nf) for parity in range(2) for which in range(2)]
            sim = Sim(N, nf, dtype, 0.5, True, q, storage=arrays_of(arrays))
            sim.start(gen, dtype, True)
            self.sims.append(sim)
        self.first = {N: next(s for s in self.sims if s.N == N) for N in self.sizes}
        self.batch = T.tl_batch_create([s.h for s in self.sims], 0)

    def state(self):
        out = []
        for N, (block, pitch, lpad) in self.sizes.items():
            sim = self.first[N]
            parity = int(sim.array(0, 0).data_ptr() != sim.storage[0].data_ptr() + (pitch + lpad) * block.element_size())
            for which in range(2):
                out.append(block[which, parity].view(-1, N, N + 2, pitch)[:, :, 1:N + 1, lpad:lpad + N])
        return out

    def __del__(self):
        if getattr(self, "batch", None):
            T.tl_batch_destroy(self.batch)
            self.batch = None


class arrays_of(list):
    """A lattice's arrays as a list with the one tensor method Sim asks for."""

    def element_size(self):
        return self[0].element_size()


class Links:
    """An SU(2) lattice and the page-locked host arrays its state is read into."""

    def __init__(self, case, seed):
        N, dt = case["N"], TORCH_DTYPE[case["dtype"]]
        self.lat = T.SU2(N, case["dtype"])
        U, E = _su2_start(N, _generator(seed))
        self.U = torch.empty((3, 4, N, N, N), dtype=dt, pin_memory=True)
        self.E = torch.empty((3, 3, N, N, N), dtype=dt, pin_memory=True)
        self.U.copy_(U)
        self.E.copy_(E)
        self.lat.set_state(self.U.numpy(), self.E.numpy())


def prepare(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        return case, Ensemble(case, seed), T.INTEGRATORS["verlet"]
    if kind == "su2":
        return case, Links(case, seed), None
    N, dtype = case["N"], case["dtype"]
    if kind == "evolve":
        sim = Sim(N, case["nf"], dtype, case["kIR"], case["expanding"], case["q"])
        sim.start(_generator(seed), dtype, case["expanding"])
        return case, sim, T.INTEGRATORS[case["integrator"]]
    if kind == "langevin":  # unit lattice spacing
        sim = Sim(N, 1, dtype, 2.0 * math.pi / N, False, 0.0)
        sim.start(_generator(seed), dtype, False)
        return case, sim, seed
    sim = Sim(N, case["nf"], dtype, case["kIR"], True, 100.0)
    if kind == "spectrum":
        sim.start(_generator(seed), dtype, True)
    return case, sim, seed


def run(state):
    case, sim, more = state
    kind = case["kind"]
    if kind == "evolve":
        T.tl_step(sim.h, case["steps"], case["dt"], more)
        return {"energies": sim.energies(), "state": sim.state()}
    if kind == "ensemble":
        T.tl_batch_step(sim.batch, case["steps"], case["dt"], more)
        return {"energies": torch.tensor([x for s in sim.sims for x in s.energies()]), "state": sim.state()}
    if kind == "spectrum":
        return [T.tl_spectrum(sim.h, sim.N, f, 0) for f in range(sim.nf)]
    if kind == "init":
        T.tl_init_fluctuations(sim.h, more, 1e-10, (3.0, 100.0, 0.0), (1.0, 0.0, 0.0),
                               fluct_pi=case["fluct_pi"])
        return {"energies": sim.energies(), "state": sim.state()}
    if kind == "langevin":
        T.tl_langevin_step(sim.h, case["steps"], 0.01, 1.0, 0.5, 1.0, more)
        return sim.array(0, 0)
    sim.lat.step(case["steps"], 0.05)
    measured = sim.lat.measure().tolist()
    if T.lib().tl_su2_get_state(sim.lat.h, sim.U.data_ptr(), sim.E.data_ptr()) != T.OK:
        raise RuntimeError("tl_su2_get_state failed")
    return {"measured": measured, "U": sim.U, "E": sim.E}


def work(case):
    """The state read once and written once per pass of the integrator (the
    scale factor of a pass needs the energies of the one before, so no two can
    share a sweep), and the arithmetic operations of the method a site."""
    kind = case["kind"]
    esz = 8 if case["dtype"] == "f64" else 4
    if kind == "ensemble":
        sites = sum(N ** 3 * nf for N, nf, _ in _ensemble_members(case)) * (case["steps"] + 1)
        return {"bytes": sites * 4 * esz, "flops": sites * 34}
    n3 = case["N"] ** 3
    if kind == "evolve":
        passes = case["steps"] * (3 if case["integrator"] == "yoshida4" else 1) + 1
        sites = n3 * case["nf"] * passes
        return {"bytes": sites * 4 * esz, "flops": sites * 34}
    if kind == "spectrum":
        return {"bytes": n3 * case["nf"] * esz, "flops": n3 * case["nf"] * (2.5 * math.log2(n3) + 5)}
    if kind == "init":
        drawn = case["nf"] * (2 if case["fluct_pi"] else 1)
        return {"bytes": 2 * n3 * case["nf"] * esz, "flops": n3 * drawn * (2.5 * math.log2(n3) + 50)}
    if kind == "langevin":
        return {"bytes": 2 * n3 * esz * case["steps"], "flops": n3 * 70 * case["steps"]}
    return {"bytes": 42 * n3 * esz * case["steps"] + 21 * n3 * esz, "flops": n3 * 650 * case["steps"]}


# --- the same passes in 64 bits -------------------------------------------------


def _laplacian(x, inv_dx2):
    out = x * -6.0
    for d in range(3):
        out += torch.roll(x, 1, d)
        out += torch.roll(x, -1, d)
    return out.mul_(inv_dx2)


class Exact:
    """Scalar fields in an expanding (alpha = 1) or static box: V = phi_0^4/4 +
    (q/2) phi_0^2 sum phi_f^2, palindromic substeps (kick/2, drift, kick/2)."""

    def __init__(self, N, kIR, q, expanding, phi, pi):
        self.dx = 2.0 * math.pi / (kIR * N)
        self.q, self.expanding = q, expanding
        self.phi, self.pi = phi, pi
        self.a, self.b = 1.0, 0.0
        if expanding:
            self.b = math.sqrt(sum(self.energies()) / 3.0)

    def energies(self):
        nf = len(self.phi)
        K = [0.5 * self.a ** -6 * float(p.square().mean()) for p in self.pi]
        G = []
        for x in self.phi:
            g = 0.0
            for d in range(3):
                g += float((torch.roll(x, -1, d) - x).square_().mean())
            G.append(0.5 * self.a ** -2 * g / self.dx ** 2)
        s0 = self.phi[0].square()
        V = 0.25 * float(s0.square().mean())
        for f in range(1, nf):
            V += 0.5 * self.q * float((s0 * self.phi[f].square()).mean())
        return K + G + [V]

    def half_kick(self, f, dt):
        x = self.phi[f]
        if f == 0:
            force = x.square()
            for y in self.phi[1:]:
                force += self.q * y.square()
        else:
            force = self.q * self.phi[0].square()
        lap = _laplacian(x, self.a ** 2 / self.dx ** 2)
        self.pi[f] += 0.5 * dt * (lap - self.a ** 4 * force.mul_(x))

    def second_derivative(self):
        if not self.expanding:
            return 0.0
        E, nf = self.energies(), len(self.phi)
        return self.a ** 3 / 3.0 * (-sum(E[:nf]) + sum(E[nf:2 * nf]) + 2.0 * E[2 * nf])

    def substep(self, dt):
        self.b += 0.5 * dt * self.acc
        for f in range(len(self.phi)):
            self.half_kick(f, dt)
        a0 = self.a
        if self.expanding:
            self.a += dt * self.b
        drift = dt * (0.5 * (a0 + self.a)) ** -2 if self.expanding else dt
        for x, p in zip(self.phi, self.pi):
            x += drift * p
        for f in range(len(self.phi)):
            self.half_kick(f, dt)
        self.acc = self.second_derivative()
        self.b += 0.5 * dt * self.acc

    def steps(self, n, dt, integrator):
        self.acc = self.second_derivative()
        w1 = 1.0 / (2.0 - 2.0 ** (1.0 / 3.0))
        weights = (w1, 1.0 - 2.0 * w1, w1) if integrator == "yoshida4" else (1.0,)
        for _ in range(n):
            for w in weights:
                self.substep(w * dt)
        return self

    def outputs(self):
        """[K.., G.., V, a, b] and [phi_0, pi_0, phi_1, ...] (a static box reports a = 1, a' = 0)."""
        return self.energies() + [self.a, self.b], [x for f in zip(self.phi, self.pi) for x in f]


def _exact_fields(N, nf, dtype, gen):
    phi, pi = [], []
    for _, which, x in _white_noise(N, nf, dtype, gen):
        (pi if which else phi).append(x.double())
    return phi, pi


def _low_product(a, b):
    """The 128-bit product of two 64-bit words held in int64, as (high, low)."""
    mask = 0xFFFFFFFF
    a0, a1, b0, b1 = a & mask, (a >> 32) & mask, b & mask, (b >> 32) & mask
    p00, p01, p10, p11 = a0 * b0, a0 * b1, a1 * b0, a1 * b1
    mid = ((p00 >> 32) & mask) + (p01 & mask) + (p10 & mask)
    high = p11 + ((p01 >> 32) & mask) + ((p10 >> 32) & mask) + (mid >> 32)
    return high, (mid << 32) | (p00 & mask)


def _signed(x):
    x &= (1 << 64) - 1
    return x - (1 << 64) if x >> 63 else x


def _philox_uniforms(counter, word, key):
    """u1 in (0, 1], u2 in [0, 1): the two outputs of Philox-2x64-10 of counter
    (counter, word) under key, 53 bits each."""
    c0, c1 = counter, torch.full_like(counter, _signed(word))
    mult = torch.full_like(counter[:1], _signed(0xD2B74407B1CE6E93))
    for r in range(10):
        high, low = _low_product(mult, c0)
        c0, c1 = high ^ _signed(key + r * 0x9E3779B97F4A7C15) ^ c1, low
    top = (1 << 53) - 1
    return (((c0 >> 11) & top) + 1).double() * 2.0 ** -53, ((c1 >> 11) & top).double() * 2.0 ** -53


def _drawn_field(N, kIR, seed, stream, meff2, momentum):
    """One Gaussian random field of power A/(2 omega) (A omega/2 for momenta), A = 1e-10."""
    i = torch.arange(N, device="cuda")
    n = torch.where(i < N // 2, i, i - N)
    nx, ny, nz = torch.arange(N // 2 + 1, device="cuda"), n.view(N, 1), n.view(N, 1, 1)
    r2 = nx * nx + ny * ny + nz * nz
    canon = (nx > 0) | ((nx == 0) & ((ny > 0) | ((ny == 0) & (nz > 0))))
    ix, iy, iz = nx, i.view(N, 1), i.view(N, 1, 1)
    own = (iz * N + iy) * N + ix
    pair = ((N - iz) % N * N + (N - iy) % N) * N + (N - ix) % N
    u1, u2 = _philox_uniforms(torch.where(canon, own, pair).reshape(-1), stream, seed)
    omega = (kIR ** 2 * r2.double() + meff2).sqrt().reshape(-1)
    power = 1e-10 * omega / 2.0 if momentum else 1e-10 / (2.0 * omega)
    amp = (power * (kIR / (2.0 * math.pi)) ** 3 * -u1.log()).sqrt()
    phase = 2.0 * math.pi * u2
    modes = torch.complex(amp * phase.cos(), torch.where(canon.reshape(-1), amp, -amp) * phase.sin())
    modes = torch.where(((r2 > 0) & (4 * r2 < N * N)).reshape(-1), modes, torch.zeros_like(modes))
    return torch.fft.irfftn(modes.view(N, N, N // 2 + 1), s=(N, N, N), norm="forward")


def _exact_init(case, seed):
    N, nf, kIR = case["N"], case["nf"], case["kIR"]
    phi, pi = [], []
    for f in range(nf):
        phi.append(_drawn_field(N, kIR, seed, f, (3.0, 100.0)[f], False) + (1.0 if f == 0 else 0.0))
        pi.append(_drawn_field(N, kIR, seed, 8 + f, (3.0, 100.0)[f], True) if case["fluct_pi"] else
                  torch.zeros((N, N, N), dtype=torch.float64, device="cuda"))
    return Exact(N, kIR, 100.0, True, phi, pi).outputs()


def _exact_spectrum(x, kIR):
    N = x.shape[0]
    d = torch.fft.fftn(x, norm="forward")
    i = torch.arange(N, device="cuda")
    n = torch.where(i < N // 2, i, i - N)
    r2 = n * n + (n * n).view(N, 1) + (n * n).view(N, 1, 1)
    length = r2.double().sqrt()
    bins = (length + 0.5).floor().long().reshape(-1)
    nb = math.ceil(math.sqrt(3.0) * N / 2.0) + 1
    count = torch.bincount(bins, minlength=nb)
    some = count.clamp(min=1).double()
    k = kIR * torch.bincount(bins, weights=length.reshape(-1), minlength=nb) / some
    P = torch.bincount(bins, weights=d.abs().square().reshape(-1), minlength=nb) / some
    return k, (2.0 * math.pi / kIR) ** 3 * P, None


def _exact_langevin(case, seed):
    N, dt = case["N"], 0.01
    (phi,), _ = _exact_fields(N, 1, case["dtype"], _generator(seed))
    draws = torch.arange(N ** 3 // 2, device="cuda")
    for s in range(case["steps"]):
        u1, u2 = _philox_uniforms(draws, (1 << 63) + s, seed)
        r, angle = (-2.0 * u1.log()).sqrt(), 2.0 * math.pi * u2
        xi = torch.stack([r * angle.cos(), r * angle.sin()], 1).view(N, N, N)
        phi = phi + dt * (_laplacian(phi, 1.0) - 0.5 * phi - 0.5 * phi ** 3) + math.sqrt(dt) * xi
    return phi


def _qmul(a, b):
    """Products of quaternions [4, ...] standing for a0 + i a.sigma."""
    out = torch.empty_like(a)
    out[0] = a[0] * b[0] - (a[1] * b[1] + a[2] * b[2] + a[3] * b[3])
    for c, d, e in ((1, 2, 3), (2, 3, 1), (3, 1, 2)):
        out[c] = a[0] * b[c] + b[0] * a[c] - (a[d] * b[e] - a[e] * b[d])
    return out


def _dagger(a):
    return torch.cat([a[:1], -a[1:]])


def _shift(x, d, s):
    return torch.roll(x, -s, x.dim() - 1 - d)


def _exact_su2(case, seed):
    N, dt = case["N"], 0.05
    U, E = _su2_start(N, _generator(seed))
    if case["dtype"] == "f32":
        U, E = U.float().double(), E.float().double()
    for _ in range(case["steps"]):
        for i in range(3):
            S = 0.0
            for j in range(3):
                if j != i:
                    Uj = _shift(U[j], j, -1)
                    S = S + _qmul(_qmul(_shift(U[j], i, 1), _dagger(_shift(U[i], j, 1))), _dagger(U[j]))
                    S = S + _qmul(_qmul(_dagger(_shift(Uj, i, 1)), _dagger(_shift(U[i], j, -1))), Uj)
            E[i] -= 2.0 * dt * _qmul(U[i], S)[1:]
        for i in range(3):
            e = E[i].square().sum(0, keepdim=True).sqrt()
            U[i] = _qmul(torch.cat([(dt * e).cos(), (dt * e).sin() / e * E[i]]), U[i])
    magnetic, G = 0.0, 0.0
    for i in range(3):
        for j in range(i + 1, 3):
            P = _qmul(_qmul(_qmul(U[i], _shift(U[j], i, 1)), _dagger(_shift(U[i], j, 1))), _dagger(U[j]))
            magnetic += float((2.0 * (1.0 - P[0])).mean())
        Um, Em = _shift(U[i], i, -1), torch.cat([torch.zeros_like(E[i][:1]), _shift(E[i], i, -1)])
        G = G + E[i] - _qmul(_qmul(_dagger(Um), Em), Um)[1:]
    g2 = G.square().sum(0)
    measured = [0.5 * float(E.square().sum((0, 1)).mean()), magnetic, float(g2.max().sqrt()),
                math.sqrt(float(g2.mean()))]
    return {"measured": measured, "U": U.cpu(), "E": E.cpu()}


def exact(case, seed):
    kind = case["kind"]
    if kind == "su2":
        return _exact_su2(case, seed)
    if kind == "langevin":
        return _exact_langevin(case, seed)
    if kind == "spectrum":
        phi, _ = _exact_fields(case["N"], case["nf"], case["dtype"], _generator(seed))
        return [_exact_spectrum(x, case["kIR"]) for x in phi]
    if kind == "init":
        energies, state = _exact_init(case, seed)
        return {"energies": energies, "state": state}
    if kind == "evolve":
        phi, pi = _exact_fields(case["N"], case["nf"], case["dtype"], _generator(seed))
        sim = Exact(case["N"], case["kIR"], case["q"], case["expanding"], phi, pi)
        energies, state = sim.steps(case["steps"], case["dt"], case["integrator"]).outputs()
        return {"energies": energies, "state": state}
    gen, energies, by_size = _generator(seed), [], {}
    for N, nf, q in _ensemble_members(case):
        phi, pi = _exact_fields(N, nf, case["dtype"], gen)
        sim = Exact(N, 0.5, q, True, phi, pi).steps(case["steps"], case["dt"], "verlet")
        energies += sim.outputs()[0]
        by_size.setdefault(N, ([], []))
        by_size[N][0].extend(sim.phi)
        by_size[N][1].extend(sim.pi)
    state = [torch.stack(x) for N in sorted(by_size) for x in by_size[N]]
    return {"energies": torch.tensor(energies), "state": state}

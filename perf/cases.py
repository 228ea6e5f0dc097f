"""Timed cases of the RK4IP library: calls a user's program makes through the public Python binding.

A case is a plain dict: the kind of call ("integrate" or "adjoint"), the lattice
(shape, box, basis), the precision, the number of paths and steps, and the options
of the problem (potential, nonlinearity, noise, scheme, pair potential, sampling).
``prepare`` builds what such a program holds (problem handle, field, sample
buffers), ``run`` makes one call on it, and ``exact`` is the same call written
plainly in torch with complex128 transforms, without this repository's code.

Fields advance in place from call to call, as a simulation does that reports
between chunks of steps.  Samples and gradients are FP64 buffers; a complex64 run
hands them on in float32, the precision it has.
"""
import math

import torch

from paper_1204_4255_gb300 import xsde

NOISES = {  # name -> (noise kind, coupling)
    "none": (xsde.XSDE_NOISE_NONE, xsde.XSDE_COUPLE_ADDITIVE),
    "real": (xsde.XSDE_NOISE_WIENER_REAL, xsde.XSDE_COUPLE_ADDITIVE),
    "complex": (xsde.XSDE_NOISE_WIENER_COMPLEX, xsde.XSDE_COUPLE_ADDITIVE),
    "phase": (xsde.XSDE_NOISE_WIENER_REAL, xsde.XSDE_COUPLE_MULTIPLICATIVE),
}


def _case(name, shape, dtype, npaths, nsteps, **more):
    c = {"call": "integrate", "shape": shape, "box": 12.0, "dtype": dtype, "npaths": npaths, "nsteps": nsteps,
         "dt": 1e-4, "g": 0.0, "trap": True, "noise": "none", "amplitude": 0.0, "scheme": "rk4ip", "basis": "",
         "charge": 0.0, "every": 0, "points": False, "state": "gas"}
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the bright soliton of the cubic NLS in double precision: one small path, a call bound by latency
        _case("soliton_1d_c128", "256", "c128", 1, 200, box=20.0, dt=1e-3, g=-1.0, trap=False, state="sech"),
        # a truncated-Wigner ensemble: additive complex noise, all moments sampled
        _case("truncated_wigner_1d", "1024", "c64", 4096, 50, box=50.0, dt=5e-4, g=0.1, trap=False,
              noise="complex", amplitude=0.01, every=25, points=True, state="wigner"),
        # an ensemble of scalar SDEs (Ornstein-Uhlenbeck), sampled
        _case("ornstein_uhlenbeck", "", "c64", 65536, 1000, dt=1e-3, trap=False, noise="real", amplitude=0.5,
              every=100, points=True, state="ones"),
        # one 2D condensate: a field that stays in L2, a chain of short launches
        _case("gpe_2d_single", "512x512", "c64", 1, 50, g=500.0),
        # many 2D condensates at once, norm and energy sampled: fields beyond L2, the benchmark's lattice
        _case("gpe_2d_ensemble", "512x512", "c64", 64, 20, g=500.0, every=20),
        # the noisy trap of many paths on an uneven lattice, an odd number of paths
        _case("noisy_trap_2d", "128x1024", "c64", 37, 20, g=100.0, noise="phase", amplitude=0.05),
        # 2D condensates in double precision
        _case("gpe_2d_c128", "256x256", "c128", 8, 10, g=500.0, every=10),
        # 3D condensates
        _case("gpe_3d", "128x128x128", "c64", 2, 10, box=10.0, g=200.0),
        # a charged condensate: the non-local pair potential, a convolution at every evaluation
        _case("charged_2d", "256x256", "c64", 16, 5, g=10.0, charge=1.0, state="gauss"),
        # a reflection-symmetric condensate on half its domain: cosine basis in x, Fourier in y
        _case("symmetric_2d", "256x512", "c64", 16, 10, box=7.0, g=20.0, basis="cos,", state="gauss"),
        # the semi-implicit scheme for a stochastic condensate
        _case("semi_implicit_2d", "512x512", "c64", 24, 20, g=500.0, noise="complex", amplitude=0.01,
              scheme="semi_implicit"),
        # the gradient of a control problem: the forward sweep and the adjoint of every step
        _case("adjoint_1d", "1024", "c64", 1, 300, call="adjoint", box=20.0, dt=1e-3, g=1.0, trap=True, state="gauss"),
    ]


# point-steps of the largest listed case, and what a double-precision draw may take of them
MOST_POINT_STEPS = 64 * 512 * 512 * 20
MOST_POINT_STEPS_C128 = MOST_POINT_STEPS // 16


def draw(rng):
    """One more case of the ranges above: lattices from the smallest to the largest of each
    family, either precision, path counts that fill no tile, with and without the options."""
    family = rng.choice(["sde", "1d", "1d", "2d", "2d", "2d", "3d", "3d", "charged", "symmetric", "semi", "adjoint"])
    dtype = rng.choice(["c64", "c64", "c128"])

    def two_to(lo, hi):
        return 1 << rng.randint(lo, hi)

    dims = {"sde": 0, "1d": 1, "adjoint": 1, "3d": 3, "charged": rng.randint(1, 2),
            "symmetric": rng.randint(1, 2)}.get(family, 2)
    lo, hi = {0: (0, 0), 1: (6, 11), 2: (6, 10), 3: (5, 7)}[dims]
    if family == "adjoint":
        lo = 8
    n = [two_to(lo, hi) for _ in range(dims)]
    most = MOST_POINT_STEPS if dtype == "c64" else MOST_POINT_STEPS_C128
    if family in ("sde", "1d") and dtype == "c128":
        most //= 4
    if family == "adjoint":
        nsteps, npaths = rng.randint(50, 300), rng.randint(1, 5)
    elif family == "sde":
        nsteps, npaths = rng.randint(100, 1000), int(2 ** rng.uniform(8, 16))
    else:
        nsteps = rng.randint(4, 60) if dims > 1 else rng.randint(20, 300)
        room = most // (math.prod(n) * nsteps)
        room = min(room, (1 << 24) // math.prod(n), 65535 // n[0] if dims == 3 else 4096)
        npaths = max(1, int(2 ** rng.uniform(0, math.log2(max(2, room)))))
        while npaths * math.prod(n) * nsteps > most and nsteps > 1:
            nsteps //= 2
    box = {0: 1.0, 1: 20.0, 2: 12.0, 3: 10.0}[dims]
    if family == "symmetric":
        box = 7.0
    dx = min([(1 if family == "symmetric" else 2) * box / k for k in n], default=1.0)
    more = {"box": box, "dt": 1e-3 if dims == 0 else min(1e-3, round(0.2 * dx * dx, 6)),
            "g": {0: 0.0, 1: 1.0, 2: 100.0, 3: 200.0}[dims], "state": "gas" if dims > 1 else "gauss"}
    if family == "sde":
        more.update(noise=rng.choice(["real", "phase"]), amplitude=0.5, every=rng.randint(20, 100), trap=False,
                    points=rng.random() < 0.5, state="ones")
    elif family == "adjoint":
        more.update(call="adjoint")
    elif family == "charged":
        more.update(charge=1.0, g=10.0, state="gauss")
    elif family == "symmetric":
        more.update(basis=rng.choice(["cos,", "sin,"] if dims == 2 else ["cos", "sin"]), g=10.0, state="gauss")
    elif family == "semi":
        more.update(scheme="semi_implicit")
    if family in ("1d", "2d", "3d", "semi"):
        more["noise"] = rng.choice(["none", "none", "complex", "phase"])
        more["amplitude"] = 0.0 if more["noise"] == "none" else 0.01
        if rng.random() < 0.4:
            more["every"] = rng.randint(1, nsteps)
            more["points"] = rng.random() < 0.3
    return _case("", "x".join(map(str, n)), dtype, npaths, nsteps, **more)


# --- the lattice and the inputs ----------------------------------------------------------

def _shape(case):
    return tuple(int(k) for k in case["shape"].split("x")) if case["shape"] else ()


def _bases(case):
    got = [b for b in case["basis"].split(",")] if case["basis"] else []
    codes = {"": xsde.XSDE_BASIS_FOURIER, "cos": xsde.XSDE_BASIS_COS, "sin": xsde.XSDE_BASIS_SIN}
    return tuple(codes[b] for b in got)


def _limits(case):
    """(xmin, xmax) per dimension: [-box, box), or (0, box) along a cosine / sine dimension."""
    bases = _bases(case) or (0,) * len(_shape(case))
    return tuple(0.0 if b else -case["box"] for b in bases), (case["box"],) * len(bases)


def _axes(case):
    lo, hi = _limits(case)
    bases = _bases(case) or (0,) * len(lo)
    out = []
    for d, n in enumerate(_shape(case)):
        x = torch.arange(n, dtype=torch.float64, device="cuda") + (0.5 if bases[d] else 0.0)
        x = lo[d] + x * ((hi[d] - lo[d]) / n)
        out.append(x.reshape([-1 if k == d else 1 for k in range(len(lo))]))
    return out


def _dV(case):
    lo, hi = _limits(case)
    return math.prod((b - a) / n for a, b, n in zip(lo, hi, _shape(case)))


def _noise_seed(seed):
    return 1000003 * (int(seed) + 1)


def _field(case, seed):
    """The initial field [npaths, *shape] in complex128, from the seed alone."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    shape, axes, P = _shape(case), _axes(case), case["npaths"]

    def normal(*s):
        return torch.randn(s, generator=gen, dtype=torch.float64, device="cuda")

    def uniform(*s):
        return torch.rand(s, generator=gen, dtype=torch.float64, device="cuda")

    col = (P,) + (1,) * len(shape)
    if case["state"] == "ones":      # SDE paths, started near 1
        psi = (1.0 + 0.01 * normal(P)).to(torch.complex128)
    elif case["state"] == "sech":    # a bright soliton, displaced and moving a little
        x0, v = uniform(*col) - 0.5, 0.2 * uniform(*col)
        psi = torch.polar(1.0 / torch.cosh(axes[0] - x0), v * axes[0])
    elif case["state"] == "wigner":  # uniform gas of density 100 with half a quantum of vacuum noise
        s = math.sqrt(1.0 / (4.0 * _dV(case)))
        psi = torch.complex(10.0 + s * normal(P, *shape), s * normal(P, *shape))
    elif case["state"] == "gas":     # Thomas-Fermi condensate of unit norm with phase noise
        g = case["g"]
        mu = math.sqrt(g / math.pi) if len(shape) == 2 else (15.0 * g / (8.0 * math.pi * 2.0 ** 1.5)) ** 0.4
        amp = (torch.clamp(mu - sum(0.5 * x * x for x in axes), min=0.0) / g).sqrt()
        amp = amp / torch.sqrt((amp * amp).sum() * _dV(case))
        psi = torch.polar(amp.expand(P, *shape).contiguous(), 0.01 * normal(P, *shape))
    else:                            # displaced Gaussian ground states
        psi = torch.ones(col, dtype=torch.complex128, device="cuda")
        bases = _bases(case) or (0,) * len(shape)
        w = 0.8 + 0.45 * uniform(*col)
        for x, b in zip(axes, bases):
            x0 = 0.0 if b else 2.0 * uniform(*col) - 1.0
            lead = math.sqrt(2.0) * x if b == xsde.XSDE_BASIS_SIN else 1.0
            psi = psi * (math.pi ** -0.25 / torch.sqrt(w) * lead * torch.exp(-0.5 * ((x - x0) / w) ** 2))
    return psi.expand(P, *shape).contiguous()


def _pair_kernel(case):
    """Fourier kernel (complex128, on the GPU) of the softened Coulomb pair potential, or None."""
    if not case["charge"]:
        return None
    shape, r2 = _shape(case), 0.25
    for d, n in enumerate(shape):
        j = torch.fft.fftfreq(n, 1.0 / n, dtype=torch.float64, device="cuda")
        r2 = r2 + ((j * (2.0 * case["box"] / n)) ** 2).reshape([-1 if k == d else 1 for k in range(len(shape))])
    return torch.fft.fftn((case["charge"] / torch.sqrt(r2) * _dV(case)).to(torch.complex128))


def _control(case, seed):
    """The control problem's potential rows [nsteps, n] and target state, FP64."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed) + 77)
    (x,), (n,) = _axes(case), _shape(case)
    t = torch.arange(case["nsteps"], dtype=torch.float64, device="cuda")[:, None] / case["nsteps"]
    V = 0.5 * x * x + torch.zeros_like(t)
    for k in range(1, 6):
        a, b, c = torch.rand(3, generator=gen, dtype=torch.float64, device="cuda")
        V = V + 0.1 * (a + 0.5) * torch.cos(2 * math.pi * (k * x / (2 * case["box"]) + b)) * torch.cos(2 * math.pi * (k * t + c))
    return V, (math.pi ** -0.25 * torch.exp(-0.5 * (x - 2.0) ** 2)).to(torch.complex128)


def _c0(case):
    return complex(-1.0, 0.0) if case["state"] == "ones" and case["noise"] == "real" else \
        complex(0.0, 1.0) if case["state"] == "ones" else 0j


def prepare(case, seed):
    shape = _shape(case)
    lo, hi = _limits(case)
    cx = torch.complex64 if case["dtype"] == "c64" else torch.complex128
    real = torch.float32 if case["dtype"] == "c64" else torch.float64
    P = xsde.Problem(shape, lo, hi, case["dtype"], basis=_bases(case))
    kind, coupling = NOISES[case["noise"]]
    ops = dict(c0=_c0(case), c2=-0.5j if shape else 0j, g=case["g"])
    state = {"case": case, "problem": P, "psi": _field(case, seed).to(cx), "real": real}
    if case["call"] == "adjoint":
        V, target = _control(case, seed)
        state.update(V=V.to(real), target=target.to(cx))
        P.set_operators(pot_kind=xsde.XSDE_POT_TABLE, V=state["V"], **ops)
        return state
    P.set_operators(pot_kind=xsde.XSDE_POT_HARMONIC if case["trap"] else xsde.XSDE_POT_NONE,
                    omega=(1.0,) * len(shape), noise_kind=kind, coupling=coupling, seed=_noise_seed(seed),
                    amplitude=case["amplitude"], **ops)
    if case["scheme"] == "semi_implicit":
        xsde.xsde_set_scheme(P.prob, xsde.XSDE_SCHEME_SEMI_IMPLICIT)
    if case["charge"]:
        P.set_nonlocal(_pair_kernel(case).cpu().numpy())
    if case["every"]:
        nsamp = case["nsteps"] // case["every"] + 1
        which = xsde.XSDE_MOM_NORM | xsde.XSDE_MOM_ENERGY
        state["per_path"] = torch.zeros((nsamp, case["npaths"], 2), dtype=torch.float64, device="cuda")
        if case["points"]:
            which |= xsde.XSDE_MOM_MOD2 | xsde.XSDE_MOM_MOD4
            state["per_point"] = torch.zeros((nsamp, math.prod(shape), 2), dtype=torch.float64, device="cuda")
        P.moments(case["every"], which, state["per_path"], state.get("per_point"))
    return state


def run(state):
    case, P, psi = state["case"], state["problem"], state["psi"]
    if case["call"] == "adjoint":
        loss, dLdV = xsde.adjoint(P, psi, state["target"], case["dt"], case["nsteps"])
        return {"loss": loss.to(state["real"]), "dLdV": dLdV.to(state["real"])}
    P.integrate(psi, case["dt"], case["nsteps"])
    out = {"psi": psi}
    for k in ("per_path", "per_point"):
        if k in state:
            out[k] = state[k].to(state["real"])
    return out


def work(case):
    pts = math.prod(_shape(case)) * case["npaths"]
    cb = 8 if case["dtype"] == "c64" else 16
    nbytes = 2 * pts * cb
    # per point and step: eight transforms at 5 log2(n) and about 100 operations of the stages
    levels = math.log2(max(2, math.prod(_shape(case)))) if _shape(case) else 0.0
    transforms = 4 if case["scheme"] == "semi_implicit" else 8 + (8 if case["charge"] else 0)
    flops = pts * case["nsteps"] * (transforms * 5 * levels + 100)
    if case["call"] == "adjoint":
        flops *= 3
        nbytes = pts * cb + math.prod(_shape(case)) * (cb + case["nsteps"] * (cb // 2) * 2)
    if case["every"]:
        nsamp = case["nsteps"] // case["every"] + 1
        nbytes += nsamp * 16 * (case["npaths"] + (math.prod(_shape(case)) if case["points"] else 0))
    return {"bytes": float(nbytes), "flops": float(flops)}


# --- the same calls in plain torch, complex128 ----------------------------------------------

def _philox_normals(seed, npts, npaths, step):
    """(z0, z1) [npaths, npts] of Philox4x32-10 at counter (point, path, step + 1, 0), Box-Muller in FP64."""
    mask = 0xFFFFFFFF
    c0 = torch.arange(npts, dtype=torch.int64, device="cuda")[None, :].expand(npaths, npts)
    c1 = torch.arange(npaths, dtype=torch.int64, device="cuda")[:, None].expand(npaths, npts)
    c2 = torch.full_like(c0, step + 1)
    c3 = torch.zeros_like(c2)
    k0, k1 = seed & mask, (seed >> 32) & mask

    def mul(m, c):   # (high, low) words of a 32 x 32 bit product, without leaving int64
        a, b = m * (c >> 16), m * (c & 0xFFFF)
        return (a + (b >> 16)) >> 16, ((a << 16) + b) & mask

    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c0)
        h1, l1 = mul(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    u0, u1 = (c0.double() + 0.5) * 2.0 ** -32, (c1.double() + 0.5) * 2.0 ** -32
    r = torch.sqrt(-2.0 * torch.log(u0))
    return r * torch.cos(2 * math.pi * u1), r * torch.sin(2 * math.pi * u1)


def _extended(u, bases, cut=None):
    """u continued evenly (cosine) or oddly (sine) to twice its length, or cut back."""
    for d, b in enumerate(bases):
        if b and cut is None:
            u = torch.cat([u, u.flip(d + 1) * (1.0 if b == xsde.XSDE_BASIS_COS else -1.0)], d + 1)
        elif b:
            u = u.narrow(d + 1, 0, cut[d])
    return u


def exact(case, seed):
    shape, dt, g = _shape(case), case["dt"], case["g"]
    bases = _bases(case) or (0,) * len(shape)
    dims = tuple(range(1, len(shape) + 1))
    cx = torch.complex64 if case["dtype"] == "c64" else torch.complex128
    psi = _field(case, seed).to(cx).to(torch.complex128)
    lo, hi = _limits(case)
    k2 = torch.zeros((), dtype=torch.float64, device="cuda")
    for d, n in enumerate(shape):
        m = n * (2 if bases[d] else 1)
        k = 2 * math.pi * torch.fft.fftfreq(m, (hi[d] - lo[d]) / n, dtype=torch.float64, device="cuda")
        k2 = k2 + (k * k).reshape([-1 if q == d else 1 for q in range(len(shape))])
    c0 = _c0(case)
    E = torch.exp((c0 + (-0.5j if shape else 0j) * k2) * (0.5 * dt))

    def D(u):
        if not shape:
            return u * E
        v = torch.fft.ifftn(torch.fft.fftn(_extended(u, bases), dim=dims) * E, dim=dims)
        return _extended(v, bases, cut=shape)

    khat = _pair_kernel(case)

    def pair(u):
        return 0.0 if khat is None else torch.fft.ifftn(torch.fft.fftn(u.abs() ** 2 + 0j, dim=dims) * khat, dim=dims).real

    trap = sum(0.5 * x * x for x in _axes(case)) if case["trap"] and shape else 0.0

    def rate(u, V, xi_a):
        return dt * (-1j * (V + pair(u) + g * (u.real ** 2 + u.imag ** 2)) * u + xi_a)

    def rk4ip(a, V, xi_a):
        def N(u):
            return rate(u, V, xi_a)
        aI, k1 = D(a), D(N(a))
        q2 = N(aI + 0.5 * k1)
        q3 = N(aI + 0.5 * q2)
        q4 = N(D(aI + q3))
        return D(aI + k1 / 6 + q2 / 3 + q3 / 3) + q4 / 6

    if case["call"] == "adjoint":
        V, target = _control(case, seed)
        real = torch.float32 if case["dtype"] == "c64" else torch.float64
        V = V.to(real).double().requires_grad_(True)
        target = target.to(cx).to(torch.complex128)
        a = psi
        for n in range(case["nsteps"]):
            a = rk4ip(a, V[n], 0.0)
        over = (target.conj() * a).sum(-1) * _dV(case)
        loss = (1.0 - over.real ** 2 - over.imag ** 2).sum()
        loss.backward()
        return {"loss": loss.detach().reshape(1), "dLdV": V.grad}

    scale = case["amplitude"] * math.sqrt(1.0 / (dt * _dV(case)))
    every, per_path, per_point = case["every"], [], []
    weight = 1.0
    for b in bases:   # the stored points are half of an extended dimension's
        weight *= 0.5 if b else 1.0
    for n in range(case["nsteps"] + 1):
        if every and n % every == 0:
            rho = psi.real ** 2 + psi.imag ** 2
            flat = rho.reshape(case["npaths"], -1)
            local = (trap * rho + 0.5 * g * rho * rho + 0.5 * pair(psi) * rho).reshape(case["npaths"], -1).sum(1)
            if shape:
                s = torch.fft.fftn(_extended(psi, bases), dim=dims)
                h = (1j * (c0 - 0.5j * k2)).real
                kin = weight * (h * (s.real ** 2 + s.imag ** 2)).reshape(case["npaths"], -1).sum(1) / h.numel()
            else:
                kin = (1j * c0).real * flat.sum(1)
            per_path.append(torch.stack([flat.sum(1) * _dV(case), (local + kin) * _dV(case)], 1))
            per_point.append(torch.stack([flat.mean(0), (flat * flat).mean(0)], 1))
        if n == case["nsteps"]:
            break
        V, xi_a = trap, 0.0
        if case["noise"] != "none":
            z0, z1 = _philox_normals(_noise_seed(seed), math.prod(shape), case["npaths"], n)
            z0, z1 = z0.reshape(psi.shape), z1.reshape(psi.shape)
            if case["noise"] == "phase":
                V = V + scale * z0
            else:
                xi_a = scale * (torch.complex(z0, z1) * math.sqrt(0.5) if case["noise"] == "complex" else z0)
        if case["scheme"] == "semi_implicit":
            aI = D(psi)
            m = aI
            for _ in range(3):
                m = aI + 0.5 * rate(m, V, xi_a)
            psi = D(2 * m - aI)
        else:
            psi = rk4ip(psi, V, xi_a)
    out = {"psi": psi}
    if every:
        out["per_path"] = torch.stack(per_path)
        if case["points"]:
            out["per_point"] = torch.stack(per_point)
    return out

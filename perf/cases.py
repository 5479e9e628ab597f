"""The work that programs have this library do, as cases that can be timed.

Four kinds of call, each through the public binding:

  lattice  one lattice: f = f^eq of device fields, n time steps, moments into
           device arrays (the use shown first in README.md, on torch tensors)
  batch    many independent lattices that stay on the device: n time steps,
           every lattice's drift sums and its moments into device arrays
  solve    a batch of small lattices from page-locked host fields to host
           moments and drift sums (lbm_batch_solve_packed / _wait)
  vn       a von Neumann sweep: the spectrum of G(k) for many (k, flow)

The sizes are those of the workloads that bench.py, lbm_inputs and the tests
run (64^2 pulse, 101^2 point source, 512 x 16 plane waves, the section 5.2
pulse at 128^2 .. 1024^2, one 8192^2 lattice, the lattice sweep of areas 32^2
.. 1024^2, small sweeps of 32^2 .. 56^2, von Neumann sweeps), and odd ones
between them.  Step counts are cut where the full run (1000 steps of 8192^2)
would only repeat itself.
"""
import math
import random

import numpy as np
import torch

from paper_1107_4543_gb300 import lbm

# relaxation rates (s_e, s_eps, s_q, s_nu): the optimized set for uniform
# flows (Table 5 A), the one for zero mean flow (Table 4 A, point source) and
# the Lallemand-Luo rates at viscosity 1e-3
RATES = {
    "OPT": (1.99, 1.962820428, 1.992761413, 1.999960001),
    "OPT-Z": (1.99044751, 2.0, 0.00875438872, 1.99044751),
    "LL": (1.64, 1.54, 1.9, 1.0 / (0.5 + 3.0 * 1e-3)),
}


def s_ll(name):
    """Rates in Lallemand-Luo order (rho, e, eps, jx, qx, jy, qy, pxx, pxy)."""
    e, eps, q, nu = RATES[name]
    return np.array([0.0, e, eps, 0.0, q, 0.0, q, nu, nu])


def lattice(name, nx, ny, dtype, steps, rates, init, u0=0.0, source=False):
    return dict(kind="lattice", name=name, nx=nx, ny=ny, dtype=dtype, steps=steps, rates=rates,
                init=init, u0=u0, source=source)


def many(kind, name, lattices, side_lo, side_hi, dtype, steps):
    return dict(kind=kind, name=name, lattices=lattices, side_lo=side_lo, side_hi=side_hi,
                dtype=dtype, steps=steps)


def listed():
    return [
        # section 5.1: acoustic point source on the paper's 101 x 101 lattice
        lattice("source_101_f32", 101, 101, "f32", 512, "OPT-Z", "rest", source=True),
        # the smallest solve: a 64^2 pulse in plain FP64
        lattice("pulse_64_f64", 64, 64, "f64", 200, "LL", "pulse"),
        # section 4.2 plane waves with a mean flow, 512 x 16
        lattice("wave_512x16_f32", 512, 16, "f32", 1000, "OPT", "wave", u0=0.1),
        # section 5.2: the pulse until t = 0.4 (0.4 N steps), fits in L2
        lattice("pulse_512_f32", 512, 512, "f32", 205, "OPT", "pulse"),
        # one large lattice: pulse plus vortices, per storage type
        lattice("large_8192_f32", 8192, 8192, "f32", 64, "OPT", "vortices"),
        lattice("large_4097x3071_f16", 4097, 3071, "f16", 100, "OPT", "vortices"),
        lattice("large_1500x1111_bf16", 1500, 1111, "bf16", 150, "LL", "vortices"),
        lattice("large_2048_f64dev", 2048, 2048, "f64dev", 25, "OPT", "vortices", u0=0.1),
        # sweeps over many lattices of mixed size (the headline workload, a
        # quarter of its lattices)
        many("batch", "sweep_128_f32", 128, 32, 1024, "f32", 500),
        many("batch", "sweep_128_f16", 128, 32, 1024, "f16", 500),
        # many small lattices, from host fields to host moments
        many("solve", "small_1024_f32", 1024, 32, 56, "f32", 500),
        # section 4.1: von Neumann sweep with mean flows
        dict(kind="vn", name="vn_32768", cases=32768),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    case = _draw(rng)
    del case["name"]
    return case


def _draw(rng):
    kind = rng.choice(["small", "small", "large", "large", "batch", "solve", "vn"])
    if kind == "small":
        nx, ny = _log(rng, 16, 700), _log(rng, 16, 700)
        dtype = rng.choice(["f32", "f32", "f16", "bf16", "f64"])
        source = rng.random() < 0.3
        init = "rest" if source else rng.choice(["pulse", "wave"])
        steps = _log(rng, 50, 1000)
        return lattice("", nx, ny, dtype, steps, rng.choice(["OPT", "LL"]), init,
                       u0=0.0 if source else rng.choice([0.0, 0.1]), source=source)
    if kind == "large":
        nx, ny = _log(rng, 700, 8192), _log(rng, 700, 8192)
        dtype = rng.choice(["f32", "f32", "f16", "f16", "bf16", "f64", "f64dev"])
        cost = {"f32": 1, "f16": 0.6, "bf16": 0.6, "f64": 30, "f64dev": 15}[dtype]
        most = max(3, min(150, int(4.0e9 / (nx * ny * cost))))
        return lattice("", nx, ny, dtype, rng.randint(min(8, most), most),
                       rng.choice(["OPT", "LL"]), "vortices", u0=rng.choice([0.0, 0.1]))
    if kind == "batch":
        hi = rng.choice([400, 700, 1024])
        return many("batch", "", _log(rng, 8, 128), 32, hi, rng.choice(["f32", "f16", "bf16"]),
                    rng.randint(51, 500))
    if kind == "solve":
        return many("solve", "", _log(rng, 64, 1024), rng.choice([16, 32]), rng.choice([48, 56, 80]),
                    rng.choice(["f32", "f16"]), rng.randint(51, 500))
    return dict(kind="vn", name="", cases=_log(rng, 257, 65536))


# ------------------------------------------------------------------ inputs
def _gauss(nx, ny, amp, b, xc, yc, dev):
    """rho' = amp exp(-ln2 eta^2 / b^2), minimum-image distance to (xc, yc)."""
    x = torch.arange(nx, dtype=torch.float64, device=dev)
    y = torch.arange(ny, dtype=torch.float64, device=dev)
    dx = (x - xc + 0.5 * nx) % nx - 0.5 * nx
    dy = (y - yc + 0.5 * ny) % ny - 0.5 * ny
    al = math.log(2.0) / (b * b)
    return torch.outer(amp * torch.exp(-al * dy * dy), torch.exp(-al * dx * dx))


def _fields(case, rng, dev="cuda"):
    """(rho, ux, uy) of one lattice, (ny, nx) float64 on `dev`."""
    nx, ny, u0 = case["nx"], case["ny"], case["u0"]
    rho = torch.ones((ny, nx), dtype=torch.float64, device=dev)
    ux = torch.full((ny, nx), float(u0), dtype=torch.float64, device=dev)
    uy = torch.zeros((ny, nx), dtype=torch.float64, device=dev)
    amp = math.exp(rng.uniform(math.log(2e-4), math.log(1e-3)))
    if case["init"] == "wave":  # right-running acoustic wave along x
        m = rng.randint(2, max(2, nx // 8))
        ph = rng.uniform(0.0, 2.0 * math.pi)
        x = torch.arange(nx, dtype=torch.float64, device=dev)
        c = torch.cos(2.0 * math.pi * m / nx * x + ph)[None, :]
        rho += amp * c
        ux += amp / math.sqrt(3.0) * c
        # and a transverse (shear) wave of a tenth of its amplitude
        uy += 0.1 * amp * torch.sin(2.0 * math.pi * rng.randint(1, 3) / nx * x)[None, :]
    elif case["init"] in ("pulse", "vortices"):
        b = max(3.0, 0.04 * min(nx, ny)) if case["init"] == "pulse" else 20.0
        rho += _gauss(nx, ny, amp, b, rng.uniform(0, nx), rng.uniform(0, ny), dev)
    if case["init"] == "vortices":  # divergence-free modes, rms about 1e-4
        x = 2.0 * math.pi / nx * torch.arange(nx, dtype=torch.float64, device=dev)
        y = 2.0 * math.pi / ny * torch.arange(ny, dtype=torch.float64, device=dev)
        for _ in range(6):
            p, q = rng.randint(1, 64), rng.choice([-1, 1]) * rng.randint(1, 64)
            a = rng.gauss(0.0, 1e-4) / math.hypot(p / nx, q / ny) / math.sqrt(6.0)
            f1, f2 = rng.uniform(0, 6.28), rng.uniform(0, 6.28)
            ux.addr_(torch.sin(q * y + f2), torch.cos(p * x + f1), alpha=-a * q / ny)
            uy.addr_(torch.cos(q * y + f2), torch.sin(p * x + f1), alpha=a * p / nx)
    return rho, ux, uy


def _source(case, rng):
    """Point source of section 5.1: (x, y, amplitude, period)."""
    return (rng.randrange(case["nx"]), rng.randrange(case["ny"]), rng.uniform(0.005, 0.01),
            rng.uniform(16.0, 24.0))


def _members(case, seed):
    """A batch's lattices: areas log-uniform between side_lo^2 and side_hi^2,
    aspect ratio log-uniform in [1/4, 4]; rates OPT or LL per lattice.  The
    sizes belong to the case, the rest to the seed."""
    shape = random.Random(case["lattices"] * 7919 + case["side_hi"])
    rng = random.Random(seed)
    out = []
    for _ in range(case["lattices"]):
        a = math.exp(shape.uniform(2 * math.log(case["side_lo"]), 2 * math.log(case["side_hi"])))
        if case["side_hi"] > 100:
            r = math.exp(shape.uniform(math.log(0.25), math.log(4.0)))
        else:
            r = 1.0
        out.append(dict(nx=max(8, int(round(math.sqrt(a * r)))),
                        ny=max(8, int(round(math.sqrt(a / r)))), rates=rng.choice(["OPT", "LL"]),
                        amp=math.exp(rng.uniform(math.log(1e-4), math.log(1e-3))),
                        xc=rng.random(), yc=rng.random()))
    return out


class State:
    """What a program keeps between calls; the handles go with it."""

    def __init__(self, case):
        self.case = case
        self.handles = []
        self.batch = None

    def __del__(self):
        if self.batch is not None:
            lbm.lbm_batch_destroy(self.batch)
        for h in self.handles:
            lbm.lbm_destroy(h)


_STREAM = []


def _stream():
    """The one stream on which the program works on its single lattices."""
    if not _STREAM:
        _STREAM.append(torch.cuda.Stream())
    return _STREAM[0]


def prepare(case, seed):
    rng = random.Random(seed)
    st = State(case)
    if case["kind"] == "lattice":
        st.fields = _fields(case, rng)
        h = lbm.lbm_create(case["nx"], case["ny"], s_ll(case["rates"]), 1.0, (case["u0"], 0.0),
                           lbm.DTYPES[case["dtype"]])
        st.handles.append(h)
        lbm.lbm_set_stream(h, _stream())
        if case["source"]:
            lbm.lbm_set_source(h, *_source(case, rng))
        st.out = tuple(torch.empty_like(st.fields[0]) for _ in range(3))
        torch.cuda.synchronize()
    elif case["kind"] in ("batch", "solve"):
        members = _members(case, seed)
        rho = []
        for m in members:
            h = lbm.lbm_create(m["nx"], m["ny"], s_ll(m["rates"]), 1.0, (0.0, 0.0),
                               lbm.DTYPES[case["dtype"]])
            st.handles.append(h)
            lbm.lbm_set_stream(h, _stream())
            rho.append(1.0 + _gauss(m["nx"], m["ny"], m["amp"], 4.0, m["xc"] * m["nx"],
                                    m["yc"] * m["ny"], "cuda"))
        if case["kind"] == "batch":
            flat = torch.cat([r.reshape(-1) for r in rho])
            zero = torch.zeros_like(flat)
            st.moments = tuple(torch.empty_like(flat) for _ in range(3))
            # member k's slices of the packed moment arrays
            st.out = list(zip(*(m.split([r.numel() for r in rho]) for m in st.moments)))
            torch.cuda.synchronize()
            for h, r, z in zip(st.handles, rho, zero.split([r.numel() for r in rho])):
                lbm.lbm_init_field_dev(h, r, z, z)
            torch.cuda.synchronize()
        else:
            nodes = sum(r.numel() for r in rho)
            st.fin = tuple(lbm.host_array(nodes) for _ in range(3))
            st.fout = tuple(lbm.host_array(nodes) for _ in range(3))
            st.drift = np.zeros((len(members), 4))
            torch.from_numpy(st.fin[0]).copy_(torch.cat([r.reshape(-1) for r in rho]))
        st.batch = lbm.lbm_batch_create(st.handles)
    else:
        r = np.random.default_rng(seed)
        n = case["cases"]
        k, th, ph = r.uniform(0.01, math.pi, n), r.uniform(0, 2 * math.pi, n), r.uniform(0, 6.28, n)
        u = r.uniform(0.0, 0.2, n)
        sets = np.stack([s_ll("OPT"), s_ll("LL")])
        st.args = (k * np.cos(th), k * np.sin(th), u * np.cos(ph), u * np.sin(ph),
                   np.ascontiguousarray(sets[r.integers(0, 2, n)]))
    return st


def run(st):
    case = st.case
    if case["kind"] == "lattice":
        h = st.handles[0]
        lbm.lbm_init_field_dev(h, *st.fields)
        lbm.lbm_step(h, case["steps"])
        lbm.lbm_moments_dev(h, *st.out)
        return {"rho": st.out[0], "ux": st.out[1], "uy": st.out[2]}
    if case["kind"] == "batch":
        lbm.lbm_batch_step(st.batch, case["steps"])
        drift = lbm.lbm_batch_drift(st.batch, len(st.handles))
        for h, out in zip(st.handles, st.out):
            lbm.lbm_moments_dev(h, *out)
        return {"rho": st.moments[0], "ux": st.moments[1], "uy": st.moments[2], "drift": drift}
    if case["kind"] == "solve":
        lbm.lbm_batch_solve_packed(st.batch, case["steps"], st.fin, st.fout, st.drift)
        lbm.lbm_batch_wait(st.batch)
        return {"rho": st.fout[0], "ux": st.fout[1], "uy": st.fout[2], "drift": st.drift}
    lam = lbm.lbm_vn_eigs(*st.args)
    # the eigenvalues come in no particular order: real and imaginary parts
    # sorted per case
    return {"spectra": torch.view_as_real(torch.from_numpy(lam)).sort(dim=1).values}


# ------------------------------------------------------------------- work
# arithmetic of one lattice update (moments, equilibrium, relaxation and
# back-transform of one node) and of one 9 x 9 complex eigenproblem (the
# Hessenberg reduction and about two QR sweeps per eigenvalue)
FLOPS_PER_UPDATE = 130
FLOPS_PER_SPECTRUM = 60000


def work(case):
    """One pass: the initial fields read, the moments written, and the
    arithmetic of every lattice update."""
    if case["kind"] == "vn":
        return {"bytes": case["cases"] * 8 * (4 + 9 + 18),
                "flops": case["cases"] * FLOPS_PER_SPECTRUM}
    if case["kind"] in ("batch", "solve"):
        nodes = sum(m["nx"] * m["ny"] for m in _members(case, 0))
    else:
        nodes = case["nx"] * case["ny"]
    return {"bytes": 48 * nodes, "flops": FLOPS_PER_UPDATE * nodes * case["steps"]}


# ------------------------------------------------------------------ exact
C = np.array([(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)])


def _moment_matrix():
    """Lallemand-Luo moments rho, jx, jy, e, eps, qx, qy, pxx, pxy of D2Q9."""
    x, y = C[:, 0].astype(float), C[:, 1].astype(float)
    c2 = x * x + y * y
    return np.stack([np.ones(9), x, y, 3 * c2 - 4, 4.5 * c2 * c2 - 10.5 * c2 + 4,
                     (3 * c2 - 5) * x, (3 * c2 - 5) * y, x * x - y * y, x * y])


def _meq(rho, jx, jy):
    q = (jx * jx + jy * jy) / rho
    return torch.stack([-2 * rho + 3 * q, rho - 3 * q, -jx, -jy, (jx * jx - jy * jy) / rho,
                        jx * jy / rho])


def _exact_lattice(case, seed):
    rng = random.Random(seed)
    rho, ux, uy = _fields(case, rng)
    src = _source(case, rng) if case["source"] else None
    M = torch.from_numpy(_moment_matrix()).cuda()
    Mi = torch.linalg.inv(M)
    e, eps, q, nu = RATES[case["rates"]]
    back = Mi[:, 3:] * torch.tensor([e, eps, q, q, nu, nu], dtype=torch.float64, device="cuda")

    def feq(r, jx, jy):
        m = torch.cat([torch.stack([r, jx, jy]), _meq(r, jx, jy)])
        return (Mi @ m.reshape(9, -1)).reshape(m.shape)

    f = feq(rho, rho * ux, rho * uy)
    for t in range(case["steps"]):
        if src is not None:
            r = torch.tensor([[1.0 + src[2] * math.sin(2 * math.pi * t / src[3])]],
                             dtype=torch.float64, device="cuda")
            f[:, src[1], src[0]] = feq(r, 0 * r, 0 * r).reshape(9)
        m = (M @ f.reshape(9, -1)).reshape(f.shape)
        d = m[3:] - _meq(m[0], m[1], m[2])
        f -= (back @ d.reshape(6, -1)).reshape(f.shape)
        del m, d
        for i in range(9):
            if C[i].any():
                f[i] = torch.roll(f[i], shifts=(int(C[i, 1]), int(C[i, 0])), dims=(0, 1))
    m = torch.stack([f.sum(0)] + [(f * torch.from_numpy(C[:, a].astype(float)).cuda()
                                   [:, None, None]).sum(0) for a in (0, 1)])
    return {"rho": m[0], "ux": m[1] / m[0], "uy": m[2] / m[0]}


def _exact_vn(case, seed):
    kx, ky, U, V, S = prepare(case, seed).args
    n = len(kx)
    M = _moment_matrix()
    Mi = np.linalg.inv(M)
    s = S[:, [0, 3, 5, 1, 2, 4, 6, 7, 8]]
    z, o = np.zeros(n), np.ones(n)
    u2 = U * U + V * V
    J = np.zeros((n, 9, 9))  # derivatives of the equilibrium moments at rho = 1, j = (U, V)
    for r, row in enumerate([(o, z, z), (z, o, z), (z, z, o), (-2 - 3 * u2, 6 * U, 6 * V),
                             (1 + 3 * u2, -6 * U, -6 * V), (z, -o, z), (z, z, -o),
                             (V * V - U * U, 2 * U, -2 * V), (-U * V, V, U)]):
        for c in range(3):
            J[:, r, c] = row[c]
    psi = np.eye(9)[None] - s[:, :, None] * (np.eye(9)[None] - J)
    psi[:, :3] = np.eye(9)[:3]
    G = np.exp(-1j * (kx[:, None] * C[:, 0] + ky[:, None] * C[:, 1]))[:, :, None] * (Mi @ psi @ M)
    lam = np.linalg.eigvals(G)
    return {"spectra": np.sort(np.stack([lam.real, lam.imag], axis=-1), axis=1)}


def exact(case, seed):
    """The outputs of run in 64-bit torch / numpy; None for the batches, and
    for runs of over about 10 s."""
    if case["kind"] == "vn":
        return _exact_vn(case, seed)
    if case["kind"] == "lattice" and case["nx"] * case["ny"] * case["steps"] <= 4.5e9:
        return _exact_lattice(case, seed)
    return None

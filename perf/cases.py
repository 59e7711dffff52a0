"""The work a user of this library has it do, as cases that can be timed and compared.

A case is a dict of plain values; ``prepare`` makes what a program holds before the
call (particles on the GPU, a context with them loaded, output buffers), ``run`` is
one pass through the public entry points of ``paper_0711_0643_gb300.nbody``, ``work``
the bytes and operations a pass cannot do without, and ``exact`` the same results
from plain torch arithmetic in 64 bits.

Kinds
-----
* ``force``: acceleration, jerk and potential of an active block against all
  particles (``nb_force_jerk_dev``), the call a host-side integrator makes per step;
* ``run``: load a system, integrate it, read the state back (``nb_init_dev``,
  ``nb_run``, ``nb_get_state``);
* ``ensemble``: the same for a batch of independent systems in one launch;
* ``energy``: the conservation check made at every output time (``nb_energy``);
* ``perturbers``: perturber lists of the binaries of a system (``nb_perturbers_dev``).

Particles are Plummer spheres in N-body units drawn on the GPU from the seed, with
equal masses or a Salpeter mass function; the library's default tuning table is used.
"""
import math

import numpy as np
import torch

from paper_0711_0643_gb300 import nbody as nb

MIXED, FP64 = "mixed", "fp64"
ETA, DT_MAX = 0.01, 1.0 / 16


def listed():
    return [
        # the smallest call: a few particles due in a small cluster, latency only
        {"name": "force_1k_s13", "kind": "force", "precision": MIXED, "n": 1000, "s": 13, "salpeter": False,
         "eps": 1.0 / 256},
        # a mean-sized block of the 65536-star model with a mass function
        {"name": "force_64k_s480", "kind": "force", "precision": MIXED, "n": 65536, "s": 480, "salpeter": True,
         "eps": 1.0 / 4096},
        # an ordinary block of a large cluster whose size is no multiple of anything
        {"name": "force_300k_s61", "kind": "force", "precision": MIXED, "n": 300007, "s": 61, "salpeter": False,
         "eps": 1e-3},
        # one particle due among a million: reading the particles is all there is to do
        {"name": "force_1m_s1", "kind": "force", "precision": MIXED, "n": 1048576, "s": 1, "salpeter": False,
         "eps": 1e-3},
        # a large block of the million-star model
        {"name": "force_1m_s1024", "kind": "force", "precision": MIXED, "n": 1048576, "s": 1024, "salpeter": False,
         "eps": 1e-3},
        # every particle: the initial forces of a run and its synchronised steps
        {"name": "force_128k_full", "kind": "force", "precision": MIXED, "n": 131072, "s": 131072, "salpeter": False,
         "eps": 1e-3},
        # the double-precision path, used to check the mixed one
        {"name": "force64_16k_s256", "kind": "force", "precision": FP64, "n": 16384, "s": 256, "salpeter": False,
         "eps": 1.0 / 1024},
        # a whole small integration, small blocks throughout
        {"name": "run_1k", "kind": "run", "precision": MIXED, "n": 1024, "t": 0.25, "salpeter": False,
         "eps": 1.0 / 256},
        # the first sixteenth of a time unit of the 16384-star integration
        {"name": "run_16k", "kind": "run", "precision": MIXED, "n": 16384, "t": 0.0625, "salpeter": False,
         "eps": 1.0 / 1024},
        # a batch of small clusters of different sizes
        {"name": "ensemble_40", "kind": "ensemble", "systems": 40, "n_lo": 256, "n_hi": 4096, "t": 0.0625},
        # the energy check at an output time
        {"name": "energy_32k", "kind": "energy", "n": 32768, "salpeter": False, "eps": 1.0 / 1024},
        # a tenth of the stars in primordial binaries, the customary threshold and list length
        {"name": "perturbers_16k", "kind": "perturbers", "n": 16384, "binaries": 1638, "gamma": 1e-7, "nmax": 256},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["force"] * 8 + ["force64"] * 2 + ["run"] * 3 + ["ensemble", "energy", "energy", "perturbers"])
    if kind == "force":
        n = _log_int(rng, 500, 1 << 20)
        return {"kind": "force", "precision": MIXED, "n": n, "s": _log_int(rng, 1, min(n, (1 << 34) // n)),
                "salpeter": rng.random() < 0.3, "eps": rng.choice([1e-3, 1.0 / 256, 1.0 / 4096])}
    if kind == "force64":
        n = _log_int(rng, 500, 1 << 16)
        return {"kind": "force", "precision": FP64, "n": n, "s": _log_int(rng, 1, min(n, (1 << 26) // n)),
                "salpeter": rng.random() < 0.3, "eps": 1e-3}
    if kind == "run":
        n = _log_int(rng, 200, 16384)
        return {"kind": "run", "precision": FP64 if n < 3000 and rng.random() < 0.3 else MIXED, "n": n, "t": 0.0625,
                "salpeter": rng.random() < 0.3, "eps": max(4.0 / n, 1.0 / 1024)}
    if kind == "ensemble":
        lo = _log_int(rng, 100, 600)
        return {"kind": "ensemble", "systems": rng.randint(3, 40), "n_lo": lo, "n_hi": _log_int(rng, lo + 1, 4096),
                "t": 0.0625}
    if kind == "energy":
        return {"kind": "energy", "n": _log_int(rng, 500, 32768), "salpeter": rng.random() < 0.3, "eps": 1.0 / 1024}
    n = _log_int(rng, 1000, 16384)
    return {"kind": "perturbers", "n": n, "binaries": _log_int(rng, 1, n // 10),
            "gamma": rng.choice([1e-7, 1e-6, 1e-5]), "nmax": rng.choice([64, 256, 256, 1000])}


# ------------------------------------------------------------------ particles

def _rng(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _uniform(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)


def _isotropic(g, r):
    z = 2.0 * _uniform(g, r.shape[0]) - 1.0
    phi = 2.0 * math.pi * _uniform(g, r.shape[0])
    rho = torch.sqrt(torch.clamp(1.0 - z * z, min=0.0))
    return r[:, None] * torch.stack([rho * torch.cos(phi), rho * torch.sin(phi), z], dim=1)


def _masses(g, n, salpeter):
    if not salpeter:
        return torch.full((n,), 1.0 / n, device="cuda", dtype=torch.float64)
    p = 1.0 - 2.35   # dN/dm ~ m^-2.35 on [0.1, 100]
    m = (0.1 ** p + _uniform(g, n) * (100.0 ** p - 0.1 ** p)) ** (1.0 / p)
    return m / m.sum()


def _plummer(g, n, salpeter=False):
    """m[n], x[n, 3], v[n, 3] of a Plummer sphere (Aarseth, Henon & Wielen 1974), E = -1/4."""
    m = _masses(g, n, salpeter)
    u = (_uniform(g, n) * 0.999).clamp(min=1e-9)
    r = 1.0 / torch.sqrt(u ** (-2.0 / 3.0) - 1.0)
    x = _isotropic(g, r)
    q = torch.full((n,), 0.3, device="cuda", dtype=torch.float64)
    todo = torch.ones(n, device="cuda", dtype=torch.bool)
    for _ in range(24):   # rejection from q^2 (1 - q^2)^(7/2)
        c, y = _uniform(g, n), 0.1 * _uniform(g, n)
        hit = todo & (y < c * c * (1.0 - c * c) ** 3.5)
        q = torch.where(hit, c, q)
        todo = todo & ~hit
    v = _isotropic(g, q * math.sqrt(2.0) * (1.0 + r * r) ** -0.25)
    x = x - (m[:, None] * x).sum(0)
    v = v - (m[:, None] * v).sum(0)
    scale = 3.0 * math.pi / 16.0
    return m, (x * scale).contiguous(), (v / math.sqrt(scale)).contiguous()


def _binaries(g, n, nb_):
    """A Plummer sphere of n - nb_ centres, nb_ of them split into pairs (i, n - nb_ + i)."""
    m, c, _ = _plummer(g, n - nb_)
    d = torch.exp(math.log(1e-4) + _uniform(g, nb_) * math.log(100.0))   # separations 1e-4 .. 1e-2
    half = 0.5 * _isotropic(g, d)
    x = torch.cat([c, c[:nb_] - half])
    x[:nb_] += half
    i = torch.arange(nb_, device="cuda", dtype=torch.int32)
    pairs = torch.stack([i, i + (n - nb_)], dim=1).contiguous()
    m = torch.full((n,), 1.0 / n, device="cuda", dtype=torch.float64)
    return m, x.contiguous(), torch.zeros_like(x), pairs


def _active(g, n, s):
    if s == n:
        return torch.arange(n, device="cuda", dtype=torch.int32)
    return torch.randperm(n, generator=g, device="cuda")[:s].sort().values.to(torch.int32)


def _systems(case, seed):
    """The ensemble's members, one after another: sizes log-uniform in [n_lo, n_hi], the largest and
    smallest among them, so that the work does not depend on the seed."""
    k, lo, hi = case["systems"], case["n_lo"], case["n_hi"]
    sizes = [max(2, int(round(lo * (hi / lo) ** (q / max(1, k - 1))))) for q in range(k)]
    g = _rng(seed)
    parts = [_plummer(g, n) for n in sizes]
    return sizes, parts, np.array([4.0 / n for n in sizes]) ** 2


# -------------------------------------------------------------------- a case

class _State:
    pass


_STREAMS = []


def _context(case):
    """A context on the program's one stream: an integrator's calls depend on one another."""
    if not _STREAMS:
        _STREAMS.append(torch.cuda.Stream())
    return nb.Context(precision=nb.NB_PREC_FP64 if case.get("precision") == FP64 else nb.NB_PREC_MIXED, eta=ETA,
                      dt_max=DT_MAX, stream=_STREAMS[0].cuda_stream)


def _load(st):
    nb.nb_init_dev(st.ctx.ctx, st.n, st.m.data_ptr(), st.x.data_ptr(), st.v.data_ptr(), st.eps2)


def prepare(case, seed):
    st = _State()
    st.kind = case["kind"]
    g = _rng(seed)
    if st.kind == "ensemble":
        sizes, parts, st.eps2 = _systems(case, seed)
        st.m, st.x, st.v = (torch.cat([p[c] for p in parts]).cpu().numpy() for c in range(3))
        st.off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
        st.t = case["t"]
        st.ctx = _context(case)
        return st
    st.n = case["n"]
    if st.kind == "perturbers":
        st.m, st.x, st.v, st.pairs = _binaries(g, st.n, case["binaries"])
        st.eps2 = 1e-6
        st.gamma, st.nmax = case["gamma"], case["nmax"]
        st.lists = torch.empty(case["binaries"], st.nmax, device="cuda", dtype=torch.int32)
        st.counts = torch.empty(case["binaries"], device="cuda", dtype=torch.int32)
    else:
        st.m, st.x, st.v = _plummer(g, st.n, case["salpeter"])
        st.eps2 = case["eps"] ** 2
    if st.kind == "force":
        st.s = case["s"]
        st.idx = _active(g, st.n, st.s)
        st.a = torch.empty(st.s, 3, device="cuda", dtype=torch.float64)
        st.k = torch.empty(st.s, 3, device="cuda", dtype=torch.float64)
        st.phi = torch.empty(st.s, device="cuda", dtype=torch.float64)
    if st.kind == "run":
        st.t = case["t"]
    st.ctx = _context(case)
    torch.cuda.synchronize()   # the particles were made on another stream
    if st.kind != "run":
        _load(st)
    return st


def run(st):
    c = st.ctx.ctx
    if st.kind == "force":
        nb.nb_force_jerk_dev(c, st.idx.data_ptr(), st.s, st.a.data_ptr(), st.k.data_ptr(), st.phi.data_ptr())
        return {"a": st.a, "k": st.k, "phi": st.phi}
    if st.kind == "run":
        _load(st)
        nb.nb_run(c, st.t)
        return nb.nb_get_state(c, st.n)
    if st.kind == "ensemble":
        nb.nb_ensemble_init(c, st.off, st.m, st.x, st.v, st.eps2)
        nb.nb_ensemble_run(c, st.t)
        return {"energy": nb.nb_ensemble_energy(c, len(st.eps2)), **nb.nb_ensemble_get_state(c, int(st.off[-1]))}
    if st.kind == "energy":
        return np.array(nb.nb_energy(c))   # E, K, W
    nb.nb_perturbers_dev(c, st.pairs.shape[0], st.pairs.data_ptr(), st.gamma, st.nmax, 0, -1, st.lists.data_ptr(),
                         st.counts.data_ptr())
    return {"lists": st.lists, "counts": st.counts}


# Block steps of a Plummer sphere per particle and time unit, eta = 0.01 (counted in runs of
# 1024 to 65536 particles: 277 to 483).
def _steps(n):
    return 30.0 * math.log2(n)


def _run_work(n, t):
    # the initial forces and every particle step against all particles; the state in and out
    return 60.0 * n * n * (1.0 + _steps(n) * t), n * (7 + 15) * 8.0


def work(case):
    """60 operations per softened force-and-jerk interaction, the usual count."""
    if case["kind"] == "force":
        n, s = case["n"], case["s"]
        rec = 40.0 if case["precision"] == MIXED else 56.0   # a predicted particle
        return {"bytes": n * rec + s * (4 + 7 * 8.0), "flops": 60.0 * n * s}
    if case["kind"] == "run":
        f, b = _run_work(case["n"], case["t"])
        return {"bytes": b, "flops": f}
    if case["kind"] == "ensemble":
        k, lo, hi = case["systems"], case["n_lo"], case["n_hi"]
        w = [_run_work(lo * (hi / lo) ** (q / max(1, k - 1)), case["t"]) for q in range(k)]
        return {"bytes": sum(b for _, b in w), "flops": sum(f for f, _ in w)}
    n = case["n"]
    if case["kind"] == "energy":   # each pair once: 3 differences, 6 for r^2, the root, the product, the sum
        return {"bytes": n * 56.0, "flops": 12.0 * n * (n - 1) / 2}
    nbin = case["binaries"]
    return {"bytes": n * 32.0 + nbin * (8.0 + 4.0 * case["nmax"] + 4.0), "flops": 14.0 * n * nbin}


# ------------------------------------------------------------- in 64 bits

def _forces(m, x, v, eps2, idx, rows=1 << 25):
    """a, k, phi of particles idx, by direct summation in chunks of about `rows` pairs."""
    n, outs = x.shape[0], []
    cols = [x[:, 0].contiguous(), x[:, 1].contiguous(), x[:, 2].contiguous(), v[:, 0].contiguous(),
            v[:, 1].contiguous(), v[:, 2].contiguous()]
    for ids in idx.long().split(max(1, rows // n)):
        d = [c[None, :] - c[ids][:, None] for c in cols]
        r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2] + eps2
        q = torch.rsqrt(r2)
        q[torch.arange(ids.shape[0], device=x.device), ids] = 0.0
        q2 = q * q
        mq = m[None, :] * q
        mu = mq * q2
        al = 3.0 * (d[0] * d[3] + d[1] * d[4] + d[2] * d[5]) * q2
        a = [(mu * d[c]).sum(1) for c in range(3)]
        k = [(mu * (d[3 + c] - al * d[c])).sum(1) for c in range(3)]
        outs.append(torch.stack(a + k + [-mq.sum(1)], dim=1))
    o = torch.cat(outs)
    return o[:, 0:3].contiguous(), o[:, 3:6].contiguous(), o[:, 6].contiguous()


def _norm(u):
    return torch.sqrt((u * u).sum(1))


def _pow2(c, dt_max):
    c = torch.where(torch.isfinite(c), c, torch.full_like(c, dt_max))
    e = torch.frexp(c).exponent - 1
    return torch.clamp(torch.ldexp(torch.ones_like(c), e), max=dt_max)


def _integrate(m, x, v, eps2, t_end):
    """Block-step Hermite integration to t_end; None where it would take long."""
    n = x.shape[0]
    x, v = x.clone(), v.clone()
    a, k, _ = _forces(m, x, v, eps2, torch.arange(n, device=x.device))
    t = torch.zeros(n, device=x.device, dtype=torch.float64)
    dt = _pow2(ETA * _norm(a) / _norm(k), DT_MAX)
    while True:
        key = t + dt
        tn = float(key.min())
        if tn > t_end:
            return x, v, a, k
        i = (key == tn).nonzero()[:, 0]
        d = (tn - t)[:, None]
        xp = x + v * d + a * d * d * 0.5 + k * d * d * d / 6.0
        vp = v + a * d + k * d * d * 0.5
        an, kn, _ = _forces(m, xp, vp, eps2, i)
        h = dt[i][:, None]
        a0, k0 = a[i], k[i]
        a2 = -6.0 * (a0 - an) / h ** 2 - (4.0 * k0 + 2.0 * kn) / h
        a3 = 12.0 * (a0 - an) / h ** 3 + 6.0 * (k0 + kn) / h ** 2
        x[i] = xp[i] + a2 * h ** 4 / 24.0 + a3 * h ** 5 / 120.0
        v[i] = vp[i] + a2 * h ** 3 / 6.0 + a3 * h ** 4 / 24.0
        a2p = a2 + a3 * h
        a[i], k[i], t[i] = an, kn, tn
        cand = torch.sqrt(ETA * (_norm(an) * _norm(a2p) + (kn * kn).sum(1)) /
                          (_norm(kn) * _norm(a3) + (a2p * a2p).sum(1)))
        q, h = _pow2(cand, DT_MAX), dt[i]
        twice = (q >= 2.0 * h) & (2.0 * h <= DT_MAX) & (torch.remainder(torch.full_like(h, tn), 2.0 * h) == 0.0)
        dt[i] = torch.where(q < h, q, torch.where(twice, 2.0 * h, h))


def _energy64(m, x, v, eps2):
    n, w = x.shape[0], 0.0
    for ids in torch.arange(n, device=x.device).split(max(1, (1 << 25) // n)):
        d = x[None, :, :] - x[ids][:, None, :]
        q = torch.rsqrt((d * d).sum(2) + eps2)
        q[torch.arange(ids.shape[0], device=x.device), ids] = 0.0
        w = w - 0.5 * (m[ids] * (q * m[None, :]).sum(1)).sum()
    k = 0.5 * (m * (v * v).sum(1)).sum()
    return float(k + w), float(k), float(w)


def exact(case, seed):
    if case["kind"] == "perturbers":   # whole numbers
        return None
    if case["kind"] == "ensemble":     # thousands of block steps, one by one
        return None
    g = _rng(seed)
    m, x, v = _plummer(g, case["n"], case["salpeter"])
    if case["kind"] == "energy":
        return np.array(_energy64(m, x, v, case["eps"] ** 2))
    if case["kind"] == "force":
        a, k, phi = _forces(m, x, v, case["eps"] ** 2, _active(g, case["n"], case["s"]))
        return {"a": a, "k": k, "phi": phi}
    # the steps themselves are left out: a rounding error decides between two powers of two
    x, v, a, k = _integrate(m, x, v, case["eps"] ** 2, case["t"])
    return {"m": m, "x": x, "v": v, "a": a, "k": k, "t": None, "dt": None}

"""The work whose speed this repository watches: output intervals of single runs, gradients
and ensembles, each through the calls of the package's public interface.

An output interval is what a run repeats from its start to its end: the wall diagnostics of
the current state and the leapfrog steps to the next output (every 10 steps in 2D, every 20
in 3D).  A pass restores a checkpoint that the program keeps on the device and advances it by
one interval, so that every pass does the same work on the same network of walls.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1710_10420_gb300 as prs

# the lattice and the physics of every run here: dx = 1, unit vacuum, walls ten sites wide
DETA, ETA0, W0, PHI0, ALPHA = 0.1, 1.0, 10.0, 1.0, 3.0
EPS = 0.1  # smoothing width of the differentiable wall area


def _interval(name, nx, ny, nz, steps, precision="fp32", repro=False, era_m=1.0, n0=150):
    return dict(name=name, kind="interval", nx=nx, ny=ny, nz=nz, steps=steps, precision=precision, repro=repro,
                era_m=era_m, n0=n0)


def listed():
    return [
        # the smallest run: 128^2 in the bit-reproducible FP64 mode that is checked against a
        # sequential evaluation; a handful of launches on a lattice of 16384 sites
        _interval("interval_2d_128_fp64_repro", 128, 128, 0, 10, "fp64", True),
        # one member of a scan over parameters, run by itself
        _interval("interval_2d_256_fp32", 256, 256, 0, 10),
        # the 2D box of the paper's scaling exponents, in both its precisions
        _interval("interval_2d_2048_fp32", 2048, 2048, 0, 10),
        _interval("interval_2d_2048_fp64", 2048, 2048, 0, 10, "fp64"),
        # the large 2D box, matter era
        _interval("interval_2d_4096_fp32", 4096, 4096, 0, 10, era_m=2.0),
        # a 2D box whose sides are nobody's power of two
        _interval("interval_2d_ragged_fp32", 2500, 1701, 0, 10),
        # the 3D box of the paper's scaling exponents
        _interval("interval_3d_128_fp32", 128, 128, 128, 20),
        # a 3D run in double precision
        _interval("interval_3d_256_fp64", 256, 256, 256, 20, "fp64"),
        # a 3D box cut to the size a study asks for
        _interval("interval_3d_ragged_fp32", 450, 421, 380, 20),
        # the largest run: the box of the throughput benchmark
        _interval("interval_3d_1024_fp32", 1024, 1024, 1024, 20),
        # the gradient of the wall area after 64 steps with respect to the state at their start
        # and to alpha, states recomputed from checkpoints
        dict(name="gradient_3d_256_fp32", kind="gradient", nx=256, ny=256, nz=256, steps=64, ckpt=16, n0=0,
             precision="fp32"),
        # an ensemble of uneven small boxes from white noise to its last output, its diagnostic
        # series and its final states
        dict(name="ensemble_mixed_fp32", kind="ensemble", runs2d_256=16, runs2d_512=4, runs3d_128=4, steps=800,
             every=20),
    ]


def _size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["interval"] * 6 + ["gradient", "ensemble"])
    if kind == "ensemble":
        return dict(kind="ensemble", runs2d_256=rng.randint(1, 24), runs2d_512=rng.randint(0, 6),
                    runs3d_128=rng.randint(0, 6), steps=rng.randint(200, 800), every=rng.choice([10, 20, 25]))
    if kind == "gradient":
        nx, ny, nz = (rng.choice([128, 256]), 8 * rng.randint(8, 32), rng.randint(48, 256))
        return dict(kind="gradient", nx=nx, ny=ny, nz=nz, steps=rng.randint(16, 64), ckpt=rng.choice([0, 8, 16, 32]),
                    n0=rng.choice([0, 100]), precision="fp32")
    precision = rng.choice(["fp32", "fp32", "fp64"])
    two_d = rng.random() < 0.5
    if two_d:
        side, steps = _size(rng, 96, 4096 if precision == "fp32" else 2048), rng.choice([10, 10, 7])
    else:
        side, steps = _size(rng, 48, 512 if precision == "fp32" else 256), rng.choice([20, 20, 13])
    stretch = rng.uniform(0.7, 1.4)
    nx, ny = int(side * stretch), int(side / stretch)
    nz = 0 if two_d else side
    if rng.random() < 0.4:  # rows as wide as a power of two, the other sides multiples of 32
        nx = min(4096 if two_d else 512, 1 << max(7, int(math.log2(nx))))
        ny, nz = max(32, ny // 32 * 32), 0 if two_d else max(32, nz // 32 * 32)
    return dict(kind="interval", nx=nx, ny=ny, nz=nz, steps=steps, precision=precision,
                repro=precision == "fp64" and rng.random() < 0.3, era_m=rng.choice([1.0, 2.0]),
                n0=rng.choice([100, 150, 300]))


# ------------------------------------------------------------------ inputs

def _shape(case):
    return (case["nx"], case["ny"]) + ((case["nz"],) if case["nz"] else ())


def _smooth(shape, length, gen, dtype):
    """A Gaussian random field of unit variance, correlated over `length` sites (array order)."""
    noise = torch.randn(shape, generator=gen, device="cuda", dtype=dtype)
    spec = torch.fft.rfftn(noise)
    del noise
    for axis, n in enumerate(shape):
        k = torch.fft.rfftfreq(n, device="cuda", dtype=dtype) if axis == len(shape) - 1 else \
            torch.fft.fftfreq(n, device="cuda", dtype=dtype)
        filt = torch.exp(-0.5 * (2.0 * math.pi * length * k) ** 2)
        spec *= filt.reshape([-1 if a == axis else 1 for a in range(len(shape))])
    field = torch.fft.irfftn(spec, s=shape)
    del spec
    return field.div_(field.std())


def _network(case, seed):
    """A formed network: domains of both vacua, tanh walls W0 wide between them, moving with
    about half the speed of light, and a little radiation in the domains; 0.05 to 0.08 sign
    changes per site, as runs have from eta = 7 to 50."""
    shape = tuple(reversed(_shape(case)))
    dtype = torch.float64 if case["precision"] == "fp64" else torch.float32
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    length = 10.0
    phi = _smooth(shape, length, gen, dtype)
    slope = length / math.sqrt(0.5 * len(shape))  # signed distance to the wall per unit of the field
    phi.mul_(math.pi / W0 * slope).tanh_()
    v = _smooth(shape, length, gen, dtype)
    v.mul_(0.5 * math.pi / W0).mul_(1.0 - phi * phi)
    ripple = _smooth(shape, 3.0, gen, dtype)
    phi.add_(ripple, alpha=0.03)
    v.add_(ripple.roll(1, 0), alpha=0.02)
    return phi.contiguous(), v.contiguous()


def _noise_runs(case, seed):
    """Per class of the ensemble: (shape, era exponents, white noise in (-1, 1) on the host)."""
    rng = np.random.Generator(np.random.PCG64(int(seed)))
    out = []
    for shape, count in (((256, 256), case["runs2d_256"]), ((512, 512), case["runs2d_512"]),
                         ((128, 64, 64), case["runs3d_128"])):
        if count:
            eras = [float(e) for e in rng.integers(1, 3, size=count)]
            phi = (rng.random((count,) + tuple(reversed(shape)), dtype=np.float32) * 2.0 - 1.0).astype(np.float32)
            out.append((shape, eras, phi))
    return out


# ------------------------------------------------------------------- passes

def prepare(case, seed):
    if case["kind"] == "ensemble":
        classes = _noise_runs(case, seed)
        runs = [prs.make_params(shape, era_m=era) for shape, eras, _ in classes for era in eras]
        zero = [np.zeros(phi.shape[1:], dtype=np.float32) for _, _, phi in classes]
        final = [(np.empty_like(phi), np.empty_like(phi)) for _, _, phi in classes]
        return dict(case=case, classes=classes, zero=zero, final=final, batch=_Batch(runs),
                    steps=[case["steps"]] * len(runs))
    phi, v = _network(case, seed)
    fp64 = case["precision"] == "fp64"
    sim = prs.Sim(_shape(case), precision=prs.PRS_FP64 if fp64 else prs.PRS_FP32, era_m=case.get("era_m", 1.0),
                  flags=prs.PRS_REPRO if case.get("repro") else 0)
    state = dict(case=case, sim=sim, phi=phi, v=v)
    if case["kind"] == "gradient":
        state["gphi"], state["gv"] = torch.empty_like(phi), torch.empty_like(v)
    return state


class _Batch:
    """An ensemble handle that is released with the object."""

    def __init__(self, runs):
        self.handle = prs.prs_batch_create(runs)
        try:  # a call of no steps: the first call on a new handle may report, once, an error left in its memory
            prs.prs_batch_run(self.handle, [0] * len(runs))
        except prs.PRSError:
            pass

    def __del__(self):
        prs.prs_batch_destroy(self.handle)


def _sums(values, fp64):
    """A run's diagnostics carry the precision of its fields."""
    return torch.tensor(values, dtype=torch.float64 if fp64 else torch.float32)


def run(state):
    case = state["case"]
    if case["kind"] == "ensemble":
        return _run_ensemble(state)
    sim = state["sim"]
    prs.prs_set_state_device(sim.handle, state["phi"], state["v"], case["n0"])
    fp64 = case["precision"] == "fp64"
    if case["kind"] == "gradient":
        J, dalpha = prs.prs_adjoint(sim.handle, case["steps"], prs.PRS_OBS_SMOOTH_AREA, EPS, case["ckpt"],
                                    state["gphi"], state["gv"])
        return dict(J=_sums([J, dalpha], fp64), gphi=state["gphi"], gv=state["gv"])
    d = prs.prs_step_measure(sim.handle, case["steps"])
    phi, v, n = sim.tensors()
    return dict(phi=phi, v=v, diagnostics=_sums([d.area_per_volume, d.gamma_v], fp64),
                counts=[d.n_links, d.n_wall, d.n_vzero, d.n_nonfinite, d.step, n])


def _run_ensemble(state):
    case, batch = state["case"], state["batch"].handle
    r = 0
    for (_, _, phi), zero in zip(state["classes"], state["zero"]):
        for k in range(len(phi)):
            prs.prs_batch_set_state(batch, r, phi[k], zero, 0)
            r += 1
    series = prs.prs_batch_run(batch, state["steps"], case["every"], case["steps"] // case["every"] + 1)
    r = 0
    for phi, v in state["final"]:
        for k in range(len(phi)):
            prs.prs_batch_get_state(batch, r, phi[k], v[k])
            r += 1
    return dict(series=series.astype(np.float32), phi=[f[0] for f in state["final"]],
                v=[f[1] for f in state["final"]])


# --------------------------------------------------------------------- work

def work(case):
    """Fields in once and out once; 2D + 9 operations a site and step (2D - 1 additions for the
    neighbours, one product and one fused multiply-add for the potential, one product, and three
    fused multiply-adds for kick and drift, each counted as two)."""
    if case["kind"] == "ensemble":
        s2 = 256 * 256 * case["runs2d_256"] + 512 * 512 * case["runs2d_512"]
        s3 = 128 * 64 * 64 * case["runs3d_128"]
        return dict(bytes=16.0 * (s2 + s3), flops=case["steps"] * (13.0 * s2 + 15.0 * s3))
    sites = 1
    for n in _shape(case):
        sites *= n
    ops = 2 * len(_shape(case)) + 9
    if case["kind"] == "gradient":  # the state in, its gradient out; a forward step and its transpose
        return dict(bytes=16.0 * sites, flops=2.0 * case["steps"] * ops * sites)
    size = 8 if case["precision"] == "fp64" else 4
    return dict(bytes=4.0 * size * sites, flops=float(case["steps"]) * ops * sites)


# ------------------------------------------------- the same in 64 bits, plainly

def _steps64(phi, v, dims, n, steps, era_m, alpha=ALPHA):
    """`steps` leapfrog steps from step n over the last `dims` axes; era_m: a number or a
    tensor that broadcasts over the fields.  Without a gradient the fields are updated in place."""
    V0 = math.pi ** 2 / (2.0 * W0 * W0)
    cV = 4.0 * V0 / PHI0 ** 2
    grad = torch.is_grad_enabled()
    for k in range(steps):
        delta = 0.5 * alpha * DETA * era_m / (ETA0 + (n + k) * DETA)
        c1, c2 = (1.0 - delta) / (1.0 + delta), DETA / (1.0 + delta)
        acc = phi * (-2.0 * dims)
        for axis in range(1, dims + 1):
            for shift in (1, -1):
                acc = acc + phi.roll(shift, -axis) if grad else acc.add_(phi.roll(shift, -axis))
        if grad:
            v = c1 * v + c2 * (acc - cV * phi * (phi * phi / PHI0 ** 2 - 1.0))
            phi = phi + DETA * v
        else:
            force = phi * phi
            force.div_(PHI0 ** 2).sub_(1.0).mul_(phi).mul_(cV)
            acc.sub_(force).mul_(c2)
            del force
            v.mul_(c1).add_(acc)
            phi.add_(v, alpha=DETA)
        del acc
    return phi, v


def _diagnostics64(phi, v):
    """(A/V, gamma v, links, wall sites, wall sites without a potential) of one field."""
    dims, shape = phi.dim(), phi.shape
    strides = [math.prod(shape[a + 1:]) for a in range(dims)]
    flat = phi.reshape(-1)
    neg = phi < 0
    wall = torch.zeros_like(neg)
    sum_w, links = 0.0, 0

    def moved(idx, axis, by):
        at = idx // strides[axis] % shape[axis]
        return idx + ((at + by) % shape[axis] - at) * strides[axis]

    for d in range(dims):
        cross = neg ^ neg.roll(-1, d)
        wall |= cross
        wall |= cross.roll(1, d)
        s = cross.reshape(-1).nonzero().reshape(-1)
        del cross
        links += s.numel()
        t = moved(s, d, 1)
        g = flat[t] - flat[s]
        num, den = g * g, g.abs()
        for e in range(dims):
            if e != d:
                g = 0.25 * ((flat[moved(s, e, 1)] - flat[moved(s, e, -1)]) +
                            (flat[moved(t, e, 1)] - flat[moved(t, e, -1)]))
                num, den = num + g * g, den + g.abs()
        sum_w += float((num.sqrt() / den).sum())
    at = wall.reshape(-1).nonzero().reshape(-1)
    pot = math.pi ** 2 / (2.0 * W0 * W0) * (flat[at] ** 2 / PHI0 ** 2 - 1.0) ** 2
    kin = v.reshape(-1)[at] ** 2
    has = pot > 0
    count = int(has.sum())
    gamma = math.sqrt(float((kin[has] / pot[has]).sum()) / (2.0 * count)) if count else 0.0
    return sum_w / flat.numel(), gamma, links, at.numel(), at.numel() - count


def _area64(phi):
    t = torch.tanh(phi / EPS)
    J = 0.0
    for axis in range(phi.dim()):
        J = J + (0.5 * (1.0 - t * t.roll(-1, axis))).sum()
    return J / phi.numel()


def exact(case, seed):
    if case["kind"] == "ensemble":
        return _exact_ensemble(case, seed)
    phi, v = (x.double() for x in _network(case, seed))
    dims, n0, steps, era = phi.dim(), case["n0"], case["steps"], case.get("era_m", 1.0)
    if case["kind"] == "gradient":
        if phi.numel() * steps > 1.1e9:  # states of every step have to fit
            return None
        alpha = torch.tensor(ALPHA, dtype=torch.float64, device="cuda", requires_grad=True)
        phi.requires_grad_(True)
        v.requires_grad_(True)
        last, _ = _steps64(phi, v, dims, n0, steps, era, alpha)
        J = _area64(last)
        J.backward()
        return dict(J=torch.tensor([J.item(), alpha.grad.item()], dtype=torch.float64), gphi=phi.grad, gv=v.grad)
    with torch.no_grad():
        area, gamma, links, walls, empty = _diagnostics64(phi, v)
        phi, v = _steps64(phi, v, dims, n0, steps, era)
    return dict(phi=phi, v=v, diagnostics=torch.tensor([area, gamma], dtype=torch.float64),
                counts=[links, walls, empty, 0, n0, n0 + steps])


def _exact_ensemble(case, seed):
    classes = _noise_runs(case, seed)
    outputs = case["steps"] // case["every"] + 1
    series = np.zeros((sum(len(eras) for _, eras, _ in classes), outputs, 4))
    phis, vs, first = [], [], 0
    with torch.no_grad():
        for shape, eras, noise in classes:
            dims = len(shape)
            phi = torch.from_numpy(noise).cuda().double()
            v = torch.zeros_like(phi)
            era = torch.tensor(eras, dtype=torch.float64, device="cuda").reshape([-1] + [1] * dims)
            n = 0
            for k in range(outputs):
                for r in range(len(eras)):
                    area, gamma, links, _, _ = _diagnostics64(phi[r], v[r])
                    series[first + r, k] = (n, area, gamma, links)
                more = min(case["every"], case["steps"] - n)
                phi, v = _steps64(phi, v, dims, n, more, era)
                n += more
            phis.append(phi)
            vs.append(v)
            first += len(eras)
    return dict(series=series, phi=phis, v=vs)

"""Performance cases of the data-consistency library: the calls a reconstruction program makes, over their range.

A case is a dict of plain values.  "op" names what one pass does, the other fields are the problem:

    step      one data-consistency step and its vector-Jacobian product (Eq. 3), plain calls
    forward   the step alone                     vjp   the vector-Jacobian product alone
    unrolled  a network's iterations on one example with the measurements kept: "form" aty (A^H y, then steps
              in normal-equations form: inference) or prepared (tables of y, then steps, then as many VJPs
              backwards: training)
    modl      the MoDL model inversion (10 conjugate-gradient steps) and its VJP
    train     one greedy module without its network: step on two-channel tensors under autograd, l1 loss,
              backward, and the gradient of a trained step size

The inputs are smooth sensitivities with sum |S|^2 = 1, ellipse phantoms, the sampling patterns of the data sets
the paper uses (random, equispaced and k-t lines, Poisson-disc planes) and measurements y = M (F S x + noise).
"""
import math

import numpy as np
import torch

import paper_2207_08393_b200 as g

# transform lengths of the library that occur in practice (smaller ones exist for tests)
LENGTHS_2D = [24, 32, 40, 46, 48, 64, 80, 92, 96, 120, 128, 160, 184, 192, 240, 256, 320, 368, 384, 512, 640]
LENGTHS_3D = [24, 32, 40, 48, 64, 80, 92, 96, 120, 128, 160, 184, 192, 240, 256, 320, 368]

DEFAULTS = {"batch": 1, "coils": 8, "frames": 1, "n0": 1, "moving_coils": False, "full_mask": False, "mask": "lines",
            "accel": 4.0, "center": 8, "eta": 1.0}


def _case(name, op, **kw):
    return dict(DEFAULTS, name=name, op=op, **kw)


def listed():
    return [
        # one small slice: the launches and the calls themselves are what it costs
        _case("slice64", "step", n1=64, n2=64),
        # short ragged series (sizes 8 x 15 and 4 x 23, odd counts) whose sensitivities move with the frames
        _case("ragged_frames", "step", batch=3, coils=5, frames=3, n1=120, n2=92, moving_coils=True, center=6),
        # multi-coil knee slices, a training batch
        _case("knee2d", "step", batch=4, coils=15, n1=640, n2=368, mask="equispaced", accel=8.0, center=15, eta=0.5),
        # multi-coil brain slices through a trained 10-iteration network
        _case("brain2d_unrolled", "unrolled", form="aty", iterations=10, batch=8, coils=16, n1=640, n2=320, center=26),
        # dynamic cardiac series, 8 iterations forward and backward
        _case("cine_unrolled", "unrolled", form="prepared", iterations=8, frames=20, n1=192, n2=160, mask="kt", accel=10.0, center=6),
        # the same series in the MoDL network's model inversion
        _case("cine_modl", "modl", frames=20, n1=192, n2=160, mask="kt", accel=10.0, center=6),
        # knee volume with a ky-kz Poisson-disc mask, each direction; the largest problems
        _case("knee3d_forward", "forward", n0=320, n1=320, n2=256, mask="poisson", accel=12.0, center=24),
        _case("knee3d_vjp", "vjp", n0=320, n1=320, n2=256, mask="poisson", accel=12.0, center=24),
        # a smaller volume, many coils: zero-filled image and two iterations
        _case("volume_unrolled", "unrolled", form="aty", iterations=2, coils=12, n0=96, n1=240, n2=184, mask="poisson", accel=8.0, center=16),
        # slices of a volume under that volume's Poisson-disc mask: every k-space sample has its own weight
        _case("slices_poisson", "step", batch=8, n1=320, n2=256, full_mask=True, mask="poisson", accel=6.0, center=24),
        # a volume with an arbitrary mask
        _case("volume_arbitrary", "step", coils=6, n0=96, n1=160, n2=128, full_mask=True, mask="poisson", accel=8.0, center=16),
        # training step of one module on brain-like slices with a trained step size
        _case("train_module", "train", batch=2, coils=12, n1=384, n2=320, center=26),
    ]


def _volume(c):
    return c["n0"] * c["n1"] * c["n2"]


def _units(c):
    return c["batch"] * c["coils"] * c["frames"] * _volume(c)


def draw(rng):
    op = rng.choice(["step", "step", "unrolled", "unrolled", "modl", "forward", "vjp", "full", "train"])
    most = {"step": 4e7, "unrolled": 2e7, "modl": 1e7, "forward": 2e8, "vjp": 2e8, "full": 3e7, "train": 2e7}[op]
    least = 1e6 if op in ("forward", "vjp") else 3e4
    while True:
        c = dict(DEFAULTS, op=op, coils=rng.randint(2, 16), eta=round(rng.uniform(0.3, 1.0), 2))
        volume = op in ("forward", "vjp") or (op in ("unrolled", "full") and rng.random() < 0.4)
        if volume:
            c.update(n0=rng.choice(LENGTHS_3D), n1=rng.choice(LENGTHS_3D), n2=rng.choice(LENGTHS_3D), mask="poisson")
        else:
            c.update(n1=rng.choice(LENGTHS_2D), n2=rng.choice(LENGTHS_2D), mask=rng.choice(["lines", "equispaced", "kt"]),
                     batch=rng.randint(1, 8), frames=rng.choice([1, 1, rng.randint(2, 24)]))
            c["moving_coils"] = c["frames"] > 1 and rng.random() < 0.3
        if op == "full":
            c.update(op="step", full_mask=True, mask="poisson")
        if op == "unrolled":
            c.update(form=rng.choice(["aty", "prepared"]), iterations=rng.randint(2, 10))
        c["accel"] = round(math.exp(rng.uniform(math.log(3.0), math.log(12.0))), 1)
        c["center"] = max(2, int(min(c["n1"], c["n2"]) * rng.uniform(0.03, 0.1)))
        # the work asked for is spread over its logarithm; take the first problem within a factor of two of it
        want = math.exp(rng.uniform(math.log(least), math.log(most)))
        if want / 2 <= _units(c) * c.get("iterations", 1) / (5 if "iterations" in c else 1) <= min(2 * want, most):
            return c


# ---------------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------------
def _axes(c, dev):
    return [torch.linspace(-1, 1, m + 1, device=dev)[:-1] if m > 1 else torch.zeros(1, device=dev) for m in (c["n0"], c["n1"], c["n2"])]


def _sens(c, rs, dev):
    """Gaussian magnitudes around the object times quadratic phases, root sum of squares 1."""
    u0, u1, u2 = _axes(c, dev)
    u0, u1, u2 = u0[:, None, None], u1[None, :, None], u2[None, None, :]
    T = c["frames"] if c["moving_coils"] else 1
    out = torch.empty((c["batch"], c["coils"], T, c["n0"], c["n1"], c["n2"]), dtype=torch.complex64, device=dev)
    for b in range(c["batch"]):
        for k in range(c["coils"]):
            sig, p = rs.uniform(0.6, 0.9), rs.uniform(-math.pi, math.pi, 8)
            for t in range(T):
                ang = 2 * math.pi * k / c["coils"] + 0.05 * t
                d = (u1 - 1.1 * math.cos(ang)) ** 2 + (u2 - 1.1 * math.sin(ang)) ** 2
                ph = p[0] + p[1] * u1 + p[2] * u2 + p[3] * u1 * u2 + p[4] * u1 ** 2 + p[5] * u2 ** 2
                if c["n0"] > 1:
                    d = d + (u0 - (0.5 if k % 2 else -0.5)) ** 2
                    ph = ph + p[6] * u0 + p[7] * u0 ** 2
                out[b, k, t] = torch.polar(torch.exp(-d / (2 * sig ** 2)), ph)
        out[b] /= torch.linalg.vector_norm(out[b], dim=0, keepdim=True)
    return out if c["moving_coils"] else out[:, :, 0].contiguous()


def _noise(shape, gen, dev, sigma):
    return torch.randn(shape, dtype=torch.complex64, device=dev, generator=gen) * sigma


def _phantom(c, rs, gen, dev):
    """Ellipses with complex amplitudes, pulsing over the frames, and texture."""
    u0, u1, u2 = _axes(c, dev)
    u0, u1, u2 = u0[:, None, None], u1[None, :, None], u2[None, None, :]
    x = _noise((c["batch"], c["frames"], c["n0"], c["n1"], c["n2"]), gen, dev, 0.05)
    for b in range(c["batch"]):
        for _ in range(12):
            p, r = rs.uniform(-0.6, 0.6, 3), rs.uniform(0.05, 0.4, 3)
            amp = complex(rs.uniform(0.1, 1) * np.exp(1j * rs.uniform(-math.pi, math.pi)))
            q = ((u1 - p[1]) / r[1]) ** 2 + ((u2 - p[2]) / r[2]) ** 2
            if c["n0"] > 1:
                q = q + ((u0 - p[0]) / r[0]) ** 2
            for t in range(c["frames"]):
                x[b, t] += amp * (q <= (1 + 0.15 * math.sin(2 * math.pi * t / c["frames"])) ** 2)
    return x


def _lines(c, n, rs):
    """1-D phase-encode pattern: fully sampled centre and random, equispaced or centre-weighted lines."""
    m = np.zeros(n, np.float32)
    lo = n // 2 - c["center"] // 2
    m[lo:lo + c["center"]] = 1
    if c["mask"] == "equispaced":
        m[rs.randint(int(c["accel"]))::int(c["accel"])] = 1
        return m
    rest = np.flatnonzero(m == 0)
    w = np.ones(rest.size) if c["mask"] == "lines" else (1 - np.abs(rest - n // 2) / (n / 2 + 1)) ** 2
    extra = min(rest.size, max(0, round(n / c["accel"]) - c["center"]))
    m[rs.choice(rest, extra, replace=False, p=w / w.sum())] = 1
    return m


def _plane(c, na, nb, rs):
    """2-D pattern: one sample in a random place of every cell (Poisson-disc-like), fully sampled centre."""
    ca = max(1, round(math.sqrt(c["accel"])))
    cb = max(1.0, c["accel"] / ca)
    ia, ib = np.meshgrid(np.arange(math.ceil(na / ca)), np.arange(math.ceil(nb / cb)), indexing="ij")
    a = (ia * ca + rs.uniform(0, ca, ia.shape)).astype(int)
    b = (ib * cb + rs.uniform(0, cb, ib.shape)).astype(int)
    ok = (a < na) & (b < nb)
    m = np.zeros((na, nb), np.float32)
    m[a[ok], b[ok]] = 1
    k = min(c["center"], na, nb)
    m[na // 2 - k // 2:na // 2 - k // 2 + k, nb // 2 - k // 2:nb // 2 - k // 2 + k] = 1
    return m


def _mask(c, rs, dev):
    """(mask as the library takes it, the same broadcast against y)."""
    B, T, n0, n1, n2 = c["batch"], c["frames"], c["n0"], c["n1"], c["n2"]
    bt = [(b, t) for b in range(B) for t in range(T)]
    if c["full_mask"]:
        # slices: each has the pattern of its own place; volumes: the pattern changes along the readout
        m = np.stack([np.stack([_plane(c, n1, n2, rs) for _ in range(n0)]) for _ in bt])
        m = torch.from_numpy(m.reshape(B, T, n0, n1, n2)).to(dev)
        return m, m[:, None]
    if n0 > 1:
        m = torch.from_numpy(np.stack([_plane(c, n1, n2, rs) for _ in bt]).reshape(B, T, n1, n2)).to(dev)
        return m, m[:, None, :, None]
    m = torch.from_numpy(np.stack([_lines(c, n2, rs) for _ in bt]).reshape(B, T, n2)).to(dev)
    return m, m[:, None, :, None, None, :]


def _measure(c, x, sens, mask, gen, dev):
    """y = M (F S x + noise), zero where nothing was sampled; one coil at a time."""
    axes = (-3, -2, -1) if c["n0"] > 1 else (-2, -1)
    y = torch.empty((c["batch"], c["coils"]) + tuple(x.shape[1:]), dtype=torch.complex64, device=dev)
    for k in range(c["coils"]):
        s = sens[:, k] if c["moving_coils"] else sens[:, k][:, None]
        f = torch.fft.fftshift(torch.fft.fftn(torch.fft.ifftshift(s * x, dim=axes), dim=axes, norm="ortho"), dim=axes)
        y[:, k] = mask[:, 0] * (f + _noise(f.shape, gen, dev, 0.01))
    return y


def prepare(case, seed):
    c = dict(DEFAULTS, **case)
    dev = torch.device("cuda")
    rs = np.random.RandomState(seed % (1 << 31))
    gen = torch.Generator(device=dev).manual_seed(seed)
    sens = _sens(c, rs, dev)
    x_true = _phantom(c, rs, gen, dev)
    mask, mask_y = _mask(c, rs, dev)
    st = {"c": c, "sens": sens, "mask": mask, "eta": c["eta"]}
    if c["op"] != "vjp":
        st["y"] = _measure(c, x_true, sens, mask_y, gen, dev)
    x = 0.8 * x_true + _noise(x_true.shape, gen, dev, 0.05)
    # cotangent: what the l1 loss sends back, unit modulus in the direction of the error, and noise
    e = x - x_true
    st["g"] = torch.view_as_complex(torch.nn.functional.normalize(torch.view_as_real(e), dim=-1)) + _noise(e.shape, gen, dev, 0.1)
    kind = g.GLEAM_MASK_FULL if c["full_mask"] else g.GLEAM_MASK_READOUT_INVARIANT
    rank = 3 if c["n0"] > 1 else 2
    shape = (c["batch"], c["coils"], c["frames"], rank, (c["n0"], c["n1"], c["n2"]), int(c["moving_coils"]), kind)
    st["x"] = x
    if c["op"] == "train":
        from paper_2207_08393_b200 import gleam_loop
        st["step"] = gleam_loop.DataConsistencyStep(st["y"], sens, mask, c["eta"], x_true, rank, kind)
        st["x_ch"] = torch.stack([x.real, x.imag], dim=1).contiguous().requires_grad_(True)
        st["shape"] = shape
        st["grad_ws"] = torch.empty(g.gleam_dc_grad_workspace_size(g.make_dims(*shape)), dtype=torch.uint8, device=dev)
    elif c["op"] == "modl":
        st["cg"] = g.ModlCG(*shape)
    else:
        st["dc"] = g.DataConsistency(*shape)
    return st


def run(state):
    s = state
    op = s["c"]["op"]
    sens, mask, eta = s["sens"], s["mask"], s["eta"]
    if op == "step":
        return s["dc"].forward(s["x"], s["y"], sens, mask, eta), s["dc"].vjp(s["g"], sens, mask, eta)
    if op == "forward":
        return s["dc"].forward(s["x"], s["y"], sens, mask, eta)
    if op == "vjp":
        return s["dc"].vjp(s["g"], sens, mask, eta)
    if op == "unrolled":
        dc, n = s["dc"], s["c"]["iterations"]
        if s["c"]["form"] == "aty":
            aty = dc.adjoint(s["y"], sens, mask)
            xs = [aty]                                 # every iterate is what a network's next block starts from
            for _ in range(n):
                xs.append(dc.forward_aty(xs[-1], aty, sens, mask, eta))
            return xs
        dc.prepare(s["y"], mask)
        x, gr = s["x"], s["g"]
        for _ in range(n):
            x = dc.forward_prepared(x, s["y"], sens, mask, eta)
        for _ in range(n):
            gr = dc.vjp(gr, sens, mask, eta)
        return x, gr
    if op == "modl":
        return s["cg"].solve(s["x"], s["y"], sens, mask, 0.05), s["cg"].solve_vjp(s["g"], sens, mask, 0.05)
    # train
    step, x_ch = s["step"], s["x_ch"]
    out = step.apply(x_ch)
    loss = step.loss(out)
    grad, = torch.autograd.grad(loss, x_ch)
    grad_eta = torch.empty(s["c"]["batch"], dtype=torch.float64, device=x_ch.device)
    g.gleam_dc_grad_eta(s["g"], s["x"], s["y"], sens, mask, grad_eta,
                        g.make_dims(*s["shape"], stream=torch.cuda.current_stream(), workspace=s["grad_ws"]))
    return out.detach(), loss.detach(), grad, grad_eta


# ---------------------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------------------
def work(case):
    c = dict(DEFAULTS, **case)
    V, U = _volume(c), _units(c)
    img = 8 * c["batch"] * c["frames"] * V
    sens = 8 * c["batch"] * c["coils"] * (c["frames"] if c["moving_coils"] else 1) * V
    pe = c["n1"] * c["n2"] if c["n0"] > 1 else c["n2"]
    ro = c["n0"] if c["n0"] > 1 else c["n1"]
    mask = 4 * c["batch"] * c["frames"] * (V if c["full_mask"] else pe)
    dens = min(1.0, 1 / c["accel"] + (c["center"] ** 2 / (c["n1"] * c["n2"]) if c["mask"] == "poisson" else 0.0))
    y = 8 * U * dens                                   # only sampled entries are read
    # A mask that does not depend on the readout leaves the readout axis untransformed on the image side;
    # the measurements are transformed along it where they were sampled.  14: S, conj(S) and their sum.
    n_fft = V if c["full_mask"] else pe
    one = 5 * U * math.log2(n_fft) + 7 * U             # A or A^H
    table = 0 if c["full_mask"] else 5 * U * dens * math.log2(ro)
    fwd = {"bytes": 2 * img + sens + mask + y, "flops": 2 * one + table}
    vjp = {"bytes": 2 * img + sens + mask, "flops": 2 * one}
    adj = {"bytes": img + sens + mask + y, "flops": one + table}
    aty = {"bytes": 3 * img + sens + mask, "flops": 2 * one}
    loss = {"bytes": 3 * img, "flops": 8 * img / 8}
    n = c.get("iterations", 1)
    calls = {"step": [(1, fwd), (1, vjp)], "forward": [(1, fwd)], "vjp": [(1, vjp)],
             "modl": [(1, adj), (20, vjp), (38, {"bytes": 0, "flops": 20 * img / 8})],
             "train": [(1, fwd), (1, vjp), (1, loss), (1, fwd)],
             "unrolled": [(1, adj), (n, aty)] if c.get("form") == "aty" else [(n, vjp), (n, vjp), (1, {"bytes": y, "flops": table})]}[c["op"]]
    return {k: sum(m * w[k] for m, w in calls) for k in ("bytes", "flops")}


def tolerance(case):
    # 32-bit transforms and sums differ by a few 1e-7 per call; ten conjugate-gradient steps on a system of
    # condition number up to 21 amplify that.
    return {"rel": 2e-5} if case["op"] == "modl" else {"rel": 5e-6, "max": 1e-4}

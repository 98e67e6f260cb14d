"""The work this library does for its users, as timed cases: gradient-residual
evaluations (device and host buffers), the projector and its adjoint on their
own, the regularised autograd loss, an L-BFGS reconstruction and the warm-start
network, over the geometries of the workloads the library is used on.

Geometries are tilt series: rotations spread over 360 degrees at each of
several tilts from 0 to at most 45 degrees, the way the measurements are taken.
The coefficient volumes are ellipsoidal objects (zero outside), the data
positive counts with an azimuthal modulation.  Everything is drawn from the
seed with torch and numpy alone; exact() restates the computation in 64 bits.
"""
import math

import numpy as np
import torch

from paper_2504_16446_gb300 import autograd, synth, tt


def listed():
    return [
        # The smallest call: one double-precision evaluation of the 16^3 cylinder geometry (30 projections),
        # the form used to check a set-up before a long reconstruction.  Launches and latency count.
        _case("eval_16_f64", "eval", "f64", 16, 16, 16, 16, 16, 2, 15, 2, 30.0, 8),
        # A region of interest, ragged in every extent, with a weighted (masked) detector: a small FP32 evaluation
        # between the interactive ones and a reconstruction's.
        _case("eval_roi_f32", "eval", "f32", 27, 22, 25, 31, 26, 4, 12, 4, 30.0, 8, weights=True),
        # The shape of the measured bone data set (247 projections of 65 x 55 pixels x 8 segments), l_max 2, with
        # weights: the everyday reconstruction's evaluation on a non-cubic odd-sized volume.
        _case("eval_247_l2_f32", "eval", "f32", 55, 65, 55, 65, 55, 2, 19, 13, 45.0, 8, weights=True),
        # The 64^3, l_max 4 evaluation that every iterative solve repeats (120 projections x 16 segments).
        _case("eval_64_l4_f32", "eval", "f32", 64, 64, 64, 64, 64, 4, 20, 6, 45.0, 16),
        # The same evaluation for a caller whose arrays live in (page-locked) host memory.
        _case("host_64_l4_f32", "host", "f32", 64, 64, 64, 64, 64, 4, 20, 6, 45.0, 16),
        # The forward model alone: simulating data, and the forward pass of an autograd model.
        _case("project_64_l4_f32", "project", "f32", 64, 64, 64, 64, 64, 4, 20, 6, 45.0, 16),
        # The adjoint alone at l_max 8 on the measured data set's shape: the backward pass of that model.
        _case("adjoint_247_l8_f32", "adjoint", "f32", 55, 65, 55, 65, 55, 8, 19, 13, 45.0, 8),
        # Squared loss + L2 + total variation, forward and backward through autograd: the 100^3, l_max 6 plywood loss.
        _case("composite_100_l6_f32", "composite", "f32", 100, 100, 100, 100, 100, 6, 45, 4, 45.0, 8),
        # The 128^3, l_max 4 evaluation on a bfloat16-storage handle: what the warm-started solve repeats.
        _case("eval_128_l4_bf16", "eval", "bf16", 128, 128, 128, 128, 128, 4, 24, 10, 45.0, 16),
        # The largest: 128^3, l_max 8, 240 projections of 128 x 128 pixels x 8 segments.
        _case("eval_128_l8_f32", "eval", "f32", 128, 128, 128, 128, 128, 8, 24, 10, 45.0, 8),
        # A whole call: an L-BFGS reconstruction from zero, three iterations, of the 64^3 workload.
        _case("lbfgs_64_l4_f32", "lbfgs", "f32", 64, 64, 64, 64, 64, 4, 20, 6, 45.0, 16),
        # The warm start's network on the gradient of a 128^3 volume (15 -> 32 -> 32 -> 32 -> 15 channels).
        _case("net_128_bf16", "net", "f32", 128, 128, 128, 1, 1, 4, 1, 1, 0.0, 1),
    ]


def _case(name, op, precision, nx, ny, nz, nj, nk, ell, rotations, tilts, max_tilt, segments, weights=False):
    case = {"name": name, "op": op, "precision": precision, "nx": nx, "ny": ny, "nz": nz, "nj": nj, "nk": nk,
            "ell": ell, "rotations": rotations, "tilts": tilts, "max_tilt": max_tilt, "segments": segments,
            "weights": weights}
    return case if name else {k: v for k, v in case.items() if k != "name"}


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same ranges, no dearer than the largest listed one."""
    while True:
        case = _draw(rng)
        if case["op"] == "net" or work(case)["flops"] <= 2e11 / (LBFGS_STEPS if case["op"] == "lbfgs" else 1):
            return case


def _draw(rng):
    op = rng.choice(["eval", "eval", "eval", "eval", "host", "project", "adjoint", "composite", "lbfgs", "net"])
    base = _log_int(rng, 14, 120)
    nx, ny, nz, nj, nk = (max(12, min(128, int(round(base * rng.uniform(0.8, 1.25))))) for _ in range(5))
    if op == "net":
        return _case("", op, "f32", nx, ny, nz, 1, 1, 4, 1, 1, 0.0, 1)
    ell = rng.choice([2, 4, 4, 6, 8])
    precision = rng.choice(["f32", "f32", "bf16", "f16"])
    if op == "eval" and base <= 24 and rng.random() < 0.5:
        precision, ell = "f64", 2
    if op == "composite":
        precision = "f32"
    tilts = rng.randint(1, 12)
    rotations = max(2, int(round(_log_int(rng, 24, 240) / tilts)))
    return _case("", op, precision, nx, ny, nz, nj, nk, ell, rotations, tilts,
                 0.0 if tilts == 1 else rng.choice([30.0, 45.0]), rng.choice([4, 8, 8, 12, 16]),
                 weights=rng.random() < 0.3)


def _setup(case):
    """Tilt series: `rotations` per tilt over 360 degrees, tilts from 0 to max_tilt, a few degrees of offset each."""
    R, T = case["rotations"], case["tilts"]
    alpha = np.array([2 * math.pi * i / R + math.radians(2.0) * t for t in range(T) for i in range(R)])
    beta = np.array([math.radians(case["max_tilt"]) * t / max(1, T - 1) for t in range(T) for _ in range(R)])
    s0, s1 = synth.segments(case["segments"])
    zero = np.zeros(R * T)
    return synth.Setup(shape=(case["nx"], case["ny"], case["nz"]), nj=case["nj"], nk=case["nk"], ell_max=case["ell"],
                       inner_angle=alpha, outer_angle=beta, seg_start=s0, seg_end=s1, j_offset=zero, k_offset=zero)


def _generator(seed, device="cuda"):
    gen = torch.Generator(device=device)
    gen.manual_seed(int(seed))
    return gen


def _volume(case, gen, dtype):
    """Coefficients of an object of three ellipsoids: a positive l = 0 part, higher orders falling with l."""
    K = (case["ell"] + 1) * (case["ell"] + 2) // 2
    shape = (case["nx"], case["ny"], case["nz"])
    ax = [torch.linspace(-1.0, 1.0, n, device="cuda", dtype=torch.float64) for n in shape]
    inside = torch.zeros(shape, dtype=torch.bool, device="cuda")
    for _ in range(3):
        p = torch.rand(6, generator=gen, device="cuda", dtype=torch.float64)
        r = [((ax[t] - (p[t] - 0.5)) / (0.3 + 0.4 * p[3 + t])) ** 2 for t in range(3)]
        inside |= r[0][:, None, None] + r[1][None, :, None] + r[2][None, None, :] <= 1.0
    scale = torch.cat([torch.full((2 * l + 1,), 0.5 / (1 + l), device="cuda") for l in range(0, case["ell"] + 1, 2)])
    c = torch.randn((*shape, K), generator=gen, device="cuda") * scale
    c[..., 0] += 2.0
    return (c * inside[..., None]).to(dtype).contiguous()


def _data(case, gen, dtype):
    """Counts over the object's shadow with an azimuthal modulation, scaled back to the model's units."""
    S, C = case["rotations"] * case["tilts"], case["segments"]
    j = torch.linspace(-1.0, 1.0, case["nj"], device="cuda")
    k = torch.linspace(-1.0, 1.0, case["nk"], device="cuda")
    shadow = torch.exp(-3.0 * (j[:, None] ** 2 + k[None, :] ** 2))
    phase = 6.28 * torch.rand(S, generator=gen, device="cuda")
    phi = math.pi * torch.arange(C, device="cuda") / C
    lobe = 1.0 + 0.5 * torch.cos(2.0 * phi[None, :] + phase[:, None])
    mean = 400.0 * shadow[None, :, :, None] * lobe[:, None, None, :]
    # A reconstruction's data come normalised, its coefficients well below one, so that the first step of the solver
    # (of unit length) is of the solution's own size.
    unit = 4e-3 if case["op"] == "lbfgs" else 1.0
    scale = unit * 0.1 * max(case["nx"], case["nz"]) / 400.0
    return (torch.poisson(mean, generator=gen) * scale).to(dtype).contiguous()


def _weights(case, gen, dtype):
    """Weights in (0, 1) with a tenth of the pixels masked."""
    shape = (case["rotations"] * case["tilts"], case["nj"], case["nk"], case["segments"])
    W = torch.rand(shape, generator=gen, device="cuda")
    keep = torch.rand(shape[:3], generator=gen, device="cuda") >= 0.1
    return (W * keep[..., None]).to(dtype).contiguous()


NET_LAYERS = [(32, 15), (32, 32), (32, 32), (15, 32)]


def _net_weights(seed):
    rng = np.random.default_rng(int(seed))
    return [rng.normal(0.0, math.sqrt(2.0 / (27 * ci)), (3, 3, 3, co, ci)).astype(np.float32) for co, ci in NET_LAYERS]


def _inputs(case, seed):
    """The arrays of one case, on the GPU, from the seed alone."""
    gen = _generator(seed)
    dtype = torch.float64 if case["precision"] == "f64" else torch.float32
    if case["op"] == "net":
        return {"x": 50.0 * _volume(case, gen, torch.float32), "w": _net_weights(seed)}
    given = {}
    if case["op"] != "adjoint":
        given["c"] = _volume(case, gen, dtype)
    if case["op"] == "adjoint":
        given["R"] = _data(case, gen, dtype) * torch.randn(case["rotations"] * case["tilts"], 1, 1, 1, generator=gen,
                                                           device="cuda", dtype=dtype)
    elif case["op"] != "project":
        given["I"] = _data(case, gen, dtype)
        given["W"] = _weights(case, gen, dtype) if case["weights"] else None
    return given


MU_L2, MU_TV, DELTA = 1e-3, 1e-2, 1e-2
LBFGS_STEPS = 3


def prepare(case, seed):
    state = {"case": case, **_inputs(case, seed)}
    if case["op"] == "net":
        state["net"] = tt.WarmStartNet(15, 15, np.concatenate([w.ravel() for w in state.pop("w")]))
        state["scale"] = float(state["x"].double().pow(2).mean().sqrt())
        return state
    state["handle"] = tt.Handle(_setup(case), case["precision"])
    if case["op"] == "host":
        for k in ("c", "I", "W"):
            if state[k] is not None:
                state[k] = state[k].cpu().pin_memory().numpy()
        state["g"] = torch.empty(state["handle"].volume_shape, dtype=torch.float32, pin_memory=True).numpy()
    elif case["op"] in ("eval", "adjoint"):
        state["g"] = torch.empty(state["handle"].volume_shape, dtype=state["handle"].dtype, device="cuda")
    elif case["op"] == "project":
        state["out"] = torch.empty(state["handle"].data_shape, dtype=state["handle"].dtype, device="cuda")
    return state


def run(state):
    op, h = state["case"]["op"], state.get("handle")
    if op == "eval":
        loss, g = h.gradient_residual(state["c"], state["I"], state["W"], out=state["g"])
        return {"loss": loss, "g": g}
    if op == "host":
        loss, g = h.gradient_residual_host(state["c"], state["I"], state["W"], state["g"])
        return {"loss": loss, "g": g}
    if op == "project":
        return {"I": h.project(state["c"], out=state["out"])}
    if op == "adjoint":
        return {"g": h.adjoint(state["R"], out=state["g"])}
    if op == "composite":
        c = state["c"].detach().requires_grad_(True)
        loss = (autograd.squared_loss(h, c, state["I"], state["W"]) + MU_L2 * autograd.l2_norm(h, c)
                + MU_TV * autograd.tv_huber(h, c, DELTA))
        loss.backward()
        return {"loss": loss.detach(), "g": c.grad}
    if op == "lbfgs":
        opt = tt.LBFGS(h, None, state["I"], state["W"], log=False)
        for _ in range(LBFGS_STEPS):
            opt.step()
        x, g, loss = opt.get()
        opt.close()
        return {"x": x, "g": g, "loss": loss}
    return {"y": state["net"].forward(state["x"], state["scale"])}


def _sizes(case):
    K = (case["ell"] + 1) * (case["ell"] + 2) // 2
    S = case["rotations"] * case["tilts"]
    nvox, npix = case["nx"] * case["ny"] * case["nz"], S * case["nj"] * case["nk"]
    size = 8 if case["precision"] == "f64" else 4
    # Four taps per plane and coefficient, then the segments; or the volume's coefficients first brought to the
    # (at most ell + 1) azimuthal modes a projection sees, whichever is less.
    samples, modes = npix * max(case["nx"], case["nz"]), min(case["segments"], case["ell"] + 1)
    sweep = min(8.0 * samples * K, 8.0 * samples * modes + 2.0 * nvox * S * modes * K)
    sweep += 2.0 * npix * case["segments"] * modes
    return nvox * K * size, npix * case["segments"] * size, sweep, nvox * K


def work(case):
    if case["op"] == "net":
        nvox = case["nx"] * case["ny"] * case["nz"]
        return {"bytes": 8.0 * 15 * nvox, "flops": 2.0 * 27 * nvox * sum(a * b for a, b in NET_LAYERS)}
    vol, data, sweep, n = _sizes(case)
    weighted = data if case["weights"] else 0
    if case["op"] in ("project", "adjoint"):
        return {"bytes": float(vol + data), "flops": sweep}
    one = {"bytes": 2.0 * vol + data + weighted, "flops": 2.0 * sweep}
    if case["op"] == "composite":
        return {"bytes": one["bytes"], "flops": one["flops"] + 30.0 * n}
    if case["op"] == "lbfgs":
        return {"bytes": (LBFGS_STEPS + 1) * one["bytes"], "flops": (2 * LBFGS_STEPS + 1) * sweep}
    return one


# ------------------------------------------------------------ in 64 bits


def _rotation(axis, t):
    x, y, z = axis
    c, s = math.cos(t), math.sin(t)
    C = 1.0 - c
    return np.array([[c + x * x * C, x * y * C - z * s, x * z * C + y * s],
                     [y * x * C + z * s, c + y * y * C, y * z * C - x * s],
                     [z * x * C - y * s, z * y * C + x * s, c + z * z * C]])


def _harmonics(q, ell):
    """Real orthonormal even-order spherical harmonics at the unit vectors q [n, 3], order (l, m = -l..l)."""
    ct, phi = np.clip(q[:, 2], -1.0, 1.0), np.arctan2(q[:, 1], q[:, 0])
    st = np.sqrt(np.maximum(0.0, 1.0 - ct * ct))
    P = {}
    for m in range(ell + 1):
        P[m, m] = np.ones_like(ct) if m == 0 else (2 * m - 1) * st * P[m - 1, m - 1]
        if m + 1 <= ell:
            P[m + 1, m] = (2 * m + 1) * ct * P[m, m]
        for l in range(m + 2, ell + 1):
            P[l, m] = ((2 * l - 1) * ct * P[l - 1, m] - (l + m - 1) * P[l - 2, m]) / (l - m)
    cols = []
    for l in range(0, ell + 1, 2):
        for m in range(-l, l + 1):
            a = abs(m)
            n = math.sqrt((2 * l + 1) / (4 * math.pi) * math.factorial(l - a) / math.factorial(l + a))
            cols.append(n * P[l, a] * (1.0 if m == 0 else math.sqrt(2.0) * (np.cos(a * phi) if m > 0 else np.sin(a * phi))))
    return np.stack(cols, axis=1)


class _Model:
    """The forward model and its transpose for one case, one projection at a time, in double precision."""

    def __init__(self, case):
        self.case, self.st = case, _setup(case)
        x, w = np.polynomial.legendre.leggauss(32)
        s0, s1 = self.st.seg_start, self.st.seg_end
        self.phi = 0.5 * (s1 + s0)[:, None] + 0.5 * (s1 - s0)[:, None] * x[None, :]
        self.w = 0.5 * w

    def projection(self, s):
        """(B [C, K], tap indices [4, n], tap weights [4, n]) with n = planes x pixels of projection s."""
        st, N = self.st, self.st.shape
        R = _rotation((1.0, 0.0, 0.0), st.outer_angle[s]) @ _rotation((0.0, 1.0, 0.0), st.inner_angle[s])
        p, j, k = (R.T @ np.array(v) for v in ((0.0, 0.0, 1.0), (0.0, 1.0, 0.0), (1.0, 0.0, 0.0)))
        q0, q90 = k, j
        q = np.cos(self.phi)[..., None] * q0 + np.sin(self.phi)[..., None] * q90
        Y = _harmonics(q.reshape(-1, 3), st.ell_max).reshape(*self.phi.shape, -1)
        B = torch.as_tensor(np.einsum("cq,cqi->ci", np.broadcast_to(self.w, self.phi.shape), Y), device="cuda")
        m = int(np.argmax(np.abs(p) >= (1.0 - 1e-12) * np.abs(p).max()))
        u, v = [t for t in range(3) if t != m]
        dj = torch.arange(st.nj, device="cuda", dtype=torch.float64) - 0.5 * (st.nj - 1)
        dk = torch.arange(st.nk, device="cuda", dtype=torch.float64) - 0.5 * (st.nk - 1)
        plane = torch.arange(N[m], device="cuda", dtype=torch.float64) - 0.5 * (N[m] - 1)

        def coordinate(t):
            slope = p[t] / p[m]
            at = (dj[:, None] * (j[t] - j[m] * slope) + dk[None, :] * (k[t] - k[m] * slope)).reshape(1, -1)
            return (at + slope * plane[:, None] + 0.5 * (N[t] - 1)).reshape(-1)

        pu, pv = coordinate(u), coordinate(v)
        pm = torch.arange(N[m], device="cuda").repeat_interleave(st.nj * st.nk)
        fu, fv = pu.floor(), pv.floor()
        stride = (N[1] * N[2], N[2], 1)
        index, weight = [], []
        for a in (0, 1):
            for b in (0, 1):
                iu, iv = fu.long() + a, fv.long() + b
                inside = (iu >= 0) & (iu < N[u]) & (iv >= 0) & (iv < N[v])
                wu, wv = (pu - fu) if a else 1.0 - (pu - fu), (pv - fv) if b else 1.0 - (pv - fv)
                weight.append(wu * wv * inside / abs(p[m]))
                index.append(pm * stride[m] + iu.clamp(0, N[u] - 1) * stride[u] + iv.clamp(0, N[v] - 1) * stride[v])
        return B, index, weight

    def forward(self, c, parts):
        B, index, weight = parts
        f, first = c.reshape(-1, c.shape[-1]), B.shape[0] < B.shape[1]
        if first:
            f = f @ B.T
        npix = self.st.nj * self.st.nk
        ray = sum((w[:, None] * f[i]).reshape(-1, npix, f.shape[1]).sum(0) for i, w in zip(index, weight))
        return (ray if first else ray @ B.T).reshape(self.st.nj, self.st.nk, -1)

    def adjoint(self, r, parts, g):
        B, index, weight = parts
        first = B.shape[1] <= B.shape[0]
        r = r.reshape(-1, r.shape[-1])
        if first:
            r = r @ B
        planes = index[0].numel() // r.shape[0]
        back = torch.zeros((g.numel() // g.shape[-1], r.shape[1]), dtype=torch.float64, device="cuda")
        rows = r.repeat(planes, 1)
        for i, w in zip(index, weight):
            back.index_add_(0, i, w[:, None] * rows)
        g += (back if first else back @ B).reshape(g.shape)

    def evaluate(self, c, I, W):
        loss = 0.0
        g = torch.zeros((*self.st.shape, self.st.K), dtype=torch.float64, device="cuda")
        for s in range(self.st.S):
            parts = self.projection(s)
            r = (self.forward(c, parts) if c is not None else 0.0) - I[s].double()
            wr = r if W is None else W[s].double() * r
            loss += float((wr * r).sum())
            self.adjoint(2.0 * wr, parts, g)
        return loss, g


def _lbfgs(model, I, W):
    """L-BFGS from zero: two-loop recursion, first step 1/|g| along -g, backtracking Armijo (c1 = 1e-4, halving)."""
    x = torch.zeros((*model.st.shape, model.st.K), dtype=torch.float64, device="cuda")
    loss, g = model.evaluate(None, I, W)
    pairs = []
    for _ in range(LBFGS_STEPS):
        q, alphas = g.clone(), []
        for s, y in reversed(pairs):
            a = float((s * q).sum() / (s * y).sum())
            alphas.append(a)
            q -= a * y
        if pairs:
            s, y = pairs[-1]
            q *= float((s * y).sum() / (y * y).sum())
        for (s, y), a in zip(pairs, reversed(alphas)):
            q += (a - float((y * q).sum() / (s * y).sum())) * s
        d, step = -q, 1.0 if pairs else 1.0 / float(g.norm())
        slope = float((g * d).sum())
        for _ in range(20):
            lt, gt = model.evaluate(x + step * d, I, W)
            if lt <= loss + 1e-4 * step * slope:
                break
            step *= 0.5
        s, y = step * d, gt - g
        if float((s * y).sum()) > 1e-10 * float(s.norm()) * float(y.norm()):
            pairs.append((s, y))
        x, loss, g = x + s, lt, gt
    return x, g, loss


def _tv(c):
    """Huber total variation per channel and its gradient (forward differences, Neumann boundary)."""
    d = []
    for t in range(3):
        e = torch.zeros_like(c)
        n = c.shape[t]
        e.narrow(t, 0, n - 1).copy_(c.narrow(t, 1, n - 1) - c.narrow(t, 0, n - 1))
        d.append(e)
    norm = (d[0] ** 2 + d[1] ** 2 + d[2] ** 2).sqrt()
    value = float(torch.where(norm <= DELTA, norm ** 2 / (2 * DELTA), norm - 0.5 * DELTA).sum())
    g = torch.zeros_like(c)
    for t in range(3):
        f = d[t] / norm.clamp(min=DELTA)
        g -= f
        n = c.shape[t]
        g.narrow(t, 1, n - 1).add_(f.narrow(t, 0, n - 1))
    return value, g


def _network(x, weights, scale):
    a = x.double() / scale
    nx, ny, nz = a.shape[:3]
    for i, w in enumerate(weights):
        w = torch.as_tensor(w, device="cuda", dtype=torch.float64)
        pad = torch.nn.functional.pad(a, (0, 0, 1, 1, 1, 1, 1, 1))
        out = torch.zeros((nx * ny * nz, w.shape[3]), dtype=torch.float64, device="cuda")
        for dx in range(3):
            for dy in range(3):
                for dz in range(3):
                    part = pad[dx:dx + nx, dy:dy + ny, dz:dz + nz].reshape(-1, a.shape[3])
                    out.addmm_(part, w[dx, dy, dz].T)
        a = out.reshape(nx, ny, nz, -1)
        if i + 1 < len(weights):
            a = a.clamp(min=0.0)
    return scale * a


def exact(case, seed):
    given = _inputs(case, seed)
    if case["op"] == "net":
        return {"y": _network(given["x"], given["w"], float(given["x"].double().pow(2).mean().sqrt()))}
    model = _Model(case)
    if case["op"] == "project":
        c = given["c"].double()
        return {"I": torch.stack([model.forward(c, model.projection(s)) for s in range(model.st.S)])}
    if case["op"] == "adjoint":
        g = torch.zeros((*model.st.shape, model.st.K), dtype=torch.float64, device="cuda")
        for s in range(model.st.S):
            model.adjoint(given["R"][s].double(), model.projection(s), g)
        return {"g": g}
    if case["op"] == "lbfgs":
        x, g, loss = _lbfgs(model, given["I"], given["W"])
        return {"x": x, "g": g, "loss": loss}
    loss, g = model.evaluate(given["c"].double(), given["I"], given["W"])
    if case["op"] == "composite":
        c = given["c"].double()
        tv, gtv = _tv(c)
        loss += MU_L2 * float((c * c).sum()) + MU_TV * tv
        g = g + 2.0 * MU_L2 * c + MU_TV * gtv
    return {"loss": loss, "g": g}

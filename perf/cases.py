"""The work that programs built on this package have it do, as cases that can be timed and compared.

A case goes through the public entry points only (`lgf.Lattice`, `lgf.Batch`, `lgf.fix`, `autograd`), on seeded
fields of the kind the tests and the benchmark use (rough-gauge SU(3) fields, `inputs.rough_gauge_field_cuda`).
Kinds:

  fix      store links, gauge-fix them, read links (and the gauge transformation) back; on a context that is kept
  oneshot  `lgf.fix` on host arrays: context, copies and clean-up in the call
  batch    an ensemble of lattices fixed by one graph launch
  wilson   Wilson-action sweeps (heat bath and overrelaxation) of stored links, and the plaquette
  step     one differentiable step forward and its vector-Jacobian product
  unroll   K differentiable steps with checkpoints, the gluon propagator of the result, and the gradient
"""
import math

import numpy as np
import torch

from paper_1301_3460_gb300 import autograd, inputs, lgf

ALPHA = 0.08  # the step of the method's runs
TOL = 1e-15   # and their stop on theta

LENGTHS = (4, 6, 8, 12, 16, 24, 32, 48, 64)  # line lengths the draw takes (those of the tests)


def _fix(name, dims, eps=0.3, iters=0, mixed=False, accel32=False, switch=1e-6, links18=False, track=True):
    # iters > 0: exactly that many iterations (a block of a longer run); 0: to theta < TOL
    return {"name": name, "kind": "fix", "dims": "x".join(map(str, dims)), "eps": eps, "iters": iters, "mixed": mixed,
            "accel32": accel32, "switch": switch, "links18": links18, "track": track}


def listed():
    return [
        # the parity lattice: a whole FP64 fix of a small field, where launches and latency count
        _fix("fix_fp64_8x4", (8, 8, 8, 8)),
        # a script's one call on a numpy field: nothing is kept, the context is made and freed in the call
        {"name": "oneshot_host_16x12x8x6", "kind": "oneshot", "dims": "16x12x8x6", "eps": 0.3},
        # ragged radix-3 extents, rows kept as 18 reals, gauge transformation not wanted
        _fix("fix_fp64_24x12x8x6_18real", (24, 12, 8, 6), links18=True, track=False),
        # the headline: a 32^4 configuration to theta < 1e-15 in FP64
        _fix("fix_fp64_32x4", (32, 32, 32, 32)),
        # a large lattice in FP64: a block of ten iterations of a longer fix (lines split over two lanes)
        _fix("fix_fp64_48x4_10it", (48, 48, 48, 48), iters=10),
        # the mixed-precision production mode at the headline size
        _fix("fix_mixed_32x4", (32, 32, 32, 32), mixed=True),
        # mixed, with the accelerator's transforms in FP32 in the FP64 iterations too, on a long time axis
        _fix("fix_mixed_accel32_32x3x64", (32, 32, 32, 64), eps=0.15, mixed=True, accel32=True),
        # an ensemble of mixed sizes in one launch
        {"name": "batch_mixed_14", "kind": "batch", "sizes": "8*16x16x16x16+4*24x24x24x24+2*32x32x32x64", "eps": 0.3},
        # configuration generation: one compound sweep (heat bath + 4 overrelaxations) in FP64 at beta = 6
        {"name": "wilson_fp64_32x4", "kind": "wilson", "dims": "32x32x32x32", "beta": 6.0, "heatbath": 1, "overrelax": 4,
         "bits": 64},
        # the same with the FP32 generator
        {"name": "wilson_fp32_32x4", "kind": "wilson", "dims": "32x32x32x32", "beta": 6.0, "heatbath": 1, "overrelax": 4,
         "bits": 32},
        # training through the fixing: one step and its vector-Jacobian product at full size
        {"name": "step_vjp_32x4", "kind": "step", "dims": "32x32x32x32", "eps": 0.3},
        # the gradient of the gluon propagator through ten unrolled steps with checkpoints
        {"name": "unroll_16x4_k10", "kind": "unroll", "dims": "16x16x16x16", "eps": 0.3, "steps": 10, "every": 5},
    ]


def _drawn_dims(rng, vmin, vmax):
    while True:
        want = math.exp(rng.uniform(math.log(vmin), math.log(vmax)))
        d = [rng.choice(LENGTHS) for _ in range(4)]
        v = d[0] * d[1] * d[2] * d[3]
        # the extents' tiles have to fit (planes up to 64x48, pencils up to 64x64)
        if abs(math.log(v / want)) < 0.35 and d[1] * (d[0] + 1) <= 3500 and d[2] * d[3] <= 4096:
            return "x".join(map(str, d))


def draw(rng):
    kind = rng.choice(("fix", "fix", "fix", "mixed", "mixed", "oneshot", "batch", "wilson", "step", "unroll"))
    eps = round(rng.uniform(0.15, 0.5), 3)
    if kind == "fix":
        c = _fix("", (4, 4, 4, 4), eps=eps, iters=rng.randint(1, 40), links18=rng.random() < 0.3, track=rng.random() < 0.7)
        c["dims"] = _drawn_dims(rng, 256, 1 << 20)
    elif kind == "mixed":
        c = _fix("", (4, 4, 4, 4), eps=eps, mixed=True, accel32=rng.random() < 0.4, switch=rng.choice((1e-6, 1e-9)))
        c["dims"] = _drawn_dims(rng, 4096, 1 << 20)
    elif kind == "oneshot":
        c = {"kind": "oneshot", "dims": _drawn_dims(rng, 256, 1 << 16), "eps": eps}
    elif kind == "batch":
        c = {"kind": "batch", "eps": eps,
             "sizes": "+".join("%d*%s" % (rng.randint(1, 3), _drawn_dims(rng, 4096, 1 << 18)) for _ in range(rng.randint(2, 3)))}
    elif kind == "wilson":
        c = {"kind": "wilson", "dims": _drawn_dims(rng, 256, 1 << 20), "beta": round(rng.uniform(5.7, 6.2), 3),
             "heatbath": rng.randint(1, 2), "overrelax": rng.randint(0, 2), "bits": rng.choice((64, 64, 32))}
    elif kind == "step":
        c = {"kind": "step", "dims": _drawn_dims(rng, 256, 1 << 20), "eps": eps}
    else:
        c = {"kind": "unroll", "dims": _drawn_dims(rng, 256, 1 << 17), "eps": eps, "steps": rng.randint(2, 12),
             "every": rng.randint(1, 6)}
    c.pop("name", None)
    return c


def _dims(text):
    return tuple(int(v) for v in text.split("x"))


def _volume(dims):
    return int(np.prod(dims))


def _sizes(case):
    out = []
    for part in case["sizes"].split("+"):
        n, d = part.split("*")
        out += [_dims(d)] * int(n)
    return out


def prepare(case, seed):
    kind = case["kind"]
    stream = torch.cuda.current_stream()
    if kind == "batch":
        sizes = _sizes(case)
        links = [inputs.rough_gauge_field_cuda(d, case["eps"], 1000 * seed + i) for i, d in enumerate(sizes)]
        return {"case": case, "batch": lgf.Batch(sizes, mixed=True, stream=stream), "links": links}
    dims = _dims(case["dims"])
    # generated configurations are far smoother than the fields the fixing starts from
    U = inputs.rough_gauge_field_cuda(dims, case.get("eps", 0.35), seed)
    s = {"case": case, "dims": dims, "links": U}
    if kind == "oneshot":
        s["links"] = U.cpu().numpy()
    elif kind == "fix":
        lat = lgf.Lattice(dims, mixed=case["mixed"], track_gauge=case["track"], links18=case["links18"], stream=stream)
        if case["mixed"]:
            lat.set_switch_tol(case["switch"])
            if case["accel32"]:
                lat.set_accel_precision(32)
        s["lat"] = lat
    elif kind == "wilson":
        s["lat"] = lgf.Lattice(dims, track_gauge=False, stream=stream)
        s["lat"].set_generator_precision(case["bits"])
        s["seed"] = seed
    elif kind == "step":
        s["lat"] = lgf.Lattice(dims, track_gauge=False, stream=stream)
        s["cotangent"] = _cotangent(dims, seed)
    else:
        s["lat"] = lgf.Lattice(dims, track_gauge=False, stream=stream)
    return s


def _cotangent(dims, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn((4, _volume(dims), 3, 3), dtype=torch.complex128, device="cuda", generator=g)


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "oneshot":
        links, gauge, info = lgf.fix(s["links"], s["dims"], ALPHA, TOL, 2000)
        return {"links": links, "gauge": gauge, "F": info["F"], "iters": info["iters"]}
    if kind == "batch":
        b = s["batch"]
        for i, U in enumerate(s["links"]):
            b.set_links(i, U)
        r = b.fix(ALPHA, TOL, 2000)
        return {"links": [b.get_links(i, device="cuda") for i in range(b.n)],
                "gauge": [b.get_gauge(i, device="cuda") for i in range(b.n)], "F": np.array(r["F"]),
                "iters": np.array(r["iters"])}
    lat = s["lat"]
    if kind == "fix":
        lat.set_links(s["links"])
        r = lat.fix(ALPHA, 0.0, c["iters"]) if c["iters"] else lat.fix(ALPHA, TOL, 2000)
        out = {"links": lat.get_links(device="cuda"), "F": r["F"], "iters": r["iters"]}
        if c["track"]:
            out["gauge"] = lat.get_gauge(device="cuda")
        return out
    if kind == "wilson":
        lat.set_links(s["links"])
        lat.wilson_sweeps(c["beta"], s["seed"], 0, c["heatbath"], c["overrelax"])
        return {"links": lat.get_links(device="cuda"), "plaquette": lat.plaquette()}
    if kind == "step":
        out = lat.step_fwd(s["links"], ALPHA)
        lat.set_links(s["links"])
        return {"links": out, "cotangent": lat.step_bwd(s["cotangent"], ALPHA)}
    U = s["links"].clone().requires_grad_(True)
    D, _ = autograd.gluon_after_fixing(U, s["dims"], c["steps"], ALPHA, c["every"], lat=lat)
    D.backward()
    return {"D": D, "grad": U.grad}


# ---------------------------------------------------------------- what a pass cannot do without

# per site: links in or out (complex128 3x3 of four directions), the same of one matrix; one iteration in FP64 reads
# and writes twelve reals per link and per gauge matrix and needs about 2650 flops (products, transforms, Gram-Schmidt)
_IO, _IO1, _ITER, _FLOPS = 4 * 144, 144, 2 * 5 * 96, 2650


def work(case):
    kind = case["kind"]
    if kind == "batch":
        V = sum(_volume(d) for d in _sizes(case))
        # about 33 FP32 iterations (half the bytes) and 12 in FP64
        return {"bytes": V * (2 * _IO + _IO1 + 45 * _ITER // 2 + 6 * _ITER), "flops": V * 45 * _FLOPS}
    V = _volume(_dims(case["dims"]))
    if kind == "wilson":
        sweeps = case["heatbath"] * (1 + case["overrelax"])
        # per link and sweep: 19 links are needed, each is written once per sweep and read at least once; 3514 flops
        return {"bytes": V * (2 * _IO + sweeps * 2 * 4 * 96 * case["bits"] // 64), "flops": V * 4 * 3514 * sweeps}
    if kind == "step":
        return {"bytes": V * 4 * _IO, "flops": V * (_FLOPS + 7000)}
    if kind == "unroll":
        return {"bytes": V * (2 * _IO + case["steps"] * 3 * _ITER), "flops": V * case["steps"] * (2 * _FLOPS + 7000)}
    n = case.get("iters") or 45
    per = _ITER * 5 // 8 if case.get("mixed") else _ITER
    return {"bytes": V * (2 * _IO + _IO1 + n * per), "flops": V * n * _FLOPS}


# ---------------------------------------------------------------- the same in plain torch, FP64

def _mm(a, b):
    return (a.unsqueeze(-1) * b.unsqueeze(-3)).sum(-2)


def _dag(a):
    return a.transpose(-1, -2).conj()


def _with_row2(m):
    # row 2 = conj(row 0 x row 1)
    r0, r1 = m[..., 0, :], m[..., 1, :]
    return torch.stack((r0, r1, torch.linalg.cross(r0, r1).conj()), -2)


class _Plain:
    """The method on a (4, V, 3, 3) field with plain torch operations."""

    def __init__(self, dims, device):
        self.dims = dims
        self.V = _volume(dims)
        p2 = torch.zeros(dims[::-1], dtype=torch.float64, device=device)
        top = 0.0
        for mu, L in enumerate(dims):
            s = 4 * torch.sin(math.pi * torch.arange(L, dtype=torch.float64, device=device) / L) ** 2
            top += float(s.max())
            shape = [1] * 4
            shape[3 - mu] = L
            p2 = p2 + s.reshape(shape)
        self.mult = torch.where(p2 > 0, top / torch.where(p2 > 0, p2, 1.0), 0.0)

    def shift(self, f, mu, d):
        # f(x + d mu) of a (V, ...) field
        g = f.reshape(self.dims[::-1] + f.shape[1:])
        return torch.roll(g, -d, 3 - mu).reshape(f.shape)

    def delta(self, U):
        M = 0
        for mu in range(4):
            M = M + self.shift(U[mu], mu, -1) - U[mu]
        D = M - _dag(M)
        tr = (D[..., 0, 0] + D[..., 1, 1] + D[..., 2, 2]) / 3
        return D - tr[..., None, None] * torch.eye(3, dtype=U.dtype, device=U.device)

    def theta(self, D):
        return float((D.real ** 2 + D.imag ** 2).sum()) / (3 * self.V)

    def F(self, U):
        return float((U[..., 0, 0] + U[..., 1, 1] + U[..., 2, 2]).real.sum()) / (12 * self.V)

    def transformation(self, D):
        cols = []
        for i in range(2):
            for j in range(3):
                k = torch.fft.fftn(D[..., i, j].reshape(self.dims[::-1]), dim=(0, 1, 2, 3))
                cols.append(torch.fft.ifftn(k * self.mult, dim=(0, 1, 2, 3)).reshape(-1))
        X = torch.stack(cols, -1).reshape(-1, 2, 3) * (0.5 * ALPHA)
        X = X + torch.eye(3, dtype=D.dtype, device=D.device)[:2]
        r0 = X[:, 0] / torch.sqrt((X[:, 0].real ** 2 + X[:, 0].imag ** 2).sum(-1, keepdim=True))
        r1 = X[:, 1] - (r0.conj() * X[:, 1]).sum(-1, keepdim=True) * r0
        r1 = r1 / torch.sqrt((r1.real ** 2 + r1.imag ** 2).sum(-1, keepdim=True))
        return _with_row2(torch.stack((r0, r1), -2))

    def step(self, U, D):
        g = self.transformation(D)
        return torch.stack([_with_row2(_mm(_mm(g[:, :2], U[mu]), _dag(self.shift(g, mu, 1)))) for mu in range(4)]), g

    def fix(self, U, iters, G=None):
        n = 0
        U = _with_row2(U)
        while True:
            D = self.delta(U)
            if (iters and n == iters) or (not iters and (self.theta(D) < TOL or n == 2000)):
                return U, G, n
            U, g = self.step(U, D)
            if G is not None:
                G = _with_row2(_mm(g[:, :2], G))
            n += 1


def _gluon(plain, U):
    # D(p) averaged over the four momenta with one k_mu = 1
    out = 0
    for mu in range(4):
        A = (U[mu] - _dag(U[mu])) / 2j
        tr = (A[..., 0, 0] + A[..., 1, 1] + A[..., 2, 2]) / 3
        A = A - tr[..., None, None] * torch.eye(3, dtype=U.dtype, device=U.device)
        A = A.reshape(plain.dims[::-1] + (3, 3))
        for nu in range(4):
            L = plain.dims[nu]
            shape = [1] * 6
            shape[3 - nu] = L
            w = torch.exp(-2j * math.pi * torch.arange(L, dtype=torch.float64, device=U.device) / L).reshape(shape)
            P = (w * A).sum((0, 1, 2, 3))
            out = out + (P.real ** 2 + P.imag ** 2).sum()
    return out * 2 / (8 * 3 * plain.V) / 4


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "wilson") or case.get("mixed"):
        # mixed fixes end within FP32 rounding of a global rotation, which no 64-bit run reproduces; generated links
        # depend on the generator's own random stream
        return None
    dims = _dims(case["dims"])
    U = inputs.rough_gauge_field_cuda(dims, case["eps"], seed)
    plain = _Plain(dims, U.device)
    if kind in ("fix", "oneshot"):
        track = case.get("track", True)
        G = torch.eye(3, dtype=U.dtype, device=U.device).expand(plain.V, 3, 3) if track else None
        links, G, n = plain.fix(U, case.get("iters", 0), G)
        out = {"links": links, "F": plain.F(links), "iters": n}
        return dict(out, gauge=G) if track else out
    U.requires_grad_(True)
    if kind == "step":
        # the step reads rows 0 and 1
        W = _with_row2(U[..., :2, :])
        out, _ = plain.step(W, plain.delta(W))
        grad, = torch.autograd.grad(out, U, _cotangent(dims, seed))
        return {"links": out.detach(), "cotangent": grad}
    W = _with_row2(U[..., :2, :])
    for _ in range(case["steps"]):
        W, _g = plain.step(W, plain.delta(W))
    D = _gluon(plain, W)
    grad, = torch.autograd.grad(D, U)
    return {"D": D.detach(), "grad": grad}

"""What a user of this framework has it do, as timed cases.

A program that gauge-fixes an ensemble keeps one handle per lattice shape and
brings configuration after configuration to it: load the links, fix to the
tolerance, take the result.  FP64 handles give back the fixed links in FP64.
Mixed handles (FP32 links, FP64-accurate tail) give back the gauge
transformation, which such a program moves to the GPU in single precision and
applies to its propagators and sources; the functional F, which selects the
Gribov copy, comes back in FP64.  The warm-start network is trained with one
training step per configuration, and its layers are run on device activations.

Kinds of cases:
  fix    load_links (device tensor), fix, functional, then store_links (FP64)
         or store_gauge (mixed)
  batch  several lattices of mixed sizes fixed by one GaugeBatch
  conv   one network layer, forward or backward with respect to its input
  train  one training step with its gradient (learning rate of the recipe)
"""
import math

import numpy as np
import torch

import paper_1208_1186_gb300 as lgf
from paper_1208_1186_gb300 import _lib

ALPHA = 0.08
MAX_ITER = 2000
LEARNING_RATE = 1e-5
# updates from a random gauge to theta < 1e-12 / 1e-15 on such inputs
UPDATES = {1e-12: 20, 1e-15: 26}


def _dims(d):
    return "x".join(str(v) for v in d)


def _fix(name, dims, dtype, tol, scale, exp_order=1):
    return {"name": name, "kind": "fix", "dims": _dims(dims), "dtype": dtype, "tol": tol, "scale": scale,
            "exp_order": exp_order}


def listed():
    return [
        # a study on a tiny lattice in plain FP64: latency and launches
        _fix("f64 8^4", (8, 8, 8, 8), "f64", 1e-12, 0.3),
        # plain FP64 on a production lattice, the yardstick of the mixed method
        _fix("f64 32^4", (32, 32, 32, 32), "f64", 1e-15, 0.5),
        # 12-real FP64 storage on extents with factors 3 and 5
        _fix("f64r12 12x18x10x20", (12, 18, 10, 20), "f64_r12", 1e-12, 0.5),
        # the exact exponential in the gauge step
        _fix("f64 16^3x32 exact exp", (16, 16, 16, 32), "f64", 1e-12, 0.5, 0),
        # mixed precision: the smallest lattice, the training-set size, the
        # headline lattice
        _fix("f32 8^4", (8, 8, 8, 8), "f32", 1e-15, 0.5),
        _fix("f32 16^4", (16, 16, 16, 16), "f32", 1e-15, 0.5),
        _fix("f32 32^4", (32, 32, 32, 32), "f32", 1e-15, 0.5),
        # the finite-temperature lattice in 12-real storage
        _fix("f32r12 48^3x8", (48, 48, 48, 8), "f32_r12", 1e-15, 0.6),
        # uneven extents with factors 2, 3 and 5
        _fix("f32 20x30x18x40", (20, 30, 18, 40), "f32", 1e-15, 0.5),
        # an ensemble of mixed sizes in one batch, two of each shape
        {"name": "batch 8 f32", "kind": "batch", "dims": "16x16x16x16,24x24x24x48,32x32x32x8,20x20x20x20",
         "each": 2, "dtype": "f32", "tol": 1e-15, "scale": 0.5},
        # the network's widest layer on an evaluation lattice
        {"name": "conv 24^4", "kind": "conv", "dims": "24x24x24x24", "layer": 1, "backward": False},
        # one training step on a training configuration
        {"name": "train 16^4", "kind": "train", "dims": "16x16x16x16", "scale": 0.5},
    ]


_EXTENTS = [n for n in range(4, 49) if n in {2 ** a * 3 ** b * 5 ** c for a in range(6) for b in range(4)
                                             for c in range(3)}]


def _draw_dims(rng, lo, hi):
    """Extents that are products of 2, 3 and 5 (mostly even ones, often a
    spatial cube), the volume near a log-uniform target in [lo, hi]."""
    want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    while True:
        pool = _EXTENTS if rng.random() < 0.2 else [n for n in _EXTENTS if n % 2 == 0]
        d = [rng.choice(pool) for _ in range(4)]
        if rng.random() < 0.6:  # spatial cube
            d = [d[0]] * 3 + [d[3]]
        V = d[0] * d[1] * d[2] * d[3]
        if 0.6 * want <= V <= min(hi, 1.6 * want) and V >= lo:
            return tuple(d)


def draw(rng):
    kind = rng.choice(["f64", "f32", "f32", "f32", "batch", "conv", "train"])
    if kind == "f64":
        dtype = rng.choice(["f64", "f64", "f64_r12"])
        tol = rng.choice([1e-12, 1e-15])
        c = _fix("", _draw_dims(rng, 1000, 400000), dtype, tol, rng.choice([0.3, 0.4, 0.5]), rng.choice([1, 1, 1, 0]))
    elif kind == "f32":
        dtype = rng.choice(["f32", "f32", "f32_r12"])
        c = _fix("", _draw_dims(rng, 1000, 1 << 20), dtype, 1e-15, rng.choice([0.4, 0.5, 0.6]),
                 rng.choice([1, 1, 1, 1, 0]))
    elif kind == "batch":
        shapes = [_draw_dims(rng, 2000, 200000) for _ in range(rng.randint(2, 4))]
        c = {"kind": "batch", "dims": ",".join(_dims(d) for d in shapes), "each": rng.randint(1, 4),
             "dtype": rng.choice(["f32", "f32_r12"]), "tol": 1e-15, "scale": 0.5}
    elif kind == "conv":
        layer = rng.randint(1, 3)
        c = {"kind": "conv", "dims": _dims(_draw_dims(rng, 2000, 331776)), "layer": layer,
             "backward": layer > 1 and rng.random() < 0.5}
    else:
        while True:
            d = _draw_dims(rng, 2000, 70000)
            if d[0] * d[1] * d[2] * d[3] % 16 == 0:
                break
        c = {"kind": "train", "dims": _dims(d), "scale": rng.choice([0.4, 0.5])}
    c.pop("name", None)
    return c


def _parse(text):
    return tuple(int(v) for v in text.split("x"))


def _members(case):
    return [_parse(t) for t in case["dims"].split(",") for _ in range(case["each"])]


# ---------------------------------------------------------------------------
# inputs: special unitary links around exp(i scale sum_a r_a lambda_a / 2), r_a
# normal (the second-order series, reunitarised), behind a random gauge
# transformation drawn the same way with scale 1
# ---------------------------------------------------------------------------
def _gell_mann(device):
    lam = np.zeros((8, 3, 3), dtype=np.complex128)
    lam[0, 0, 1] = lam[0, 1, 0] = 1
    lam[1, 0, 1], lam[1, 1, 0] = -1j, 1j
    lam[2, 0, 0], lam[2, 1, 1] = 1, -1
    lam[3, 0, 2] = lam[3, 2, 0] = 1
    lam[4, 0, 2], lam[4, 2, 0] = -1j, 1j
    lam[5, 1, 2] = lam[5, 2, 1] = 1
    lam[6, 1, 2], lam[6, 2, 1] = -1j, 1j
    lam[7, 0, 0] = lam[7, 1, 1] = 1 / math.sqrt(3)
    lam[7, 2, 2] = -2 / math.sqrt(3)
    return torch.from_numpy(lam).to(device)


def _mm(a, b):
    """Products of 3x3 matrices, elementwise (batched GEMMs are slow at 3x3)."""
    return a[..., :, :1] * b[..., :1, :] + a[..., :, 1:2] * b[..., 1:2, :] + a[..., :, 2:] * b[..., 2:, :]


def _cross(a, b):
    a0, a1, a2 = a.unbind(-1)
    b0, b1, b2 = b.unbind(-1)
    return torch.stack((a1 * b2 - a2 * b1, a2 * b0 - a0 * b2, a0 * b1 - a1 * b0), -1)


def _reunit(m):
    """Gram-Schmidt on rows 1 and 2, row 3 their conjugated cross product."""
    def unit(r):
        return r / (r.real ** 2 + r.imag ** 2).sum(-1, keepdim=True).sqrt()
    r1 = unit(m[..., 0, :])
    r2 = m[..., 1, :]
    r2 = unit(r2 - (r1.conj() * r2).sum(-1, keepdim=True) * r1)
    return torch.stack((r1, r2, _cross(r1, r2).conj()), -2)


def _random_su3(n, scale, gen):
    out = torch.empty((n, 3, 3), dtype=torch.complex128, device="cuda")
    basis = torch.view_as_real((0.5j * scale) * _gell_mann("cuda")).reshape(8, 18)
    eye = torch.eye(3, dtype=torch.complex128, device="cuda")
    for a in range(0, n, 1 << 20):
        m = min(1 << 20, n - a)
        r = torch.randn((m, 8), dtype=torch.float64, device="cuda", generator=gen)
        X = torch.view_as_complex((r @ basis).reshape(m, 3, 3, 2))
        out[a:a + m] = _reunit(eye + X + 0.5 * _mm(X, X))
    return out


def _roll_fwd(a, mu):
    """a(x + mu) for fields of shape (Lt, Lz, Ly, Lx, ...)."""
    return torch.roll(a, -1, 3 - mu)


def _links(dims, scale, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    shape = (dims[3], dims[2], dims[1], dims[0])
    V = int(np.prod(dims))
    U = _random_su3(4 * V, scale, gen).reshape(shape + (4, 3, 3))
    g = _random_su3(V, 1.0, gen).reshape(shape + (3, 3))
    for mu in range(4):
        U[..., mu, :, :] = _mm(_mm(g, U[..., mu, :, :]), _roll_fwd(g, mu).mH)
    return U


def _mixed(dtype):
    return dtype.startswith("f32")


def _handle(dims, dtype, exp_order=1):
    gf = lgf.GaugeFixer(dims, dtype, alpha=ALPHA)
    if exp_order != 1:
        gf.set_param(_lib.LGF_EXP_ORDER, exp_order)
    return gf


def _pinned(shape):
    return torch.empty(shape, dtype=torch.complex128, pin_memory=True)


def _network(seed):
    """A network as it is after some training: weights of its usual size,
    the last layer no longer near zero."""
    net = lgf.WarmStartNet(seed=seed)
    rng = np.random.default_rng(seed)
    p = net.get_params()
    n3 = 81 * 32 * 8 + 8
    p[-n3:] = (0.004 * rng.standard_normal(n3)).astype(np.float32)
    net.set_params(p)
    return net, p


_WIDTHS = {1: (48, 32), 2: (32, 32), 3: (32, 16)}


def _conv_inputs(case, seed):
    dims = _parse(case["dims"])
    V = int(np.prod(dims))
    k, n = _WIDTHS[case["layer"]]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if not case["backward"]:
        x = torch.randn((V, k), device="cuda", generator=gen)
        if case["layer"] > 1:
            x = torch.relu(x)
        else:
            x[:, 38:] = 0  # features: 32 link coefficients, 6 plaquettes, padding
        return x.to(torch.bfloat16), None
    x = torch.randn((V, n), device="cuda", generator=gen)
    if case["layer"] == 3:
        x[:, 8:] = 0
    mask = torch.relu(torch.randn((V, k), device="cuda", generator=gen))
    return x.to(torch.bfloat16), mask.to(torch.bfloat16)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "fix":
        dims = _parse(case["dims"])
        gf = _handle(dims, case["dtype"], case["exp_order"])
        field = (3, 3) if _mixed(case["dtype"]) else (4, 3, 3)
        return {"case": case, "gf": gf, "U": _links(dims, case["scale"], seed), "out": _pinned(gf.shape + field)}
    if kind == "batch":
        members = _members(case)
        fixers = [_handle(d, case["dtype"]) for d in members]
        return {"case": case, "fixers": fixers, "batch": lgf.GaugeBatch(fixers),
                "U": [_links(d, case["scale"], 1000 * seed + i) for i, d in enumerate(members)],
                "out": [_pinned(gf.shape + (3, 3)) for gf in fixers]}
    net, _ = _network(seed)
    if kind == "conv":
        x, mask = _conv_inputs(case, seed)
        return {"case": case, "net": net, "x": x, "mask": mask, "dims": _parse(case["dims"])}
    gf = _handle(_parse(case["dims"]), "f32")
    return {"case": case, "net": net, "gf": gf, "U": _links(_parse(case["dims"]), case["scale"], seed)}


def _gauge_to_gpu(gf, pinned):
    """The applied gauge transformation as single-precision device tensor."""
    gf.store_gauge(pinned.numpy())
    return pinned.to("cuda", non_blocking=True).to(torch.complex64)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "fix":
        gf = state["gf"]
        gf.load_links(state["U"])
        _, converged = gf.fix(case["tol"], MAX_ITER)
        if not converged:
            raise RuntimeError("not converged")
        F, _ = gf.functional()
        if _mixed(case["dtype"]):
            return {"F": F, "G": _gauge_to_gpu(gf, state["out"])}
        return {"F": F, "U": gf.store_links(state["out"].numpy())}
    if kind == "batch":
        for gf, U in zip(state["fixers"], state["U"]):
            gf.load_links(U)
        _, converged = state["batch"].fix(case["tol"], MAX_ITER)
        if not all(converged):
            raise RuntimeError("not converged")
        return {"G": [_gauge_to_gpu(gf, out) for gf, out in zip(state["fixers"], state["out"])]}
    if kind == "conv":
        return {"y": state["net"].conv(case["layer"], case["backward"], state["x"], state["dims"], state["mask"])}
    state["gf"].load_links(state["U"])
    F, grad = state["net"].train_step(state["gf"], LEARNING_RATE, want_grad=True)
    return {"F": F, "grad": grad}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _fix_work(dims, dtype, tol, exp_order=1):
    """Input links in and the result out once.  Flops per site and update: the
    gradient's and the update's SU(3) products (8 of 216 flops), the forward
    and inverse line transforms of four complex fields at 5 log2 L flops per
    point, and the projection."""
    V = float(np.prod(dims))
    fft = sum(2 * 4 * 5 * math.log2(L) for L in dims)
    step = 8 * 216 + fft + 300 + (0 if exp_order == 1 else 2 * 216)
    return V * (576 + (144 if _mixed(dtype) else 576)), V * UPDATES[tol] * step


def work(case):
    kind = case["kind"]
    if kind == "fix":
        b, f = _fix_work(_parse(case["dims"]), case["dtype"], case["tol"], case["exp_order"])
        return {"bytes": b, "flops": f}
    if kind == "batch":
        w = [_fix_work(d, case["dtype"], case["tol"]) for d in _members(case)]
        return {"bytes": sum(x[0] for x in w), "flops": sum(x[1] for x in w)}
    V = float(np.prod(_parse(case["dims"])))
    if kind == "conv":
        k, n = _WIDTHS[case["layer"]]
        mask = 2 * V * k if case["backward"] else 0
        return {"bytes": 2 * V * (k + n) + mask + 2 * 81 * k * n, "flops": 2 * 81 * k * n * V}
    # forward, and both gradients of each layer but the first layer's input
    macs = 81 * (48 * 32 + 32 * 32 + 32 * 8)
    return {"bytes": V * 576 + V * 288, "flops": V * 2 * (2 * macs + 81 * (32 * 32 + 32 * 8))}


# ---------------------------------------------------------------------------
# the same results in 64 bits
# ---------------------------------------------------------------------------
def _delta(U):
    A = torch.zeros_like(U[..., 0, :, :])
    for mu in range(4):
        u = U[..., mu, :, :]
        A += torch.roll(u, 1, 3 - mu) - u
    D = A - A.mH
    tr = torch.diagonal(D, dim1=-2, dim2=-1).sum(-1) / 3
    return D - tr[..., None, None] * torch.eye(3, dtype=D.dtype, device=D.device)


def _expm(X):
    """exp of anti-Hermitian 3x3 matrices: Taylor series of X / 8, squared
    three times (|X| stays below about 5 here)."""
    X = X / 8
    eye = torch.eye(3, dtype=X.dtype, device=X.device)
    E = eye + X / 18
    for k in range(17, 0, -1):
        E = eye + _mm(X, E) / k
    for _ in range(3):
        E = _mm(E, E)
    return E


def _acceleration(dims):
    p2 = 0
    for a, L in enumerate(dims):
        s = 4 * torch.sin(math.pi * torch.arange(L, dtype=torch.float64, device="cuda") / L) ** 2
        p2 = p2 + s.reshape([L if i == 3 - a else 1 for i in range(4)])
    k = p2.max() / torch.where(p2 > 0, p2, 1.0)
    k[0, 0, 0, 0] = 0
    return k[..., None, None]


def _functional(U):
    return float(torch.diagonal(U, dim1=-2, dim2=-1).real.sum() / (12 * U[..., 0, 0, 0].numel()))


def _exact_fix(dims, U, tol, exp_order):
    K = _acceleration(dims)
    eye = torch.eye(3, dtype=U.dtype, device=U.device)
    G = eye.expand(U.shape[:4] + (3, 3)).contiguous()
    V = float(np.prod(dims))
    for _ in range(MAX_ITER):
        D = _delta(U)
        if float((D.real ** 2 + D.imag ** 2).sum()) / (3 * V) < tol:
            break
        X = 0.5 * ALPHA * torch.fft.ifftn(K * torch.fft.fftn(D, dim=(0, 1, 2, 3)), dim=(0, 1, 2, 3))
        g = _reunit(eye + X if exp_order == 1 else _expm(X))
        for mu in range(4):
            U[..., mu, :, :] = _mm(_mm(g, U[..., mu, :, :]), _roll_fwd(g, mu).mH)
        G = _reunit(_mm(g, G))
    return _functional(U), U, G


def _taps():
    return [(t // 27 - 1, (t // 9) % 3 - 1, (t // 3) % 3 - 1, t % 3 - 1) for t in range(81)]


def _conv64(x, W, b):
    """x (Lt, Lz, Ly, Lx, in), W (81, in, out)."""
    y = torch.zeros(x.shape[:4] + (W.shape[2],), dtype=x.dtype, device=x.device) + b
    for W_t, off in zip(W, _taps()):
        y += torch.roll(x, [-o for o in off], (0, 1, 2, 3)) @ W_t
    return y


def _conv64_bwd(x, W, gy):
    gx = torch.zeros_like(x)
    gW = torch.empty_like(W)
    for t, off in enumerate(_taps()):
        gW[t] = torch.roll(x, [-o for o in off], (0, 1, 2, 3)).reshape(-1, W.shape[1]).T @ gy.reshape(-1, W.shape[2])
        gx += torch.roll(gy @ W[t].T, off, (0, 1, 2, 3))
    return gx, gW, gy.reshape(-1, W.shape[2]).sum(0)


def _layers(p):
    p = torch.from_numpy(p.astype(np.float64)).cuda()
    out, o = [], 0
    for k, n in ((48, 32), (32, 32), (32, 8)):
        out.append((p[o:o + 81 * k * n].reshape(81, k, n), p[o + 81 * k * n:o + 81 * k * n + n]))
        o += 81 * k * n + n
    return out


def _coefficients(A):
    """c_a with sum_a c_a i lambda_a / 2 = A, A traceless anti-Hermitian."""
    return (-1j * torch.einsum("aij,...ji->...a", _gell_mann("cuda"), A)).real


def _features(U):
    A = 0.5 * (U - U.mH)
    tr = torch.diagonal(A, dim1=-2, dim2=-1).sum(-1) / 3
    A = A - tr[..., None, None] * torch.eye(3, dtype=A.dtype, device=A.device)
    f = torch.zeros(U.shape[:4] + (48,), dtype=torch.float64, device="cuda")
    f[..., :32] = _coefficients(A).reshape(U.shape[:4] + (32,))
    k = 32
    for mu in range(4):
        for nu in range(mu + 1, 4):
            u, v = U[..., mu, :, :], U[..., nu, :, :]
            P = _mm(_mm(u, _roll_fwd(v, mu)), _mm(v, _roll_fwd(u, nu)).mH)
            f[..., k] = torch.diagonal(P, dim1=-2, dim2=-1).sum(-1).real / 3
            k += 1
    return f


def _exact_conv(case, seed):
    x, mask = _conv_inputs(case, seed)
    dims = _parse(case["dims"])
    shape = (dims[3], dims[2], dims[1], dims[0])
    net, p = _network(seed)
    net.close()
    W, b = _layers(p)[case["layer"] - 1]
    W = W.to(torch.bfloat16).double()
    x = x.double().reshape(shape + (-1,))
    if not case["backward"]:
        y = _conv64(x, W, b)
        y = torch.relu(y) if case["layer"] < 3 else torch.nn.functional.pad(y, (0, 8))
    else:
        y = torch.zeros(shape + (W.shape[1],), dtype=torch.float64, device="cuda")
        for W_t, off in zip(W, _taps()):
            y += torch.roll(x[..., :W.shape[2]] @ W_t.T, off, (0, 1, 2, 3))
        y = torch.where(mask.reshape(y.shape) > 0, y, 0.0)
    return {"y": y.reshape(-1, y.shape[-1])}


def _exact_train(case, seed):
    dims = _parse(case["dims"])
    U = _links(dims, case["scale"], seed)
    net, p = _network(seed)
    net.close()
    (W1, b1), (W2, b2), (W3, b3) = _layers(p)
    x = _features(U)
    z1 = _conv64(x, W1, b1)
    a1 = torch.relu(z1)
    z2 = _conv64(a1, W2, b2)
    a2 = torch.relu(z2)
    c = _conv64(a2, W3, b3)
    g0 = _expm(0.5j * torch.einsum("...a,aij->...ij", c.to(torch.complex128), _gell_mann("cuda")))
    for mu in range(4):
        U[..., mu, :, :] = _mm(_mm(g0, U[..., mu, :, :]), _roll_fwd(g0, mu).mH)
    F = _functional(U)
    # dL/dc_a = -<i lambda_a / 2, Delta> / (24 V), half the coefficients of Delta
    gc = -0.5 * _coefficients(_delta(U)) / (24 * float(np.prod(dims)))
    ga2, gW3, gb3 = _conv64_bwd(a2, W3, gc)
    gz2 = torch.where(z2 > 0, ga2, 0.0)
    ga1, gW2, gb2 = _conv64_bwd(a1, W2, gz2)
    gz1 = torch.where(z1 > 0, ga1, 0.0)
    _, gW1, gb1 = _conv64_bwd(x, W1, gz1)
    grad = torch.cat([t.reshape(-1) for t in (gW1, gb1, gW2, gb2, gW3, gb3)])
    return {"F": F, "grad": grad.cpu().numpy()}


def exact(case, seed):
    kind = case["kind"]
    if kind == "conv":
        return _exact_conv(case, seed)
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "batch":
        members = _members(case)
        if sum(float(np.prod(d)) for d in members) > 6e6:
            return None
        return {"G": [_exact_fix(d, _links(d, case["scale"], 1000 * seed + i), case["tol"], 1)[2]
                      for i, d in enumerate(members)]}
    dims = _parse(case["dims"])
    F, U, G = _exact_fix(dims, _links(dims, case["scale"], seed), case["tol"], case["exp_order"])
    return {"F": F, "G": G} if _mixed(case["dtype"]) else {"F": F, "U": U}

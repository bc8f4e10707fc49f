"""The work that users of this package have it do, as timed cases.

Every case calls the public entry points on arrays already on the GPU, as a
program does that keeps its handle, network and output buffers:

  forward     intensities of a known matrix (tmr_forward): checking a result,
              making synthetic data
  grad        loss and gradient of all rows (tmr_grad): a caller's own optimiser
  track       retrieval that starts from the matrix measured before
              (tmr_retrieve_from): a fiber that drifted since, or a resumed run
  spectral    retrieval from intensities alone, 16 Lanczos steps and a fixed
              number of L-BFGS iterations (tmr_retrieve)
  fit         the rows' phase offsets from defocus images (tmr_defocus_fit),
              near those of the last fit, with the same-grid operator or the angular-spectrum one
  preprocess  camera frames to rows (tmr_preprocess)
  mlp_train   one step of the learned initialiser's training at its batch size,
              and the weights after it
  mlp_forward the network's proposals for a chunk of rows

Sizes are those of the paper's workloads as this repository runs them (64 to
4096 modes, 64 to 20000 pixels, 1 to 8 masks, 1e3 to 1e5 photons per pixel).
Retrieval cases use data that every row of the problem can be recovered from
(six or more masks, or a start near the solution): rows that are not
recoverable end wherever rounding leads them and would compare with nothing.
Inputs come from torch alone, so that they do not depend on the library.
"""
import math

import torch

import paper_2302_13524_gb300 as tmr

DEV = "cuda"
C128, F64 = torch.complex128, torch.float64
GEOM = dict(wavelength=0.532, na=0.22, z_d=20.0, pixel=0.9)  # the angular-spectrum operator, in micrometres
LR = 3e-4


def listed():
    return [
        # the smallest problem of the repository's configurations: launch latency
        dict(name="forward_64", op="forward", N=64, M=128, J=4),
        # the largest transform and matrix: 1 GB of intensities written
        dict(name="forward_4096", op="forward", N=4096, M=16384, J=4),
        # the paper-scale workload's matrix
        dict(name="grad_2048", op="grad", N=2048, M=8192, J=4, cost="intensity"),
        # a length that is no power of two (the paper's own matrix is 2286 wide)
        dict(name="grad_2286", op="grad", N=2286, M=8192, J=4, cost="intensity"),
        # the paper-scale retrieval, re-run on a fiber that drifted
        dict(name="track_2048", op="track", N=2048, M=8192, J=4, iters=20, drift=0.3, photons=1e4, tol=0.0, graph=True),
        # retrieval from scratch with more masks
        dict(name="spectral_1024", op="spectral", N=1024, M=4096, J=8, iters=20, rank=550, photons=1e4),
        # uneven noise and early exit per row, length 2286
        dict(name="batch_2286", op="track", N=2286, M=2048, J=4, iters=300, drift=0.3, photons=1e4, tol=1e-6, graph=True),
        # the largest transform, a cluster of CTAs per row
        dict(name="track_4096", op="track", N=4096, M=4096, J=4, iters=20, drift=0.3, photons=1e4, tol=0.0, graph=False),
        # the paper-scale defocus fit
        dict(name="fit_128x64", op="fit", kind=0, N=2048, ny=128, nx=64, J=4, Nd=50),
        # the camera workload's frames
        dict(name="preprocess_8192", op="preprocess", K=8192, H=256, W=128, pix="u16"),
        # the learned initialiser at the paper-scale workload: training and proposals
        dict(name="mlp_train_256", op="mlp_train", n_in=8192, h1=1024, h2=1024, n_out=4096, B=256),
        dict(name="mlp_forward_2048", op="mlp_forward", n_in=8192, h1=1024, h2=1024, n_out=4096, B=2048),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["forward", "grad", "grad", "track", "track", "spectral", "fit", "preprocess", "mlp_train", "mlp_forward"])
    pow2 = rng.random() < 0.6
    if op in ("forward", "grad"):
        N = 2 ** rng.randint(6, 12) if pow2 else _log(rng, 64, 4000)
        J = rng.randint(1, 8)
        most = 2 ** 27 if op == "forward" and pow2 else 2 ** 25  # intensities of one pass
        c = dict(op=op, N=N, M=_log(rng, 100, min(20000, most // (J * N))), J=J)
        return dict(c, cost=rng.choice(["intensity", "intensity", "amplitude"])) if op == "grad" else c
    if op in ("track", "spectral"):
        J = rng.choice([4, 6, 8]) if op == "track" else rng.choice([6, 8])
        N = 2 ** rng.randint(8, 12) if pow2 else _log(rng, 200, 2300)
        iters = rng.randint(5, 40)
        most = (2 ** 29 if pow2 else 2 ** 27) // (J * N * (iters + 16))
        c = dict(op=op, N=N, M=_log(rng, 64, max(128, min(8192, most))), J=J, iters=iters, photons=float(_log(rng, 1000, 100000)))
        if op == "spectral":
            return dict(c, rank=N // 2 + rng.randint(0, 64))
        return dict(c, drift=round(rng.uniform(0.05, 0.3), 3), tol=0.0, graph=rng.random() < 0.5)
    if op == "fit":
        kind = rng.randint(0, 1)
        ny, nx = rng.choice([(32, 32), (64, 32), (64, 64), (128, 64)])
        return dict(op=op, kind=kind, N=2 ** rng.randint(7, 11), ny=ny, nx=nx, J=4, Nd=rng.randint(20, 50))
    if op == "preprocess":
        # odd sides too: the half grid drops the last row or column
        H, W = _log(rng, 40, 256), _log(rng, 40, 256)
        return dict(op=op, K=min(8192, _log(rng, 100, 2 ** 28 // (H * W))), H=H, W=W, pix=rng.choice(["u16", "u16", "f32"]))
    n = 2 ** rng.randint(8, 11)  # modes; 4 masks
    h1, h2 = 64 * rng.randint(2, 16), 64 * rng.randint(2, 16)
    B = _log(rng, 64, 512) if op == "mlp_train" else _log(rng, 64, 2048)
    return dict(op=op, n_in=4 * n, h1=h1, h2=h2, n_out=2 * n, B=B)


# ---- inputs ---------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _cnormal(g, *shape):
    return torch.view_as_complex(torch.randn(*shape, 2, generator=g, device=DEV) * math.sqrt(0.5))


def _phases(g, *shape):
    return torch.polar(torch.ones(shape, device=DEV), 2 * math.pi * torch.rand(shape, generator=g, device=DEV))


def _intensities(T, masks, g, photons):
    """|F(d_j .* t)|^2 of every row and mask with shot noise, in blocks of rows."""
    M, (J, N) = T.shape[0], masks.shape
    Y = torch.empty((M, J, N), device=DEV)
    step = max(1, 2 ** 24 // (J * N))
    for r in range(0, M, step):
        z = torch.fft.fft(masks * T[r:r + step, None])
        Y[r:r + step] = z.real.square() + z.imag.square()
    if photons:
        s = photons / float(Y.mean())
        for r in range(0, M, step):
            Y[r:r + step] = torch.poisson(Y[r:r + step] * s, generator=g) / s
    return Y


def _signed(n, dtype=torch.int64):
    k = torch.arange(n, device=DEV)
    return torch.where(2 * k < n, k, k - n).to(dtype)


def _transfer(c):
    """The operator's transfer function on the pixel grid's frequencies, 64 bits."""
    ny, nx = c["ny"], c["nx"]
    ky, kx = _signed(ny, F64)[:, None], _signed(nx, F64)[None, :]
    if c["kind"] == 0:
        return torch.polar(torch.ones((ny, nx), dtype=F64, device=DEV), -0.05 * (ky ** 2 + kx ** 2))
    lam, ps = GEOM["wavelength"], GEOM["pixel"]
    rho2 = (lam * kx / (nx * ps)) ** 2 + (lam * ky / (ny * ps)) ** 2
    arg = 2 * math.pi / lam * (1 - rho2).clamp(min=0).sqrt() * GEOM["z_d"]
    return torch.polar((rho2.sqrt() <= GEOM["na"]).to(F64), arg)


def _image_field(c, x, h):
    """The defocus-plane fields of the fields x [..., ny, nx]."""
    X = torch.fft.fft2(x) * h
    if c["kind"] == 0:
        return torch.fft.ifft2(X)
    ny, nx = c["ny"], c["nx"]
    pad = torch.zeros(X.shape[:-2] + (2 * ny, 2 * nx), dtype=X.dtype, device=DEV)
    pad[..., (_signed(ny) % (2 * ny))[:, None], (_signed(nx) % (2 * nx))[None, :]] = X
    return torch.fft.ifft2(pad) * 4


def _fields(c, T, masks, incident):
    """The fields c_n on the pixel grid, [Nd, ny, nx]."""
    Z = T @ incident.T if c["kind"] else torch.fft.fft(masks[0] * T)[:, :c["Nd"]]
    return Z.T.reshape(c["Nd"], c["ny"], c["nx"]).contiguous()


def _options(c):
    o = dict(init="spectral", power_iters=16, lanczos=1)
    if c["op"] == "track":
        o.update(tol=c["tol"], use_graph=int(c["graph"]))
    if c["op"] == "grad":
        o.update(cost=c["cost"])
    if c["op"] == "fit":
        o.update(phase_iters=100, phase_tol=1e-4)
    return o


def _empty(shape, dtype=torch.float32):
    return torch.empty(shape, dtype=dtype, device=DEV)


def _inputs(c, seed):
    """The arrays that a pass reads, made from the seed alone."""
    g, op = _gen(seed), c["op"]
    if op == "preprocess":
        K, H, W = c["K"], c["H"], c["W"]
        yy, xx = torch.arange(H, device=DEV)[:, None], torch.arange(W, device=DEV)[None, :]
        core = ((yy - H / 2 + 0.5) / (0.45 * H)) ** 2 + ((xx - W / 2 + 0.5) / (0.45 * W)) ** 2 <= 1
        frames = _empty((K, H, W), torch.int16 if c["pix"] == "u16" else torch.float32)
        for k in range(0, K, 512):
            n = min(512, K - k)
            lam = _empty((n, H, W)).exponential_(1 / 2000.0, generator=g) * core + 2.0
            counts = torch.poisson(lam, generator=g).clamp(max=65535)
            frames[k:k + n] = counts.to(torch.int32).to(torch.int16) if c["pix"] == "u16" else counts
        return dict(frames=frames)
    if op.startswith("mlp"):
        dims = [c["n_in"], c["h1"], c["h2"], c["n_out"]]
        params = torch.cat([p for a, b in zip(dims, dims[1:]) for p in (
            (torch.rand(b * a, generator=g, device=DEV) * 2 - 1) * math.sqrt(3 / a), torch.zeros(b, device=DEV))])
        X = _empty((c["B"], c["n_in"])).exponential_(1.0, generator=g)  # speckle intensities
        X = (X / X.mean(1, keepdim=True)).sqrt()
        T = torch.randn(c["B"], c["n_out"], generator=g, device=DEV)
        return dict(params=params, X=X, T=T)
    N, J = c["N"], c["J"]
    M = c["ny"] * c["nx"] if op == "fit" else c["M"]
    masks = _phases(g, J, N)
    if op == "spectral":  # the mode model: every row in one subspace of the inputs
        T = (_cnormal(g, M, c["rank"]) @ _cnormal(g, c["rank"], N)) * math.sqrt(1 / (c["rank"] * N))
    else:
        T = _cnormal(g, M, N) * math.sqrt(1 / N)
    if op == "forward":
        return dict(masks=masks, T=T)
    if op == "grad":  # a matrix part of the way to the one that was measured
        return dict(masks=masks, T=T + 0.2 * _cnormal(g, M, N) * math.sqrt(1 / N), Y=_intensities(T, masks, g, 1e4))
    if op == "track":
        T0 = T + c["drift"] * _cnormal(g, M, N) * math.sqrt(1 / N)
        if c["tol"] > 0:  # photon levels over two decades, log-uniform
            Y = _intensities(T, masks, g, None)
            s = 10 ** (3 + 2 * torch.rand(M, 1, 1, generator=g, device=DEV)) / float(Y.mean())
            return dict(masks=masks, T0=T0, Y=torch.poisson(Y.mul_(s), generator=g).div_(s))
        return dict(masks=masks, T0=T0, Y=_intensities(T, masks, g, c["photons"]))
    if op == "spectral":
        return dict(masks=masks, Y=_intensities(T, masks, g, c["photons"]))
    incident = _phases(g, c["Nd"], N) if c["kind"] else None
    w = _image_field(c, _fields(c, T, masks, incident), _transfer(c).to(T.dtype))
    I = w.real.square() + w.imag.square()
    s = 1e4 / float(I.mean())
    I = (torch.poisson(I * s, generator=g) / s).reshape(c["Nd"], -1).contiguous()
    off = 0.5 * torch.randn(M, 1, generator=g, device=DEV)  # the rows' phases moved since the last fit
    return dict(masks=masks, incident=incident, T=T * torch.polar(torch.ones_like(off), off), I=I)


def prepare(case, seed):
    c, op = case, case["op"]
    s = dict(_inputs(c, seed), case=c)
    if op == "preprocess":
        ny, nx = tmr.half_grid(c["H"], c["W"])
        s["wb"] = tmr.tmr_preprocess_workspace_bytes(c["K"], c["H"], c["W"])
        s.update(y=_empty((ny * nx, c["K"])), mask=_empty(ny * nx, torch.uint8), energy=_empty(ny * nx, F64),
                 n_inside=_empty(1, torch.int32), ws=_empty(max(s["wb"], 1), torch.uint8))
    elif op.startswith("mlp"):
        s["net"] = tmr.tmr_mlp_create(c["n_in"], c["h1"], c["h2"], c["n_out"])
        tmr.tmr_mlp_set_loss(s["net"], "phase")
        tmr.tmr_mlp_set_params(s["net"], s["params"])
        s.update(loss=_empty(1), out=torch.empty_like(s["params"]), Yn=_empty((c["B"], c["n_out"])))
    else:
        M, dop = c.get("M"), None
        if op == "fit":
            M = c["ny"] * c["nx"]
            dop = dict(kind=c["kind"], ny=c["ny"], nx=c["nx"], n_defocus=c["Nd"], coef=0.05)
            if c["kind"]:
                dop.update(GEOM, incident=s["incident"])
        s["h"] = tmr.tmr_create(c["N"], M, c["J"], s["masks"], dop, _options(c))
        if op == "forward":
            s["Yo"] = _empty((M, c["J"], c["N"]))
        else:
            s.update(To=_empty((M, c["N"]), torch.complex64), status=_empty(M, torch.int32), iters=_empty(M, torch.int32),
                     loss=_empty(M))
    return s


def run(state):
    s, c = state, state["case"]
    op = c["op"]
    if op == "forward":
        tmr.tmr_forward(s["h"], s["T"], s["Yo"])
        return s["Yo"]
    if op == "grad":
        tmr.tmr_grad(s["h"], s["T"], s["Y"], s["loss"], s["To"])
        return dict(loss=s["loss"], G=s["To"])
    if op == "track":
        if c["tol"] > 0:  # the iteration a row stops at hangs on its loss's last bits: not asked for
            tmr.tmr_retrieve_from(s["h"], s["T0"], s["Y"], None, c["iters"], s["To"], s["status"], None, s["loss"])
            return dict(T=s["To"], loss=s["loss"], status=s["status"])
        tmr.tmr_retrieve_from(s["h"], s["T0"], s["Y"], None, c["iters"], s["To"], s["status"], s["iters"], s["loss"])
        return dict(T=s["To"], loss=s["loss"], status=s["status"], iters=s["iters"])
    if op == "spectral":
        tmr.tmr_retrieve(s["h"], s["Y"], None, c["iters"], s["To"], s["status"], s["iters"], s["loss"])
        return dict(T=s["To"], loss=s["loss"], status=s["status"], iters=s["iters"])
    if op == "fit":
        tmr.tmr_defocus_fit(s["h"], s["T"], s["I"], None, s["To"])
        return s["To"]
    if op == "preprocess":
        tmr.tmr_preprocess(s["frames"], c["K"], c["H"], c["W"], 0, 0.999, s["y"], s["mask"], s["energy"], s["n_inside"],
                           s["ws"], s["wb"])
        return dict(y=s["y"], mask=s["mask"], energy=s["energy"], n_inside=s["n_inside"])
    if op == "mlp_train":
        tmr.tmr_mlp_train_step(s["net"], s["X"], s["T"], c["B"], LR, s["loss"])
        tmr.tmr_mlp_get_params(s["net"], s["out"])
        return dict(loss=s["loss"], params=s["out"])
    tmr.tmr_mlp_forward(s["net"], s["X"], c["B"], s["Yn"])
    return s["Yn"]


def work(case):
    """Bytes: every input read and output written once.  Operations: the
    transforms at 5 N log2 N each (whatever the length), the products of the
    network, and the vector work beside them."""
    c, op = case, case["op"]
    if op == "preprocess":
        ny, nx = tmr.half_grid(c["H"], c["W"])
        M = ny * nx
        return dict(bytes=M * c["K"] * ((2 if c["pix"] == "u16" else 4) + 4) + 9 * M, flops=M * c["K"])
    if op.startswith("mlp"):
        w = c["n_in"] * c["h1"] + c["h1"] * c["h2"] + c["h2"] * c["n_out"]
        p = w + c["h1"] + c["h2"] + c["n_out"]
        if op == "mlp_forward":
            return dict(bytes=4 * (c["B"] * (c["n_in"] + c["n_out"]) + p), flops=2 * c["B"] * w)
        return dict(bytes=4 * (c["B"] * (c["n_in"] + c["n_out"]) + 7 * p), flops=6 * c["B"] * w + 12 * p)
    N, J = c["N"], c["J"]
    fft = 5 * N * math.log2(N)
    if op == "fit":
        P = c["ny"] * c["nx"]
        img = c["Nd"] * P
        return dict(bytes=16 * P * N + 4 * img * (4 if c["kind"] else 1),
                    flops=20 * img * math.log2(P) * (5 if c["kind"] else 2) * 20 + (8 * N * img if c["kind"] else P * fft))
    M = c["M"]
    if op == "forward":
        return dict(bytes=M * (8 * N + 4 * J * N), flops=M * J * (fft + 9 * N))
    if op == "grad":
        return dict(bytes=M * (16 * N + 4 * J * N), flops=M * J * (2 * fft + 20 * N))
    iters = c["iters"] if not c.get("tol") else 25
    products = iters + (16 if op == "spectral" else 1)
    return dict(bytes=M * ((16 if op == "track" else 8) * N + 4 * J * N), flops=M * (products * J * (2 * fft + 40 * N) + iters * 110 * N))


# ---- the same in 64 bits ----------------------------------------------------------
def _coef(cost, z, y):
    """(c, loss) of the row cost at the fields z: u = c z and g = scale Q^H u."""
    if cost == "amplitude":
        a, m = y.clamp(min=0).sqrt(), z.abs()
        return torch.where(m > 0, (m - a) / m, 0.0), (a - m).square().sum((1, 2))
    r = y - z.real.square() - z.imag.square()
    return r, r.square().sum((1, 2))


def _adjoint(u, d):
    return (torch.fft.ifft(u, norm="forward") * d.conj()).sum(1)


def _grad64(T, Y, d, cost):
    z = torch.fft.fft(d * T[:, None])
    r, f = _coef(cost, z, Y)
    return f, (2.0 if cost == "amplitude" else -4.0) * _adjoint(z * r, d), z


def _step64(q1, q2, q3, q4):
    """The global minimiser of q1 a + q2 a^2 + q3 a^3 + q4 a^4, q4 > 0."""
    b, c, d = 0.75 * q3 / q4, 0.5 * q2 / q4, 0.25 * q1 / q4
    p, q = c - b * b / 3, 2 * b ** 3 / 27 - b * c / 3 + d
    disc = (q / 2) ** 2 + (p / 3) ** 3
    u = -q / 2 - torch.copysign(disc.clamp(min=0).sqrt(), q)
    u = torch.copysign(u.abs() ** (1 / 3), u)
    r = (-p / 3).clamp(min=0).sqrt()
    th = torch.acos((-q / 2 / r ** 3).clamp(-1, 1).nan_to_num()) / 3
    roots = [torch.where(disc > 0, u - p / (3 * u), 2 * r * torch.cos(th - k * 2 * math.pi / 3)) - b / 3 for k in range(3)]
    a = torch.stack(roots)
    for _ in range(3):
        a = a - (((4 * q4 * a + 3 * q3) * a + 2 * q2) * a + q1) / ((12 * q4 * a + 6 * q3) * a + 2 * q2)
    phi = (((q4 * a + q3) * a + q2) * a + q1) * a
    return a.gather(0, phi.argmin(0, keepdim=True))[0]


def _dot(a, b):
    return (a.conj() * b).real.sum(1)


def _direction(g, pairs):
    """-H g by the two-loop recursion over (s, y, s.y)."""
    q, al = g.clone(), []
    for s, y, sy in reversed(pairs):
        al.append(_dot(s, q) / sy)
        q -= al[-1][:, None] * y
    if pairs:
        s, y, sy = pairs[-1]
        q *= (sy / _dot(y, y))[:, None]
    for (s, y, sy), a in zip(pairs, reversed(al)):
        q += (a - _dot(y, q) / sy)[:, None] * s
    return -q


def _lbfgs64(T, Y, d, iters, tol):
    T, Y = T.clone(), Y.to(F64)
    f, g, z = _grad64(T, Y, d, "intensity")
    loss, live, pairs = f.clone(), torch.ones_like(f, dtype=torch.bool), []
    out = T.clone()
    for _ in range(iters):
        p = _direction(g, pairs)
        w = torch.fft.fft(d * p[:, None])
        r, a, b = Y - z.real.square() - z.imag.square(), (z.conj() * w).real, w.real.square() + w.imag.square()
        al = _step64(-4 * (r * a).sum((1, 2)), (4 * a * a - 2 * r * b).sum((1, 2)), 4 * (a * b).sum((1, 2)), (b * b).sum((1, 2)))
        T = T + al[:, None] * p
        fn, gn, z = _grad64(T, Y, d, "intensity")
        y = gn - g
        pairs = (pairs + [(al[:, None] * p, y, _dot(al[:, None] * p, y))])[-5:]
        out[live], loss[live] = T[live], fn[live]
        if tol > 0:
            live &= (f - fn).abs() / f >= tol
            if not live.any():
                break
        f, g = fn, gn
    return out, loss, torch.where(live, 0, 1).to(torch.int32)


def _philox(rows, N):
    """The documented random start: Philox4x32-10 of counter (n, row, 0, 0), key 0, and Box-Muller."""
    c = [torch.arange(N, device=DEV)[None, :].expand(len(rows), N), rows[:, None].expand(len(rows), N)]
    c += [torch.zeros_like(c[0])] * 2
    k0 = k1 = 0
    mask = 0xFFFFFFFF

    def mul(x, m):  # high and low words, in 63-bit integers
        lo, hi = (x & 0xFFFF) * m, (x >> 16) * m
        t = hi + (lo >> 16)
        return t >> 16, ((t & 0xFFFF) << 16) | (lo & 0xFFFF)

    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
        (h0, l0), (h1, l1) = mul(c[0], 0xD2511F53), mul(c[2], 0xCD9E8D57)
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
    u0, u1 = ((x.to(F64) + 0.5) / 2 ** 32 for x in c[:2])
    return torch.polar((-2 * u0.log()).sqrt(), 2 * math.pi * u1)


def _spectral64(rows, Y, d, k=16, clip=2.0):
    """The leading eigenvector of Q^H diag(min(y / mean, 2)) Q / (J N) by k Lanczos steps, at the rows' norms."""
    Y = Y.to(F64)
    J, N = d.shape
    tau = (Y / Y.mean((1, 2), keepdim=True)).clamp(max=clip)
    v = _philox(rows, N)
    V, alpha, beta = [v / v.norm(dim=1, keepdim=True)], [], []
    for j in range(k):
        w = _adjoint(torch.fft.fft(d * V[j][:, None]) * tau, d) / (J * N)
        a = 0
        for _ in range(2):
            B = torch.stack(V, 1)
            h = torch.einsum("rln,rn->rl", B.conj(), w)
            w = w - torch.einsum("rl,rln->rn", h, B)
            a = a + h[:, j].real
        alpha.append(a)
        beta.append(w.norm(dim=1))
        V.append(w / beta[-1][:, None])
    t3 = torch.diag_embed(torch.stack(alpha, 1)) + torch.diag_embed(torch.stack(beta[:-1], 1), 1) + torch.diag_embed(torch.stack(beta[:-1], 1), -1)
    s = torch.linalg.eigh(t3.cpu())[1][:, :, -1].to(DEV)
    s = s * torch.where(s[:, :1] < 0, -1.0, 1.0)
    t = torch.einsum("rl,rln->rn", s.to(C128), torch.stack(V[:k], 1))
    return t / t.norm(dim=1, keepdim=True) * (Y.sum((1, 2)) / (J * N)).sqrt()[:, None]


def _fit64(c, T, masks, incident, I, iters=100, tol=1e-4, m=5):
    cn, h = _fields(c, T, masks, incident), _transfer(c)
    I = I.to(F64).reshape((c["Nd"],) + ((2 * c["ny"], 2 * c["nx"]) if c["kind"] else (c["ny"], c["nx"])))

    def f_and_g(phi):
        ph = phi.reshape(c["ny"], c["nx"]).clone().requires_grad_(True)
        w = _image_field(c, cn * torch.polar(torch.ones_like(ph), ph), h)
        f = (I - w.real.square() - w.imag.square()).square().sum()
        return float(f.detach()), torch.autograd.grad(f, ph)[0].reshape(1, -1)

    phi = torch.zeros((1, T.shape[0]), dtype=F64, device=DEV)
    f, g = f_and_g(phi)
    pairs = []
    for _ in range(iters):
        p = _direction(g, pairs) if pairs else -g / g.abs().max()
        gp = float((g * p).sum())
        if not gp < 0:
            pairs, p = [], -g / g.abs().max()
            gp = float((g * p).sum())
        a = 1.0
        for _ in range(31):
            fn, gn = f_and_g(phi + a * p)
            if fn <= f + 1e-4 * a * gp:
                break
            a *= 0.5
        else:
            break
        s, y = a * p, gn - g
        if float((s * y).sum()) > 1e-10 * float(s.norm() * y.norm()):
            pairs = (pairs + [(s, y, (s * y).sum(1))])[-m:]
        phi, stop = phi + s, f - fn <= tol * f
        f, g = fn, gn
        if stop:
            break
    u = torch.polar(torch.ones_like(phi[0]), phi[0])
    u = u * torch.polar(torch.ones((), dtype=F64, device=DEV), -(T.abs().square().sum(1) * u).sum().angle())
    return T * u[:, None]


def _net64(c, params, X):
    x, o, dims = X, 0, [c["n_in"], c["h1"], c["h2"], c["n_out"]]
    for i, (a, b) in enumerate(zip(dims, dims[1:])):
        x = x @ params[o:o + a * b].reshape(b, a).T + params[o + a * b:o + a * b + b]
        x = torch.nn.functional.gelu(x) if i < 2 else x
        o += a * b + b
    return x


def exact(case, seed):
    c, op, s = case, case["op"], _inputs(case, seed)
    if op == "preprocess":
        x = s["frames"][:, ::2, ::2].reshape(c["K"], -1)
        y = torch.empty((x.shape[1], c["K"]), dtype=F64, device=DEV)
        for k in range(0, c["K"], 1024):
            v = x[k:k + 1024]
            y[:, k:k + 1024] = ((v.to(torch.int32) & 0xFFFF) if c["pix"] == "u16" else v).to(F64).T
        E = y.sum(1)
        top = E.sort(descending=True)[0]
        n = int((top.cumsum(0) >= 0.999 * E.sum()).nonzero()[0])
        mask = E >= top[n]
        return dict(y=y * mask[:, None], mask=mask.to(torch.uint8), energy=E, n_inside=mask.sum().to(torch.int32).reshape(1))
    if op.startswith("mlp"):
        P, X, T = s["params"].to(F64), s["X"].to(F64), s["T"].to(F64)
        if op == "mlp_forward":
            return _net64(c, P, X)
        P.requires_grad_(True)
        y, n = _net64(c, P, X), c["n_out"] // 2
        yc, tc = torch.complex(y[:, :n], y[:, n:]), torch.complex(T[:, :n], T[:, n:])
        al = (yc.conj() * tc).sum(1, keepdim=True).detach()
        loss = (yc - tc * al.conj() / al.abs()).abs().square().sum() / (c["B"] * c["n_out"])
        g = torch.autograd.grad(loss, P)[0]
        # the first step of Adam from zero moments: both bias corrections cancel
        return dict(loss=loss.detach().reshape(1), params=P.detach() - LR * g / (g.abs() + 1e-8))
    d = s["masks"].to(C128)
    if op == "fit":
        return _fit64(c, s["T"].to(C128), d, s["incident"].to(C128) if c["kind"] else None, s["I"])
    M, step = c["M"], max(1, 2 ** 23 // (c["J"] * c["N"]))
    got = []
    for r in range(0, M, step):
        b = slice(r, min(M, r + step))
        if op == "forward":
            z = torch.fft.fft(d * s["T"][b, None].to(C128))
            got.append((z.real.square() + z.imag.square(),))
        elif op == "grad":
            f, g, _ = _grad64(s["T"][b].to(C128), s["Y"][b].to(F64), d, c["cost"])
            got.append((f, g))
        else:
            T0 = s["T0"][b].to(C128) if op == "track" else _spectral64(torch.arange(M, device=DEV)[b], s["Y"][b], d)
            got.append(_lbfgs64(T0, s["Y"][b], d, c["iters"], c.get("tol", 0.0)))
    out = [torch.cat(x) for x in zip(*got)]
    if op == "forward":
        return out[0]
    if op == "grad":
        return dict(loss=out[0], G=out[1])
    return dict(T=out[0], loss=out[1], status=out[2])

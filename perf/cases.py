"""Timed cases of the T2 Shuffling solver: what a reconstruction program calls, on seeded inputs.

The cases follow a scan through the library: pre-processing of the sparse readout lines, the operators
A, A^H and A^H A, the LLR prox, whole solves (FISTA and ADMM) and post-processing.  Sizes are the
repository's scan configurations (64x48 single slices, the 320-slice 256x160 knee scan, Table I's
288-slice 260x240 scan with two map sets and 12x12 blocks, the 240x128 and 192x192 batch scans) and
matrices in between that no configuration names.  Inputs are smooth coil maps, a multi-tissue ellipsoid
phantom with T2 in 20-200 ms, variable-density echo masks and 1 % noise, made on the GPU from the seed.
"""
import math

import numpy as np
import torch

from paper_1809_04195_gb300 import t2sh

PI = math.pi
# even products of 2, 3, 5 and 13 (the lengths the solver takes) from 48 to 288
SMOOTH = [n for n in range(48, 290, 2) if any(n == 2 ** a * 3 ** b * 5 ** c * 13 ** d for a in range(1, 9)
                                              for b in range(6) for c in range(4) for d in range(3))]
CONFIGURED = [48, 64, 96, 128, 160, 192, 240, 256, 260]


def _case(name, op, ny, nz, C, S, T=80, K=4, M=1, b=8, frac=0.05, lam=0.005, iters=0, form="proj", nx=0, nchan=0,
          levels=0, cg=0):
    c = dict(op=op, ny=ny, nz=nz, C=C, S=S, T=T, K=K, M=M, b=b, frac=frac, lam=lam, iters=iters, form=form, nx=nx,
             nchan=nchan, levels=levels, cg=cg)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # one small slice: an interactive or per-slice solver applying A^H A, bound by launches and latency
        _case("normal_64x48_1slice", "normal", 64, 48, 8, 1, T=32, frac=0.10),
        # the knee scan in one launch per pass: the operator every solver iteration applies
        _case("normal_256x160_320slices", "normal", 256, 160, 12, 320),
        # Table I: 260-point columns, two map sets
        _case("normal_260x240_288slices_m2", "normal", 260, 240, 7, 288, M=2, b=12, frac=1 / 139),
        # a matrix that no configuration names (9 = 3 * 3 in one length, 45 = 9 * 5 in the other)
        _case("normal_180x144_48slices", "normal", 180, 144, 10, 48),
        # the prox alone, as a program with its own proximal loop calls it: ragged 12x12 blocks, two map sets
        _case("llr_260x240_288slices_m2", "llr", 260, 240, 1, 288, T=16, M=2, b=12, frac=0.2, lam=0.0125),
        # A^H y of per-echo k-space (the form the scanner's sorted data have), 80 echoes at 5 %
        _case("adjoint_te_240x128_24slices", "adjoint", 240, 128, 8, 24, form="te"),
        # A x per echo: data consistency and simulation, writes all 80 echoes
        _case("forward_te_256x160_8slices", "forward", 256, 160, 12, 8, form="te"),
        # the smallest whole call: plan and 50 FISTA iterations of one slice
        _case("solve_64x48_1slice", "solve", 64, 48, 8, 1, T=32, frac=0.10, lam=0.01, iters=50, form="te"),
        # the whole knee scan: plan and 100 FISTA iterations
        _case("solve_256x160_320slices", "solve", 256, 160, 12, 320, iters=100),
        # ADMM with conjugate-gradient inner solves on a share of the 192x192, 16-coil scan
        _case("admm_192x192_32slices", "admm", 192, 192, 16, 32, iters=3, cg=3),
        # sparse readout lines of the Table I scan: compression of 16 channels to 7, decoupling, projection
        _case("preprocess_260x240_nx288", "preprocess", 260, 240, 7, 288, M=2, frac=1 / 139, nx=288, nchan=16),
        # after the solve: wavelet soft-threshold of the knee volume and its three TE images
        _case("post_256x160_320slices", "post", 256, 160, 12, 320, levels=3),
    ]


def draw(rng):
    op = rng.choice(["normal", "normal", "llr", "forward", "adjoint", "solve", "admm", "preprocess", "post"])
    size = lambda: rng.choice(CONFIGURED if rng.random() < 0.5 else SMOOTH)  # noqa: E731
    logint = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(max(lo, hi))))))  # noqa: E731
    ny, nz = size(), size()
    C, T, K = rng.randint(4, 16), rng.randint(16, 96), rng.choice([2, 3, 4, 4, 4, 4, 6])
    M, b = rng.choice([1, 1, 2]), rng.choice([6, 8, 8, 12])
    frac, lam = rng.uniform(0.01, 0.10), rng.uniform(0.002, 0.02)
    form = rng.choice(["te", "proj"])
    points = ny * nz * C * K
    # slices: up to a whole scan, and no more k-space than the largest listed case of the kind holds
    most = {"normal": 600e6, "llr": 600e6, "forward": 50e6, "adjoint": 50e6, "solve": 600e6, "admm": 70e6,
            "preprocess": 400e6, "post": 400e6}[op]
    if form == "te" and op in ("forward", "adjoint", "solve"):
        most = min(most, 400e6 * K / T)
    elif op in ("forward", "adjoint"):
        most = 400e6
    S = logint(1, max(1, min(320, int(most // points))))
    case = _case("", op, ny, nz, C, S, T=T, K=K, M=M, b=b, frac=frac, lam=lam, form=form)
    if op == "solve":
        case["iters"] = min(rng.randint(10, 100), max(2, int(20e9 / (points * S))))
    if op == "admm":
        case["iters"], case["cg"] = rng.randint(1, 4), rng.randint(1, 4)
    if op == "preprocess":
        case.update(nx=max(48, size()), nchan=16, frac=min(frac, 0.02), C=rng.randint(4, 12))
    if op == "post":
        S = max(8, S // 8 * 8)
        case["S"], case["levels"] = S, max(v for v in range(4) if not ny % 2 ** v and not nz % 2 ** v)
    return case


# ------------------------------------------------------------------------------------------------
# Inputs
# ------------------------------------------------------------------------------------------------
DEV = "cuda"


def _basis(T, K):
    """Top-K left singular vectors of simulated decays exp(-t / T2) [T][K], and the echo times (ms)."""
    t = (np.arange(T) + 1.0) * 5.0
    u = np.linalg.svd(np.exp(-t[:, None] / np.linspace(20, 200, 256)[None]), full_matrices=False)[0][:, :K]
    sg = np.where(u[np.abs(u).argmax(0), np.arange(K)] < 0, -1.0, 1.0)
    return (u * sg).astype(np.float32), t


def _mask(T, ny, nz, frac, rng):
    ky, kz = (np.arange(ny) - ny // 2) / (ny / 2), (np.arange(nz) - nz // 2) / (nz / 2)
    r = np.sqrt(ky[:, None] ** 2 + kz[None] ** 2)
    p = np.clip(1 - r / r.max(), 0, 1) ** 2 + 0.02
    for _ in range(20):
        p = np.clip(p * frac / p.mean(), 0, 1)
    m = (rng.random((T, ny, nz), dtype=np.float32) < p[None].astype(np.float32)).astype(np.uint8)
    m[0, ny // 2 - 3:ny // 2 + 3, nz // 2 - 3:nz // 2 + 3] = 1
    return m


def _grid(ny, nz):
    y = torch.linspace(-1, 1, ny + 1, device=DEV)[:-1]
    z = torch.linspace(-1, 1, nz + 1, device=DEV)[:-1]
    return y[:, None], z[None, :]


def _maps(c, rng):
    """Smooth coils on a ring [S][C][M][ny][nz], each pixel's S^H S with largest eigenvalue 1."""
    S, C, M, ny, nz = c["S"], c["C"], c["M"], c["ny"], c["nz"]
    y, z = _grid(ny, nz)
    out = torch.empty((S, C, M, ny, nz), dtype=torch.complex64, device=DEV)
    ang = torch.tensor(rng.uniform(0, 2 * PI, (S, M, 1)) + 2 * PI * np.arange(C) / C, device=DEV, dtype=torch.float32)
    ph = torch.tensor(rng.uniform(-PI, PI, (3, S, M, C)), device=DEV, dtype=torch.float32)
    for m in range(M):
        for j in range(C):
            a = ang[:, m, j, None, None]
            g = torch.exp(-((y - 1.1 * torch.cos(a)) ** 2 + (z - 1.1 * torch.sin(a)) ** 2) / 1.28) * (0.3 if m else 1.0)
            q = ph[:, :, m, j, None, None]
            out[:, j, m] = torch.polar(g, q[0] + q[1] * y + q[2] * z)
    lam = torch.zeros((S, ny, nz), device=DEV)
    if M == 1:
        for j in range(C):
            lam += out[:, j, 0].abs() ** 2
    else:
        a, d, o = torch.zeros_like(lam), torch.zeros_like(lam), torch.zeros_like(lam, dtype=torch.complex64)
        for j in range(C):
            a += out[:, j, 0].abs() ** 2
            d += out[:, j, 1].abs() ** 2
            o += out[:, j, 0].conj() * out[:, j, 1]
        lam = (a + d) / 2 + torch.sqrt(((a - d) / 2) ** 2 + o.abs() ** 2)
    out *= (1 / lam.sqrt())[:, None, None]
    return out


def _alpha(c, phi, te, rng, gen, noise=0.01):
    """Basis coefficients of a 3D ellipsoid phantom with a smooth phase [S][M][K][ny][nz]."""
    S, M, K, ny, nz = c["S"], c["M"], c["K"], c["ny"], c["nz"]
    y, z = _grid(ny, nz)
    x = ((torch.arange(S, device=DEV) + 0.5) * (2.0 / S) - 1)[:, None, None]
    lab = torch.zeros((S, ny, nz), dtype=torch.int64, device=DEV)
    coef = np.zeros((15, K))
    for e in range(14):
        cen, ax = (np.zeros(3), np.array([0.95, 0.8, 0.7])) if not e else (rng.uniform(-0.5, 0.5, 3), rng.uniform(0.1, 0.4, 3))
        lab[((x - cen[0]) / ax[0]) ** 2 + ((y - cen[1]) / ax[1]) ** 2 + ((z - cen[2]) / ax[2]) ** 2 <= 1] = e + 1
        coef[e + 1] = rng.uniform(0.2, 1) * (np.exp(-te / rng.uniform(20, 200)) @ phi)
    coef = torch.tensor(coef, dtype=torch.float32, device=DEV)
    out = torch.empty((S, M, K, ny, nz), dtype=torch.complex64, device=DEV)
    torch.view_as_real(out).normal_(0, noise / math.sqrt(2), generator=gen)
    for m in range(M):
        a, b = rng.uniform(-1, 1, 2)
        phase = torch.polar(torch.full_like(y * z, 0.2 if m else 1.0), a * y + b * z)
        for k in range(K):
            out[:, m, k] += coef[:, k][lab] * phase
    return out


def _fft2c(v, inverse=False):
    f = torch.fft.ifft2 if inverse else torch.fft.fft2
    return torch.fft.fftshift(f(torch.fft.ifftshift(v, dim=(-2, -1)), norm="ortho"), dim=(-2, -1))


def _psi(phi, mask, dt=torch.float64):
    """Phi^T P(n) Phi [K][K][ny][nz]."""
    T, K = phi.shape
    out = torch.zeros((K, K) + tuple(mask.shape[1:]), dtype=dt, device=DEV)
    p, m = phi.to(dt), mask.to(dt)
    for t in range(T):
        out += (p[t][:, None] * p[t][None, :])[:, :, None, None] * m[t]
    return out


def _sense(x, maps):
    """sum_m S_cm x_mk: [s][M][K].. with [s][C][M].. -> [s][C][K].."""
    v = maps[:, :, 0, None] * x[:, None, 0]
    for m in range(1, maps.shape[2]):
        v = v + maps[:, :, m, None] * x[:, None, m]
    return v


def _apply_psi(v, psi):
    return torch.stack([sum(psi[k, l] * v[:, :, l] for l in range(v.shape[2])) for k in range(v.shape[2])], 2)


def _chunks(c, per):
    """Slice ranges whose coil images (per bytes a value) stay near 8 GB."""
    n = max(1, int(8e9 / (c["C"] * c["K"] * c["ny"] * c["nz"] * per)))
    return [(s, min(c["S"], s + n)) for s in range(0, c["S"], n)]


def _scan(c, seed):
    """phi, mask, maps, alpha, generator of a scan."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    phi, te = _basis(c["T"], c["K"])
    mask = torch.from_numpy(_mask(c["T"], c["ny"], c["nz"], c["frac"], rng)).to(DEV)
    maps = _maps(c, rng)
    alpha = _alpha(c, phi.astype(np.float64), te, rng, gen)
    return torch.from_numpy(phi).to(DEV), mask, maps, alpha, gen


def _kspace(c, phi, mask, maps, alpha, gen, scale=True):
    """Noisy k-space of the phantom: per echo [S][C][T].. or projected [S][C][K].., largest magnitude 1."""
    te = c["form"] == "te"
    out = torch.empty((c["S"], c["C"], c["T"] if te else c["K"], c["ny"], c["nz"]), dtype=torch.complex64, device=DEV)
    m = mask.to(torch.float32)
    if not te:
        psi = _psi(phi, mask)
        ev, U = np.linalg.eigh(psi.permute(2, 3, 0, 1).cpu().numpy())
        root = torch.from_numpy((U * np.sqrt(np.clip(ev, 0, None))[..., None, :]) @ U.swapaxes(-1, -2))
        root, psi = root.permute(2, 3, 0, 1).to(DEV, torch.float32), psi.to(torch.float32)
    sig = None
    for s0, s1 in _chunks(c, 40):
        f = _fft2c(_sense(alpha[s0:s1], maps[s0:s1]))
        if sig is None:
            sig = 0.01 * float(f[:, :, 0].abs().max())
        w = torch.empty((s1 - s0,) + (tuple(out.shape[1:2]) if te else tuple(out.shape[1:3])) + (c["ny"], c["nz"]),
                        dtype=torch.complex64, device=DEV)
        if te:
            for t in range(c["T"]):
                torch.view_as_real(w).normal_(0, sig / math.sqrt(2), generator=gen)
                for k in range(c["K"]):
                    w += phi[t, k] * f[:, :, k]
                out[s0:s1, :, t] = w * m[t]
        else:
            torch.view_as_real(w).normal_(0, sig / math.sqrt(2), generator=gen)
            out[s0:s1] = _apply_psi(f, psi) + _apply_psi(w, root)
        del f, w
    if scale:
        out /= max(float(out[s].abs().max()) for s in range(c["S"]))
    return out


def _lines(c, seed):
    """Sparse readout lines [n][nchan][nx] (a low-rank channel mix, energy towards the k-space centre), their
    echo, ky and kz indices, and the basis."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    t, ky, kz = (a.astype(np.int32) for a in np.nonzero(_mask(c["T"], c["ny"], c["nz"], c["frac"], rng)))
    n, ch, nx = len(t), c["nchan"], c["nx"]
    g = torch.empty((n, ch, nx), dtype=torch.complex64, device=DEV)
    torch.view_as_real(g).normal_(0, 1, generator=gen)
    q = np.linalg.qr(rng.normal(size=(ch, ch)) + 1j * rng.normal(size=(ch, ch)))[0] * 0.7 ** np.arange(ch)
    lines = torch.matmul(torch.from_numpy(q.astype(np.complex64)).to(DEV), g)
    r = np.sqrt(((ky - c["ny"] // 2) / c["ny"]) ** 2 + ((kz - c["nz"] // 2) / c["nz"]) ** 2)
    rx = np.abs(np.arange(nx) - nx // 2) / nx
    lines *= torch.from_numpy((1 / (0.02 + r[:, None] ** 2 + rx[None] ** 2)).astype(np.float32)).to(DEV)[:, None]
    return lines, t, ky, kz, torch.from_numpy(_basis(c["T"], c["K"])[0]).to(DEV)


def _window(c):
    return min(24, c["ny"], c["nz"], c["nx"])


def _dims(c, seed):
    return t2sh.make_dims(c["ny"], c["nz"], c["C"], c["T"], c["K"], nslices=c["S"], nmaps=c["M"], block=c["b"],
                          lam=c["lam"], iters=c["iters"], seed=seed)


def _shift(c, seed):
    """The shift a prox call is given."""
    return (seed * 5 + 3) % c["b"], (seed * 7 + 5) % c["b"]


TAU = 0.05        # the prox's threshold: 1 % noise falls below it, tissue stays
WAVELET_TAU = 0.02
TE = (3, 9, 17)   # echoes at 20, 50 and 90 ms


def _echoes(c):
    return [t for t in TE if t < c["T"]]


def prepare(case, seed):
    c = case
    st = {"case": c, "seed": seed}
    if c["op"] == "preprocess":
        st["lines"], st["t"], st["ky"], st["kz"], st["phi"] = _lines(c, seed)
        return st
    phi, mask, maps, alpha, gen = _scan(c, seed)
    st["dims"] = _dims(c, seed)
    st["form"] = t2sh.KSPACE_TE if c["form"] == "te" else t2sh.KSPACE_PROJ
    if c["op"] in ("solve", "admm"):
        # one scan: its own masks, maps and k-space, so the plan belongs to the call
        st["phi"], st["mask"], st["maps"] = phi, mask, maps
        st["y"] = _kspace(c, phi, mask, maps, alpha, gen)
        return st
    st["plan"] = t2sh.Plan(st["dims"], phi, mask, maps)
    st["x"] = _kspace(c, phi, mask, maps, alpha, gen) if c["op"] == "adjoint" else alpha
    return st


def run(state):
    c = state["case"]
    op = c["op"]
    if op == "preprocess":
        idx = (state["t"], state["ky"], state["kz"])
        w = t2sh.coil_compression(state["lines"], *idx, c["ny"], c["nz"], c["T"], window=_window(c), ncomp=c["C"])
        ytil, mask = t2sh.preprocess(state["lines"], *idx, w, state["phi"], c["ny"], c["nz"])
        return {"w": w, "ytil": ytil, "mask": mask}
    if op in ("solve", "admm"):
        with t2sh.Plan(state["dims"], state["phi"], state["mask"], state["maps"]) as p:
            if op == "admm":
                return p.solve_admm(state["y"], state["form"], rho=0.5, cg_iters=c["cg"])
            return p.solve(state["y"], state["form"])
    p = state["plan"]
    if op == "normal":
        return p.normal_op(state["x"])
    if op == "forward":
        return p.forward(state["x"], state["form"])
    if op == "adjoint":
        return p.adjoint(state["x"], state["form"])
    if op == "llr":
        return p.llr_prox(state["x"].clone(), TAU, *_shift(c, state["seed"]))  # the caller keeps its iterate
    a = state["x"].clone()  # post: the solved coefficients are kept
    if c["levels"]:
        a = p.wavelet_denoise(a, WAVELET_TAU, c["levels"])
    return {"alpha": a, "te": p.postprocess(a, _echoes(c), 0.65)}


def work(case):
    c = case
    N = c["ny"] * c["nz"]
    vec, ksp, maps = (c["S"] * n * N for n in (c["M"] * c["K"], c["C"] * c["K"], c["C"] * c["M"]))
    fft = 5 * math.log2(N)
    psi = c["K"] * (c["K"] + 1) // 2 * N * 4
    sense = 8 * c["S"] * c["C"] * c["M"] * c["K"] * N
    normal = 2 * sense + ksp * (2 * fft + 4 * c["K"])
    svt = vec * (16 * c["K"] + 4)
    samples = c["S"] * c["C"] * c["T"] * c["frac"] * N  # acquired values of per-echo data
    mask = c["T"] * N
    te = c["form"] == "te"
    op = c["op"]
    if op == "normal":
        return {"bytes": 8 * (2 * vec + maps) + psi, "flops": normal}
    if op == "llr":
        return {"bytes": 8 * 2 * vec, "flops": svt}
    if op == "adjoint":
        return {"bytes": 8 * (vec + maps + (samples if te else ksp)) + (mask if te else 0),
                "flops": sense + ksp * fft + (4 * samples * c["K"] if te else 0)}
    if op == "forward":
        out = c["S"] * c["C"] * c["T"] * N if te else ksp
        return {"bytes": 8 * (vec + maps + out) + (mask if te else psi),
                "flops": sense + ksp * fft + 4 * (samples if te else ksp) * c["K"]}
    if op in ("solve", "admm"):
        per = (1 + c["cg"]) * (normal + 24 * vec) if op == "admm" else normal + 10 * vec
        return {"bytes": 8 * (vec + maps + (samples if te else ksp)) + mask, "flops": c["iters"] * (per + svt)}
    if op == "preprocess":
        n = c["T"] * c["frac"] * N
        return {"bytes": 8 * n * c["nchan"] * c["nx"] + 8 * c["nx"] * c["C"] * c["K"] * N + mask,
                "flops": n * c["nx"] * c["C"] * (8 * c["nchan"] + 5 * math.log2(c["nx"]) + 4 * c["K"])}
    nte = len(_echoes(c))
    line = 5 * math.log2(c["nz"])
    return {"bytes": 8 * (2 * vec + maps) + 4 * c["S"] * nte * N,
            "flops": nte * c["S"] * N * (4 * c["M"] * c["K"] + c["C"] * (8 * c["M"] + 3 * line + 8)) + 40 * vec}


# ------------------------------------------------------------------------------------------------
# The same in 64 bits
# ------------------------------------------------------------------------------------------------
def _svt(blk, tau):
    """Singular-value soft threshold of [..][pixels][K], through the Gram matrix."""
    g = (blk.mH @ blk).cpu().numpy()
    ev, v = np.linalg.eigh(g)
    s = np.sqrt(np.clip(ev, 0, None))
    f = np.where(s > tau, 1 - tau / np.where(s > tau, s, 1), 0.0)
    return blk @ torch.from_numpy((v * f[..., None, :]) @ v.conj().swapaxes(-1, -2)).to(blk.device)


def _llr(x, b, tau, sy, sz):
    """The prox of [S][M][K][ny][nz]: zeros appended to the last blocks leave their singular values."""
    S, M, K, ny, nz = x.shape
    v = torch.roll(x, (-sy, -sz), (-2, -1))
    gy, gz = -(-ny // b), -(-nz // b)
    v = torch.nn.functional.pad(v, (0, gz * b - nz, 0, gy * b - ny))
    v = v.reshape(S, M, K, gy, b, gz, b).permute(0, 1, 3, 5, 4, 6, 2).reshape(S, M, gy, gz, b * b, K)
    v = _svt(v, tau).reshape(S, M, gy, gz, b, b, K).permute(0, 1, 6, 2, 4, 3, 5).reshape(S, M, K, gy * b, gz * b)
    return torch.roll(v[..., :ny, :nz], (sy, sz), (-2, -1))


def _by_slices(c, f, x):
    return torch.cat([f(x[s0:s1].to(torch.complex128), s0, s1) for s0, s1 in _chunks(c, 160)])


def _unsense(v, maps):
    return torch.stack([(maps[:, :, m, None].conj() * v).sum(1) for m in range(maps.shape[2])], 1)


def _normal64(c, maps, psi):
    def f(x, s0, s1):
        m = maps[s0:s1].to(torch.complex128)
        return _unsense(_fft2c(_apply_psi(_fft2c(_sense(x, m)), psi), True), m)
    return lambda x: _by_slices(c, f, x)


def _adjoint64(c, phi, mask, maps, y):
    def f(v, s0, s1):
        if c["form"] == "te":
            p, v0 = phi.to(torch.float64), v * mask
            v = torch.stack([sum(p[t, k] * v0[:, :, t] for t in range(c["T"])) for k in range(c["K"])], 2)
        return _unsense(_fft2c(v, True), maps[s0:s1].to(torch.complex128))
    per = max(1, int(8e9 / (c["C"] * y.shape[2] * c["ny"] * c["nz"] * 48)))
    return torch.cat([f(y[s:s + per].to(torch.complex128), s, min(c["S"], s + per)) for s in range(0, c["S"], per)])


def _shifts(seed, iters, b):
    """SplitMix64 outputs: low and high words modulo the block edge."""
    out, mask = [], (1 << 64) - 1
    for i in range(iters):
        z = (seed + (i + 1) * 0x9E3779B97F4A7C15) & mask
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
        z ^= z >> 31
        out.append(((z & 0xFFFFFFFF) % b, (z >> 32) % b))
    return out


def _step(maps, psi):
    a = sum(maps[:, j, 0].to(torch.complex128).abs() ** 2 for j in range(maps.shape[1]))
    if maps.shape[2] > 1:
        m = maps.to(torch.complex128)
        d = sum(m[:, j, 1].abs() ** 2 for j in range(m.shape[1]))
        o = sum(m[:, j, 0].conj() * m[:, j, 1] for j in range(m.shape[1])).abs()
        a = (a + d) / 2 + torch.sqrt(((a - d) / 2) ** 2 + o ** 2)
    return 1 / (float(a.max()) * float(np.linalg.eigvalsh(psi.permute(2, 3, 0, 1).cpu().numpy()).max()))


def _fista64(c, seed, phi, mask, maps, y):
    psi = _psi(phi, mask)
    A, mu, aty = _normal64(c, maps, psi), _step(maps, psi), _adjoint64(c, phi, mask, maps, y)
    x = z = torch.zeros_like(aty)
    t = 1.0
    for sy, sz in _shifts(seed, c["iters"], c["b"]):
        xn = _llr(z - mu * (A(z) - aty), c["b"], mu * c["lam"], sy, sz)
        tn = (1 + math.sqrt(1 + 4 * t * t)) / 2
        x, z, t = xn, xn + (t - 1) / tn * (xn - x), tn
    return x


def _admm64(c, seed, phi, mask, maps, y, rho=0.5):
    N, aty = _normal64(c, maps, _psi(phi, mask)), _adjoint64(c, phi, mask, maps, y)
    dot = lambda a, b: (a.conj() * b).real.sum((1, 2, 3, 4), keepdim=True)  # noqa: E731
    quot = lambda a, b: torch.where(b != 0, a / torch.where(b != 0, b, torch.ones_like(b)), torch.zeros_like(b))  # noqa: E731
    a = v = u = torch.zeros_like(aty)
    for sy, sz in _shifts(seed, c["iters"], c["b"]):
        r = aty + rho * (v - u) - N(a) - rho * a
        p, rr = r, dot(r, r)
        for _ in range(c["cg"]):
            q = N(p) + rho * p
            s = quot(rr, dot(p, q))
            a, r = a + s * p, r - s * q
            rn = dot(r, r)
            p, rr = r + quot(rn, rr) * p, rn
        v = _llr(a + u, c["b"], c["lam"] / rho, sy, sz)
        u = u + a - v
    return v


def _forward64(c, phi, mask, maps, x):
    """A x [S][C][T].., or projected [S][C][K].."""
    n = c["T"] if c["form"] == "te" else c["K"]
    out = torch.empty((c["S"], c["C"], n, c["ny"], c["nz"]), dtype=torch.complex128, device=DEV)
    psi, p = _psi(phi, mask), phi.to(torch.float64)
    for s0, s1 in _chunks(c, 160):
        f = _fft2c(_sense(x[s0:s1].to(torch.complex128), maps[s0:s1].to(torch.complex128)))
        if c["form"] == "te":
            for t in range(c["T"]):
                out[s0:s1, :, t] = mask[t] * sum(p[t, k] * f[:, :, k] for k in range(c["K"]))
        else:
            out[s0:s1] = _apply_psi(f, psi)
    return out


def _haar(v, dim):
    s, d = v.unflatten(dim, (-1, 2)).movedim(dim + 1, 0)
    return (s + d) / math.sqrt(2), (s - d) / math.sqrt(2)


def _denoise64(a, tau, levels):
    """Soft-thresholded details of a Haar pyramid over (slice, y, z) of [S][..][ny][nz]."""
    if not levels:
        return a
    dims = (0, a.dim() - 2, a.dim() - 1)
    parts = [a]
    for d in dims:
        parts = [q for p in parts for q in _haar(p, d)]
    soft = lambda q: q * torch.clamp(1 - tau / q.abs().clamp_min(1e-300), min=0)  # noqa: E731
    parts = [_denoise64(parts[0], tau, levels - 1)] + [soft(q) for q in parts[1:]]
    for d in reversed(dims):
        parts = [torch.stack(((s + t) / math.sqrt(2), (s - t) / math.sqrt(2)), d + 1).flatten(d, d + 1)
                 for s, t in zip(parts[::2], parts[1::2])]
    return parts[0]


def _te_images64(c, phi, maps, a):
    """Homodyne along z (step weights, phase of the two-sided band) and root sum of squares."""
    nz, te = c["nz"], _echoes(c)
    w = math.ceil(float(np.float32(0.65)) * nz) - nz // 2
    d = torch.arange(nz, device=DEV) - nz // 2
    band = ((d >= -w) & (d <= w)).to(torch.float64)
    high = torch.where(d < -w, 0.0, torch.where(d <= w, 1.0, 2.0)).to(torch.float64)
    f = lambda v, inv: torch.fft.fftshift((torch.fft.ifft if inv else torch.fft.fft)(torch.fft.ifftshift(v, dim=-1)), dim=-1)  # noqa: E731
    out = torch.empty((c["S"], len(te), c["ny"], nz), dtype=torch.float64, device=DEV)
    for s0, s1 in _chunks(c, 160):
        for i, t in enumerate(te):
            x = (a[s0:s1] * phi[t].to(torch.float64)[:, None, None]).sum(2, keepdim=True)
            k = f(_sense(x, maps[s0:s1].to(torch.complex128))[:, :, 0], False)
            h, l = f(k * high, True), f(k * band, True)
            m = l.abs()
            o = torch.where(m > 0, (h * l.conj()).real / torch.where(m > 0, m, torch.ones_like(m)), h.real)
            out[s0:s1, i] = (o ** 2).sum(1).sqrt()
    return out


def _preprocess64(c, lines, t, ky, kz, phi):
    ny, nz, nx, win, ch = c["ny"], c["nz"], c["nx"], _window(c), c["nchan"]
    pix = ky.astype(np.int64) * nz + kz
    y0, z0, x0 = ny // 2 - win // 2, nz // 2 - win // 2, nx // 2 - win // 2
    inside = np.nonzero((ky >= y0) & (ky < y0 + win) & (kz >= z0) & (kz < z0 + win))[0]
    _, seg, count = np.unique(pix[inside], return_inverse=True, return_counts=True)
    X = torch.zeros((len(count), ch, win), dtype=torch.complex128, device=DEV)
    X.index_add_(0, torch.from_numpy(seg).to(DEV), lines[torch.from_numpy(inside).to(DEV)][:, :, x0:x0 + win].to(torch.complex128))
    X /= torch.from_numpy(count).to(DEV, torch.float64)[:, None, None]
    X = X.permute(0, 2, 1).reshape(-1, ch)
    ev, v = np.linalg.eigh((X.mH @ X).cpu().numpy())
    w = v[:, ::-1][:, :c["C"]]
    top = w[np.abs(w).argmax(0), np.arange(c["C"])]
    w = torch.from_numpy(np.ascontiguousarray(w * (top.conj() / np.abs(top)))).to(DEV)
    out = torch.zeros((ny * nz, c["C"], c["K"], nx), dtype=torch.complex128, device=DEV)
    tt, at = torch.from_numpy(t).to(DEV, torch.int64), torch.from_numpy(pix).to(DEV)
    for j in range(0, len(t), 8192):
        q = torch.einsum("jcx,cd->jdx", lines[j:j + 8192].to(torch.complex128), w)
        q = torch.fft.fftshift(torch.fft.ifft(torch.fft.ifftshift(q, dim=-1), norm="ortho"), dim=-1)
        out.index_add_(0, at[j:j + 8192], q[:, :, None] * phi.to(torch.float64)[tt[j:j + 8192]][:, None, :, None])
    mask = torch.zeros((c["T"], ny * nz), dtype=torch.uint8, device=DEV)
    mask[tt, at] = 1
    return {"w": w, "ytil": out.permute(3, 1, 2, 0).reshape(nx, c["C"], c["K"], ny, nz), "mask": None}


def exact(case, seed):
    c = case
    op = c["op"]
    if op == "preprocess":
        return _preprocess64(c, *_lines(c, seed))
    points = c["S"] * c["C"] * c["K"] * c["ny"] * c["nz"]
    if op in ("solve", "admm") and c["iters"] * (1 + c["cg"]) * points > 2e9:
        return None  # minutes in 64 bits
    phi, mask, maps, alpha, gen = _scan(c, seed)
    if op in ("solve", "admm", "adjoint"):
        y = _kspace(c, phi, mask, maps, alpha, gen)
        del alpha
        if op == "adjoint":
            return _adjoint64(c, phi, mask, maps, y)
        return (_fista64 if op == "solve" else _admm64)(c, seed, phi, mask, maps, y)
    if op == "normal":
        return _normal64(c, maps, _psi(phi, mask))(alpha)
    if op == "forward":
        return _forward64(c, phi, mask, maps, alpha)
    del gen
    if op == "llr":
        sy, sz = _shift(c, seed)
        return torch.cat([_llr(alpha[s:s + 16].to(torch.complex128), c["b"], TAU, sy, sz) for s in range(0, c["S"], 16)])
    a = _denoise64(alpha.to(torch.complex128), WAVELET_TAU, c["levels"])
    return {"alpha": a, "te": _te_images64(c, phi, maps, a)}

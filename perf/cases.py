"""Cases that stand for the use of the framework, for measuring it.

A case is one call a user's program makes: the forward model (simulating data,
previewing an estimate), the data term and its gradients (one step of the
automatic-differentiation reconstructor), one LSQML epoch, and the relaxed-probe,
multislice, split-BF16 and batched-serving forms of them. Inputs follow the
workloads of the benchmark (Hermite-Gaussian probe modes, Fermat-spiral scans,
objects with smoothed random phase, Poisson counts) and are made with torch alone.
``exact`` evaluates the same call in complex128 with torch.
"""
import math

import torch

from paper_2510_20929_gb300 import api, autograd

EPS = 1.0          # one count, as in the benchmark
DELTA, LAM = 0.1, 1e-6
DZ, WAVELENGTH, PIXEL = 2e-6, 0.1e-9, 10e-9
MARGIN = 1.0 / 64.0
HG = [(0, 0), (1, 0), (0, 1), (1, 1), (2, 0), (0, 2), (2, 1), (1, 2)]


def _case(name, kind, N, M, J, H, W=None, **kw):
    c = {"kind": kind, "N": N, "M": M, "J": J, "H": H, "W": H if W is None else W, "counts": 1e6,
         "noise": "gaussian", "batch": min(256, J)}
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a live preview: the patterns of a few scan points while an alignment is turned
        _case("preview64", "forward", 64, 1, 16, 256),
        # the plain LSQML reconstruction (the benchmark's raster64): one short epoch, replayed as a graph
        _case("small64_epoch", "epoch", 64, 1, 100, 256, counts=1e4, graph=True),
        # simulating a whole multi-mode scan (the benchmark makes its data this way)
        _case("simulate128", "forward", 128, 5, 4096, 1024),
        # a gradient step on Poisson counts over an object of odd sides
        _case("poisson128_term", "term", 128, 3, 1000, 777, 801, noise="poisson"),
        # the headline workload: one LSQML epoch over 4096 positions
        _case("spiral128_epoch", "epoch", 128, 5, 4096, 1024),
        # Poisson LSQML with position correction, compact minibatches and the accumulate-once update
        _case("compact64_epoch", "epoch", 64, 4, 2999, 700, 650, noise="poisson", batch=128, counts=2e5,
              compact=True, positions=True),
        # the Adam reconstructor at the 256 window: loss and gradients of 8 modes with position errors
        _case("adam256_term", "term", 256, 8, 512, 2048, pos_error=1.5),
        # batched serving: reconstructions of uneven size and window, replayed as one graph
        _case("serve_epoch", "serve", 0, 1, 0, 0, windows="64,128,192,256", counts_of="100,2000,400,900",
              positions_of="2500,1400,900,700"),
        # orthogonal probe relaxation over 8 eigenmodes, weights updated
        _case("relaxed192_epoch", "opr", 192, 1, 900, 1024, K=8, counts=3000.0),
        # multislice gradients (4 slices of 2048^2, 4 modes), incident waves kept
        _case("slices256_term", "ms_term", 256, 4, 256, 2048, S=4),
        # multislice LSQML with a ragged last minibatch
        _case("slices128_epoch", "ms_epoch", 128, 2, 777, 900, S=3, batch=128),
        # gradients with the split-BF16 far field on the tensor cores
        _case("split128_term", "term", 128, 5, 1024, 1024, precision="bf16x3"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["forward", "term", "epoch", "epoch", "opr", "ms_term", "ms_epoch", "split", "serve"])
    noise = rng.choice(["gaussian", "poisson"])
    if kind == "serve":
        n = rng.randint(2, 5)
        Ns = [rng.choice([64, 128, 192, 256]) for _ in range(n)]
        Js = [_log_int(rng, 300, 1200) for _ in range(n)]
        return _case(None, "serve", 0, 1, 0, 0, noise=noise, windows=",".join(map(str, Ns)),
                     counts_of=",".join(str(_log_int(rng, 100, 3000)) for _ in range(n)),
                     positions_of=",".join(map(str, Js)))
    N = rng.choice([32, 64, 128] if kind == "split" else [16, 32, 64, 64, 128, 128, 192, 256])
    S = rng.randint(2, 4) if kind.startswith("ms") else 1
    M = rng.choice([1, 1, 2, 3, 4] if kind in ("opr", "ms_term", "ms_epoch") else [1, 1, 2, 3, 5, 8])
    # positions, log-uniform, within the work (points of all modes and slices) of the largest listed case
    most = min(4096, int(1.2e8 / (N * N * M * S)))
    J = _log_int(rng, 16, max(17, most))
    side = N + 16 + int(rng.uniform(0.5, 3.0) * N * min(5.0, 1.0 + math.sqrt(J) / 32.0))
    H, W = side + rng.randint(0, 64), side + rng.randint(0, 64)
    c = dict(S=S, noise=noise, batch=min(J, rng.choice([64, 100, 128, 256])), counts=float(_log_int(rng, 3e3, 1e6)))
    if kind == "opr":
        c["K"] = rng.randint(1, 8)
    if kind == "split":
        kind, c["precision"] = "term", "bf16x3"
    if kind == "epoch":
        c["compact"], c["positions"] = rng.random() < 0.3, rng.random() < 0.3
    if kind == "term" and rng.random() < 0.5:
        c["pos_error"] = 1.5
    return _case(None, kind, N, M, J, H, W, **c)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _object(H, W, gen, dev, amp_lo=0.8, phase_max=0.5):
    amp = amp_lo + (1.0 - amp_lo) * torch.rand(H, W, generator=gen, device=dev)
    fy, fx = torch.fft.fftfreq(H, device=dev)[:, None], torch.fft.fftfreq(W, device=dev)[None]
    blur = torch.exp(-2.0 * (math.pi * 3.0) ** 2 * (fy * fy + fx * fx))
    ph = torch.fft.ifft2(torch.fft.fft2(torch.randn(H, W, generator=gen, device=dev)) * blur).real
    return torch.polar(amp, ph * (phase_max / ph.abs().max()))


def _modes(N, powers, dev):
    """Orthonormal Hermite-Gaussian modes of the given power fractions (waist N/5, quadratic phase)."""
    a = torch.arange(N, dtype=torch.float64, device=dev) - N / 2
    y, x = a[:, None], a[None]
    r2, s = y * y + x * x, math.sqrt(2.0) * 5.0 / N
    h = [torch.ones_like, lambda t: 2 * t, lambda t: 4 * t * t - 2]
    raw = torch.stack([h[m](s * y) * h[n](s * x) * torch.exp(-r2 * (5.0 / N) ** 2) for m, n in HG[:len(powers)]])
    q, _ = torch.linalg.qr(raw.reshape(len(powers), -1).T)
    p = torch.tensor(powers, dtype=torch.float64, device=dev)
    q = (q.T * torch.sqrt(p / p.sum())[:, None]).reshape(len(powers), N, N)
    return (q * torch.polar(torch.ones_like(r2), 1.28 / N * r2)).to(torch.complex64)


def _spiral(J, N, H, W, dev):
    n = torch.arange(J, dtype=torch.float64, device=dev)
    r = ((min(H, W) - N) / 2 - 6) * torch.sqrt(n / max(J, 1))
    th = n * math.radians(137.508)
    return torch.stack([H / 2 + r * torch.sin(th), W / 2 + r * torch.cos(th)], 1).float()


def _clip(pos, N, H, W):
    hi = torch.tensor([H - N / 2 - MARGIN, W - N / 2 - MARGIN], dtype=pos.dtype, device=pos.device)
    return torch.minimum(pos.clamp(min=N / 2), hi).contiguous()


def _problem(c, gen, dev):
    """True model, counts drawn from it, and the estimate a reconstruction starts from."""
    N, M, J, H, W = c["N"], c["M"], c["J"], c["H"], c["W"]
    S, K = c.get("S", 1), c.get("K", 0)
    O = torch.stack([_object(H, W, gen, dev, 0.8 ** (1.0 / S), 0.5 / S) for _ in range(S)])
    pos = _spiral(J, N, H, W, dev)
    p = {"noise": c["noise"], "eps": EPS, "batch": c["batch"], "S": S, "K": K}
    if K:
        P = _modes(N, [1.0] + [0.3 * 0.6 ** k for k in range(K - 1)], dev)
        w = 1.0 + 0.1 * torch.randn(J, K, generator=gen, device=dev)
        rest = _modes(N, [0.3 * 0.5 ** k for k in range(M - 1)], dev) * 0.3 if M > 1 else None
        p["U"], p["w_true"], p["rest"] = P, w, rest
    else:
        P, w, rest = _modes(N, [0.5 ** k for k in range(M)], dev), None, None
    I = torch.empty(J, N, N, device=dev)
    Hf = _propagator(N, dev).to(torch.complex64) if S > 1 else None
    step = max(1, int(3e7 / (N * N * M)))
    for j in range(0, J, step):
        I[j:j + step] = _intensity(O, _probe_of(P, w, rest, slice(j, j + step)), pos[j:j + step], Hf)
    scale = c["counts"] * J / I.double().sum().item()
    p["meas"] = torch.poisson(I * scale, generator=gen)
    if K:
        p["U"] = p["U"] * math.sqrt(scale)
        p["rest"] = rest * math.sqrt(scale) if rest is not None else None
        p["w"] = torch.ones_like(w)
    else:
        p["probe"] = P * math.sqrt(scale)
    if c.get("pos_error"):
        pos = pos + c["pos_error"] * torch.randn(J, 2, generator=gen, device=dev)
    p["pos"] = _clip(pos, N, H, W)
    p["object"] = O if c["kind"] == "forward" else torch.ones_like(O)
    if c.get("positions") or c["kind"].endswith("term"):   # past the start: positions matter once there is structure
        p["object"] = torch.polar(torch.ones_like(O.abs()), 0.5 * O.angle())
    if S == 1:
        p["object"] = p["object"][0].contiguous()
    p["order"] = torch.randperm(J, generator=gen, device=dev).to(torch.int32)
    if c.get("compact"):   # minibatches of neighbours: strips of the scan, each walked along x
        strip = torch.floor(p["pos"][:, 0] / (N // 2))
        p["order"] = torch.argsort(strip * (4.0 * W) + p["pos"][:, 1]).to(torch.int32)
    p["compact"], p["positions"] = bool(c.get("compact")), bool(c.get("positions"))
    p["kind"], p["graph"], p["precision"] = c["kind"], bool(c.get("graph")), c.get("precision", "fp32")
    return p


def _parts(case):
    """The reconstructions of a case (several in a serving case)."""
    if case["kind"] != "serve":
        return [case]
    out = []
    for N, J, counts in zip(*([float(v) for v in case[k].split(",")] for k in ("windows", "positions_of", "counts_of"))):
        N, J = int(N), int(J)
        side = int(math.ceil(2 * (0.6 * 0.4 * N / math.sqrt(math.pi) * math.sqrt(J) + N / 2 + 2) / 32.0) * 32)
        out.append(_case(None, "epoch", N, 1, J, side, noise=case["noise"], counts=counts, graph=True))
    return out


def _inputs(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed))
    return [_problem(c, gen, dev) for c in _parts(case)]


def prepare(case, seed):
    parts = _inputs(case, seed)
    for p in parts:
        p.pop("w_true", None)
        p["opts"] = api.make_opts(p["noise"], batch=p["batch"], delta_o=DELTA, delta_p=DELTA, lam=LAM, eps=EPS,
                                  graph=p["graph"], update_positions=p["positions"],
                                  object_per_epoch=p["compact"], precision=p["precision"])
        if p["K"]:
            p["opr"] = api.make_opr_opts(p["K"])
        if p["S"] > 1:
            p["ms"] = api.make_multislice(p["S"], DZ, WAVELENGTH, PIXEL)
        if p["kind"] in ("term", "ms_term"):
            for k in ("object", "probe", "pos"):
                p[k].requires_grad_(True)
        if p["kind"] == "forward":
            del p["meas"]
    return {"kind": case["kind"], "parts": parts}


def run(state):
    if state["kind"] == "serve":
        recons = [(p["object"], p["probe"], p["pos"], p["meas"], p["order"]) for p in state["parts"]]
        losses = api.lsqml_epoch_batched(recons, [p["opts"] for p in state["parts"]], check=False)
        return {"losses": losses, "objects": [r[0] for r in recons], "probes": [r[1] for r in recons]}
    p, kind = state["parts"][0], state["kind"]
    if kind == "forward":
        return {"intensity": api.forward(p["object"], p["probe"], p["pos"], check=False)}
    if kind in ("term", "ms_term"):
        for k in ("object", "probe", "pos"):
            p[k].grad = None
        if kind == "term":
            loss = autograd.data_term(p["object"], p["probe"], p["pos"], p["meas"], p["noise"], EPS, p["precision"])
        else:
            loss = autograd.data_term_ms(p["object"], p["probe"], p["pos"], p["meas"], p["ms"], p["noise"], EPS)
        loss.backward()
        return {"loss": loss.detach(), "object": p["object"].grad, "probe": p["probe"].grad, "pos": p["pos"].grad}
    if kind == "epoch":
        loss, _ = api.lsqml_epoch(p["object"], p["probe"], p["pos"], p["meas"], p["order"], p["opts"], check=False)
        out = {"loss": loss, "object": p["object"], "probe": p["probe"]}
        if p["positions"]:
            out["pos"] = p["pos"]
        return out
    if kind == "opr":
        loss, _ = api.lsqml_epoch_opr(p["object"], p["U"], p["w"], p["rest"], p["pos"], p["meas"], p["order"],
                                      p["opts"], p["opr"], check=False)
        out = {"loss": loss, "object": p["object"], "U": p["U"], "w": p["w"]}
        if p["rest"] is not None:
            out["rest"] = p["rest"]
        return out
    loss, _ = api.lsqml_epoch_ms(p["object"], p["probe"], p["pos"], p["meas"], p["order"], p["ms"], p["opts"],
                                 check=False)
    return {"loss": loss, "object": p["object"], "probe": p["probe"]}


def work(case):
    """Inputs read once, outputs written once; 5 n log2 n operations per transform of n points
    plus the pointwise products of every mode and slice."""
    nbytes = flops = 0.0
    for c in _parts(case):
        N, M, J, S, K, kind = c["N"], c["M"], c["J"], c.get("S", 1), c.get("K", 0), c["kind"]
        n, o = N * N, c["H"] * c["W"] * S
        probe = n * (K + M - 1 if K else M)
        nbytes += 4.0 * J * n + 8.0 * J + 16.0 * (o + probe) + (8.0 * J * K if K else 0.0)
        if kind == "forward":
            nbytes -= 8.0 * (o + probe)
        transforms = 1 + 2 * (S - 1)
        if kind != "forward":
            transforms *= 2
        if kind == "ms_epoch":
            transforms += 4 * (S - 1)
        flops += J * n * (M * (transforms * 10.0 * math.log2(N) + 40.0 * S) + 30.0 * K)
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------
# The same calls in 64 bits
# ---------------------------------------------------------------------------
def _propagator(N, dev):
    f = torch.fft.fftfreq(N, d=PIXEL, dtype=torch.float64, device=dev)
    f2 = f[:, None] ** 2 + f[None] ** 2
    il = 1.0 / WAVELENGTH
    inside = f2 < il * il
    kz = torch.sqrt(torch.where(inside, il * il - f2, torch.zeros_like(f2)))
    Hf = torch.polar(torch.ones_like(f2), 2 * math.pi * DZ * (-f2 / (kz + il)))
    return torch.where(inside, Hf, torch.zeros_like(Hf))


def _fft(x):
    return torch.fft.fft2(x, norm="ortho")


def _ifft(x):
    return torch.fft.ifft2(x, norm="ortho")


def _tiles(pos, N, W):
    """Flat indices of the (N+1)^2 object tiles and the bilinear fractions."""
    r = pos - N / 2
    t = torch.floor(r)
    f = (r - t)[:, :, None, None]
    a = torch.arange(N + 1, device=pos.device)
    t = t.long()
    return (t[:, 0, None, None] + a[:, None]) * W + t[:, 1, None, None] + a, f[:, 0], f[:, 1]


def _extract(O, tiles):
    """Patches of one plane, and their derivatives in the position."""
    idx, fy, fx = tiles
    v = O.reshape(-1)[idx]
    a, b, c, d = v[:, :-1, :-1], v[:, :-1, 1:], v[:, 1:, :-1], v[:, 1:, 1:]
    o = (1 - fy) * ((1 - fx) * a + fx * b) + fy * ((1 - fx) * c + fx * d)
    return o, (1 - fx) * (c - a) + fx * (d - b), (1 - fy) * (b - a) + fy * (d - c)


def _scatter(into, patch, tiles):
    """into += sum_j S_j^T patch_j."""
    idx, fy, fx = tiles
    tile = torch.zeros(idx.shape, dtype=patch.dtype, device=patch.device)
    for dy in (0, 1):
        for dx in (0, 1):
            wy, wx = (fy if dy else 1 - fy), (fx if dx else 1 - fx)
            tile[:, dy:tile.shape[1] - 1 + dy, dx:tile.shape[2] - 1 + dx] += wy * wx * patch
    if patch.is_complex():
        torch.view_as_real(into).reshape(-1, 2).index_add_(0, idx.reshape(-1), torch.view_as_real(tile).reshape(-1, 2))
    else:
        into.reshape(-1).index_add_(0, idx.reshape(-1), tile.reshape(-1))


def _probe_of(P, w, rest, j):
    """Modes per position [B or 1, M, N, N]."""
    if w is None:
        return P[None]
    p0 = torch.einsum("bk,kyx->byx", w[j].to(P.dtype), P)[:, None]
    return p0 if rest is None else torch.cat([p0, rest[None].expand(p0.shape[0], -1, -1, -1)], 1)


def _waves(O, P, tiles, Hf):
    """Exit waves of the last slice, each slice's incident waves and (patch, derivatives)."""
    inc, patches, psi = [], [], P
    for s in range(O.shape[0]):
        if s:
            psi = _ifft(Hf * _fft(psi))
        inc.append(psi)
        patches.append(_extract(O[s], tiles))
        psi = psi * patches[s][0][:, None]
    return psi, inc, patches


def _intensity(O, P, pos, Hf):
    psi, _, _ = _waves(O, P, _tiles(pos, P.shape[-1], O.shape[-1]), Hf)
    return _fft(psi).abs().square().sum(1)


def _dot(a, b, dims):
    return (a.conj() * b).real.sum(dims)


def _solve(a11, a12, a22, b1, b2):
    tr = 0.5 * LAM * (a11 + a22)
    a11, a22 = a11 + tr, a22 + tr
    det = a11 * a22 - a12 * a12
    one = torch.ones_like(det)

    def lone(b, a):
        return torch.where(a > 0, b / torch.where(a > 0, a, one), torch.zeros_like(b))

    safe = torch.where(det > 0, det, one)
    return (torch.where(det > 0, (a22 * b1 - a12 * b2) / safe, lone(b1, a11)),
            torch.where(det > 0, (a11 * b2 - a12 * b1) / safe, lone(b2, a22)))


def _data(I, meas, noise):
    """Loss, dL/dI and the exit-wave factor rho - 1."""
    Ie = I + EPS
    if noise == "gaussian":
        rho = torch.sqrt(meas) / torch.sqrt(Ie)
        return (torch.sqrt(Ie) - torch.sqrt(meas)).square().sum(), 1 - rho, rho - 1
    return (I - meas * torch.log(Ie)).sum(), 1 - meas / Ie, 0.5 * (meas / Ie - 1)


def _exact_term(p, O, P, pos, Hf):
    N, W = P.shape[-1], O.shape[-1]
    gO, gP, gr = torch.zeros_like(O), torch.zeros_like(P), torch.zeros_like(pos)
    loss = torch.zeros((), dtype=torch.float64, device=O.device)
    step = max(1, int(2e7 / (N * N * P.shape[0] * O.shape[0])))
    for j in range(0, pos.shape[0], step):
        tiles = _tiles(pos[j:j + step], N, W)
        psi, inc, patches = _waves(O, P[None], tiles, Hf)
        Psi = _fft(psi)
        val, dI, _ = _data(Psi.abs().square().sum(1), p["meas"][j:j + step].double(), p["noise"])
        loss += val
        g = _ifft(2 * dI[:, None] * Psi)
        for s in reversed(range(O.shape[0])):
            o, dy, dx = patches[s]
            go = (inc[s].conj() * g).sum(1)
            _scatter(gO[s], go, tiles)
            gr[j:j + step, 0] += _dot(go, dy, (1, 2))
            gr[j:j + step, 1] += _dot(go, dx, (1, 2))
            g = o.conj()[:, None] * g
            if s:
                g = _ifft(Hf.conj() * _fft(g))
        gP += g.sum(0)
    return {"loss": loss, "object": gO if p["S"] > 1 else gO[0], "probe": gP, "pos": gr}


def _exact_epoch(p, O, P, pos, Hf):
    """One LSQML epoch (any number of slices; with K > 0 a relaxed primary mode)."""
    S, H, W = O.shape
    K, N, noise = p["K"], P.shape[-1], p["noise"]
    w = p["w"].double() if K else None
    rest = p["rest"].to(P.dtype) if K and p["rest"] is not None else None
    order = p["order"].long()
    loss = torch.zeros((), dtype=torch.float64, device=O.device)
    O_epoch = torch.zeros_like(O)
    for b in range(0, order.shape[0], p["batch"]):
        idx = order[b:b + p["batch"]]
        tiles = _tiles(pos[idx], N, W)
        Pj = _probe_of(P, w, rest, idx)
        psi, inc, patches = _waves(O, Pj, tiles, Hf)
        Psi = _fft(psi)
        val, _, fac = _data(Psi.abs().square().sum(1), p["meas"][idx].double(), noise)
        loss += val
        chi = last = _ifft(fac[:, None] * Psi)
        acc, ill = torch.zeros_like(O), torch.zeros(O.shape, dtype=torch.float64, device=O.device)
        g = [None] * S
        for s in reversed(range(S)):
            g[s] = (inc[s].conj() * chi).sum(1)
            _scatter(acc[s], g[s], tiles)
            _scatter(ill[s], inc[s].abs().square().sum(1).expand(len(idx), N, N), tiles)
            entry = chi
            chi = patches[s][0].conj()[:, None] * chi
            if s:
                chi = _ifft(Hf.conj() * _fft(chi))
        o = patches[0][0]
        o2 = o.abs().square()
        Dp = o2.sum(0)
        damp = Dp.max()
        if K:
            D = torch.einsum("bk,byx->kyx", w[idx].square(), o2)
            damp = torch.maximum(damp, D.max())
            dU = torch.einsum("bk,byx->kyx", w[idx].to(P.dtype), chi[:, 0]) / (D + DELTA * damp)
            drest = chi[:, 1:].sum(0) / (Dp + DELTA * damp)
            dP = _probe_of(dU, w, drest if rest is not None else None, idx)
        else:
            dP = (chi.sum(0) / (Dp + DELTA * damp))[None]
        ill = ill + DELTA * ill.reshape(S, -1).max(1).values[:, None, None]
        dirs = [_extract(acc[s] / ill[s], tiles)[0][:, None] for s in range(S)]
        u, v = dirs[0] * Pj, o[:, None] * dP
        for s in range(1, S):
            u = _ifft(Hf * _fft(u)) * patches[s][0][:, None] + inc[s] * dirs[s]
            v = _ifft(Hf * _fft(v)) * patches[s][0][:, None]
        d3 = (1, 2, 3)
        aO, aP = _solve(_dot(u, u, d3), _dot(u, v, d3), _dot(v, v, d3), _dot(u, last, d3), _dot(v, last, d3))
        upd = torch.zeros_like(O)
        for s in range(S):
            _scatter(upd[s], aO[:, None, None] * g[s], tiles)
        upd = upd / ill
        if p["positions"]:
            dy, dx = patches[0][1:]
            Sp = Pj.abs().square().sum(1)
            d2 = (1, 2)
            sy, sx = _solve((Sp * dy.abs().square()).sum(d2), (Sp * (dy.conj() * dx).real).sum(d2),
                            (Sp * dx.abs().square()).sum(d2), _dot(dy, g[0], d2), _dot(dx, g[0], d2))
            pos[idx] = _clip(pos[idx] + torch.stack([sy, sx], 1).clamp(-1.0, 1.0), N, H, W)
        if K:
            dw = _weights(P, o2, entry[:, 0], o, w.shape[1])
            w[idx] += dw
            P = P + aP.mean() * dU
            rest = rest + aP.mean() * drest if rest is not None else None
        else:
            P = P + aP.mean() * dP[0]
        if p["compact"]:
            O_epoch += upd
        else:
            O = O + upd
    O = O + O_epoch
    out = {"loss": loss, "object": O if S > 1 else O[0]}
    if K:
        out.update({"U": P, "w": w})
        if rest is not None:
            out["rest"] = rest
        return out
    out["probe"] = P
    if p["positions"]:
        out["pos"] = pos
    return out


def _weights(U, o2, chi0, o, K):
    """Damped least-squares fit of the primary mode's exit-wave change by the eigenmodes' exit waves."""
    n = U.shape[-1] ** 2
    prod = torch.stack([(U[m].conj() * U[k]).real for m in range(K) for k in range(K)]).reshape(K * K, n)
    A = (o2.reshape(-1, n) @ prod.T).reshape(-1, K, K)
    b = ((o.conj() * chi0).reshape(-1, n) @ U.conj().reshape(K, n).T).real
    damp = LAM * A.diagonal(dim1=1, dim2=2).sum(1) / K
    return torch.linalg.solve(A + damp[:, None, None] * torch.eye(K, dtype=A.dtype, device=A.device), b[:, :, None])[:, :, 0]


def exact(case, seed):
    got = []
    for p in _inputs(case, seed):
        O = p["object"].to(torch.complex128).reshape(p["S"], p["object"].shape[-2], -1)
        P = p["U" if p["K"] else "probe"].to(torch.complex128)
        pos = p["pos"].double()
        Hf = _propagator(P.shape[-1], O.device) if p["S"] > 1 else None
        if p["kind"] == "forward":
            step = max(1, int(2e7 / P.numel()))
            got.append({"intensity": torch.cat([_intensity(O, P[None], pos[j:j + step], Hf)
                                                for j in range(0, pos.shape[0], step)])})
        elif p["kind"] in ("term", "ms_term"):
            got.append(_exact_term(p, O, P, pos, Hf))
        else:
            got.append(_exact_epoch(p, O, P, pos, Hf))
    if case["kind"] != "serve":
        return got[0]
    return {"losses": torch.stack([g["loss"] for g in got]), "objects": [g["object"] for g in got],
            "probes": [g["probe"] for g in got]}

"""The work that a user of this library has it do, as measured cases.

Every case is one call sequence of a forecast-analysis program: it holds an ensemble, data,
perturbations (or a seed) and rhat on the device, a plan, and calls the analysis; or it trains the
learned-spectrum network.  Analyses update the ensemble in place, as in use; the ensemble is the
output.  Fields are stationary Gaussian fields drawn from a seeded generator on the device.

``exact`` computes the same outputs in FP64 with torch alone: unitary DFTs of the whole fields, the
sample spectra, the gains and the update of eq. (spectral-multi-enkf), the DST-I by odd extension,
the bilinear morphing, the network by autograd, Philox4x32-10 in integer arithmetic.
"""

from __future__ import annotations

import math

import torch

from paper_1001_1588_gb300 import abi, torch_api

DEV = "cuda"
LINES = (16, 24, 32, 48, 64, 96, 128, 192, 256, 384, 512, 768, 1024, 1536, 2048, 3072, 4096)
SIDES = (64, 96, 128, 192, 256, 384, 512, 768, 1024)
ELLS = (8.0, 8.0 * 16.0 ** (1 / 3), 8.0 * 16.0 ** (2 / 3), 128.0)   # Matern-3/2 lengths, geometric 8..128
DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}
SIZE = {"f32": 4, "bf16": 2}


def listed():
    return [
        # the smallest real call: one 64 x 64 field, five members, everything observed; a program on a
        # coarse grid calls this every few model steps and waits for it
        _analysis("plain_64", 64, 64, 5, "f32", "1", "flat"),
        # a three-variable model state on 512 x 512 with the paper's ensemble size, one variable observed
        _analysis("plain_3x512", 512, 512, 5, "f32", "100", "flat"),
        # the headline analysis: four variables on 4096 x 4096, 20 members, two observed, BF16 storage
        _analysis("large_4x4096_bf16", 4096, 4096, 20, "bf16", "1100", "inverse"),
        # a 3 * 2^a grid (the other supported family of sizes), BF16, odd member count
        _analysis("ragged_3x1536x768_bf16", 1536, 768, 25, "bf16", "100", "flat"),
        # the morphing filter's extended state (T_x, T_y, r^(1), r^(2)) on a wide domain: three observed of
        # four, FP32, odd member count
        _analysis("extended_4x1024x2048_f32", 1024, 2048, 15, "f32", "1110", "flat"),
        # perturbations drawn by the library instead of passed in
        dict(_analysis("seeded_4x2048_bf16", 2048, 2048, 20, "bf16", "1100", "inverse"), kind="seeded"),
        # two observed variables coupled through their cross-covariance
        dict(_analysis("coupled_3x2048_bf16", 2048, 2048, 20, "bf16", "110", "inverse"), kind="coupled"),
        # the paper's real sine transform: a grid with boundary nodes that keep the forecast
        dict(_analysis("sine_4x1025_bf16", 1025, 1025, 20, "bf16", "1100", "flat"), kind="sine"),
        # 256 independent analyses of uneven sizes in one call
        {"name": "batched_256", "kind": "batched", "count": 256, "max_side": 1024, "storage": "f32"},
        # the morphing transform of the members, the new reference and the inverse transform
        {"name": "morph_2x2048", "kind": "morph", "ny": 2048, "nx": 2048, "blocks": 2, "members": 20, "n_iter": 20,
         "tol": 1e-5},
        # the analysis with a learned spectrum: plain estimate, network, analysis with the returned table
        {"name": "learned_1024", "kind": "learned", "ny": 1024, "nx": 1024, "members": 5},
        # one training step of that network: gradient of a batch of 256 pairs and the Adam update
        {"name": "train_256", "kind": "train", "batch": 256},
    ]


def _analysis(name, ny, nx, members, storage, observed, rhat):
    return {"name": name, "kind": "analysis", "ny": ny, "nx": nx, "members": members, "storage": storage,
            "observed": observed, "rhat": rhat}


# ------------------------------------------------------------------ drawn cases
def _log_choice(rng, values, lo, hi):
    """One of the ascending ``values`` in [lo, hi], spread over the logarithm of their range."""
    v = [x for x in values if lo <= x <= hi]
    x = math.exp(rng.uniform(math.log(v[0]) - 0.2, math.log(v[-1]) + 0.2))
    return min(v, key=lambda c: abs(math.log(c / x)))


def draw(rng):
    kind = rng.choice(("analysis", "analysis", "analysis", "analysis", "analysis", "seeded", "coupled", "sine",
                       "batched", "morph", "learned", "train"))
    if kind == "train":
        return {"kind": kind, "batch": int(round(math.exp(rng.uniform(math.log(4), math.log(2048)))))}
    if kind == "batched":
        return {"kind": kind, "count": int(round(math.exp(rng.uniform(math.log(8), math.log(256))))),
                "max_side": rng.choice((192, 384, 768, 1024)), "storage": rng.choice(("f32", "bf16"))}
    if kind == "morph":
        ny, nx = (int(round(math.exp(rng.uniform(math.log(61), math.log(2500))))) for _ in range(2))
        return {"kind": kind, "ny": ny, "nx": nx, "blocks": rng.randint(1, 3), "members": rng.randint(2, 20),
                "n_iter": 20, "tol": rng.choice((1e-5, 1e-4))}
    if kind == "learned":
        return {"kind": kind, "ny": _log_choice(rng, LINES, 64, 2048), "nx": _log_choice(rng, LINES, 64, 2048),
                "members": 5}
    while True:
        M = rng.randint(1, 4)
        n_obs = rng.randint(1, min(M, 2)) if (kind != "analysis" or rng.random() < 0.85) else M
        mask = [1] * n_obs + [0] * (M - n_obs)
        rng.shuffle(mask)
        c = {"kind": kind, "ny": _log_choice(rng, LINES, 48, 4096), "nx": _log_choice(rng, LINES, 48, 4096),
             "members": rng.randint(3, 25), "storage": rng.choice(("f32", "bf16")),
             "observed": "".join(map(str, mask)), "rhat": rng.choice(("flat", "inverse"))}
        if kind == "sine":
            c["ny"], c["nx"] = min(c["ny"], 2048) + 1, min(c["nx"], 2048) + 1
        # at most a quarter of the largest listed case's ensemble points (the sine form works on 4x the
        # points), and one column's tables and staged innovations within a plan's limits
        points = c["ny"] * c["nx"] * M * c["members"] * (4 if kind == "sine" else 1)
        col = c["ny"] * (2 if kind == "sine" else 1)
        tables = n_obs + 2 * n_obs * (M - n_obs) + (2 if kind == "coupled" and n_obs == 2 else 0)
        if (points <= 4096 * 4096 * 80 // 4 and col * (4 * tables + 16.5) <= 226 * 1024
                and col * (16 * n_obs + 8.5) <= 226 * 1024):
            return c


# ------------------------------------------------------------------ inputs
def _xi2(ny, nx):
    ky = torch.fft.fftfreq(ny, device=DEV, dtype=torch.float64)[:, None]
    kx = torch.fft.rfftfreq(nx, device=DEV, dtype=torch.float64)[None, :]
    return ky ** 2 + kx ** 2


def _unit(S, nx):
    """S scaled to mean 1 over the full grid (a field of point variance 1)."""
    w = torch.full((S.shape[-1],), 2.0, dtype=S.dtype, device=DEV)
    w[0] = w[-1] = 1.0
    return S / ((S * w).sum() / (S.shape[0] * nx))


def _matern(ny, nx, ell):
    return _unit((3.0 / ell ** 2 + 4.0 * math.pi ** 2 * _xi2(ny, nx)) ** -2.5, nx)


def _se(ny, nx, ell):
    return _unit(torch.exp(-2.0 * math.pi ** 2 * ell ** 2 * _xi2(ny, nx)), nx)


def _field(amp, z):
    """F^-1(amp F z) of white fields z [..., ny, nx], amp the square root of the spectrum."""
    Z = torch.fft.rfft2(z, norm="ortho")
    Z *= amp
    return torch.fft.irfft2(Z, s=z.shape[-2:], norm="ortho")


def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _rhat(kind, n_obs, ny, nx):
    if kind == "flat":
        return torch.full((n_obs, ny, nx // 2 + 1), 0.1, dtype=torch.float64, device=DEV)
    k = torch.sqrt((torch.fft.fftfreq(ny, device=DEV, dtype=torch.float64)[:, None] * ny) ** 2
                   + torch.arange(nx // 2 + 1, device=DEV, dtype=torch.float64)[None, :] ** 2)
    return (0.1 / torch.clamp(k, min=1.0))[None].repeat(n_obs, 1, 1).contiguous()


def _periodic_inputs(case, seed, ny, nx):
    """Matern-3/2 blocks correlated through a shared latent field (0.6), data = a further draw plus
    noise of spectrum rhat, perturbations of spectrum rhat."""
    g, dt, N = _generator(seed), DTYPES[case["storage"]], case["members"]
    obs = [i for i, o in enumerate(case["observed"]) if o == "1"]
    M = len(case["observed"])
    amp = [_matern(ny, nx, ELLS[b]).sqrt().float() for b in range(M)]
    rhat = _rhat(case["rhat"], len(obs), ny, nx)
    sr = rhat[0].sqrt().float()
    ens = torch.empty(M, N, ny, nx, dtype=dt, device=DEV)
    truth = torch.empty(M, ny, nx, device=DEV)
    for k in range(N + 1):
        z0 = torch.randn(ny, nx, device=DEV, generator=g)
        for b in range(M):
            u = _field(amp[b], 0.6 * z0 + 0.8 * torch.randn(ny, nx, device=DEV, generator=g))
            (truth[b] if k == N else ens[b, k]).copy_(u)
    data = torch.stack([truth[o] + _field(sr, torch.randn(ny, nx, device=DEV, generator=g)) for o in obs])
    pert = torch.empty(N, len(obs), ny, nx, dtype=dt, device=DEV)
    for k in range(N):
        pert[k] = _field(sr, torch.randn(len(obs), ny, nx, device=DEV, generator=g))
    return {"ensemble": ens, "data": data.contiguous(), "perturbations": pert, "rhat": rhat}


def _batched_shapes(case):
    """Shapes of the batch: sides up to max_side, square or 2:1, 5..25 members (fixed by the case alone)."""
    import random
    rng = random.Random(20260004)
    sides = [s for s in SIDES if s <= case["max_side"]]
    out = []
    for _ in range(case["count"]):
        s = rng.choice(sides)
        ny = s if rng.random() < 0.5 else s // 2
        out.append((ny, s, rng.randint(5, 25), math.exp(rng.uniform(math.log(2), math.log(64))),
                    math.exp(rng.uniform(math.log(0.01), 0.0))))
    return out


def _batched_inputs(case, seed):
    g, dt, shapes = _generator(seed), DTYPES[case["storage"]], _batched_shapes(case)
    sizes = [N * ny * nx for ny, nx, N, _, _ in shapes]           # multiples of 16 elements
    flat = torch.empty(sum(sizes), dtype=dt, device=DEV)          # one buffer for all ensembles
    items, at = [], 0
    for (ny, nx, N, ell, r), n in zip(shapes, sizes):
        ens = flat[at:at + n].view(N, ny, nx)
        at += n
        u = _field(_se(ny, nx, ell).sqrt().float(), torch.randn(N + 1, ny, nx, device=DEV, generator=g))
        ens.copy_(u[:N])
        noise = math.sqrt(r) * torch.randn(N + 1, ny, nx, device=DEV, generator=g)
        items.append({"ensemble": ens, "data": (u[N] + noise[N]).contiguous(), "perturbations": noise[:N].to(dt),
                      "rhat": torch.full((ny, nx // 2 + 1), r, dtype=torch.float64, device=DEV)})
    return flat, items


def _sine_inputs(case, seed):
    """Fields on ny x nx nodes with zero change wanted on the boundary: cut out of a periodic draw of twice the size."""
    ny, nx = case["ny"], case["nx"]
    s = _periodic_inputs(dict(case, rhat="flat"), seed, 2 * (ny - 1), 2 * (nx - 1))
    for name in ("ensemble", "data", "perturbations"):
        s[name] = s[name][..., :ny, :nx].contiguous()
    s["rhat"] = torch.full((len(s["data"]), ny - 2, nx - 2), 0.1, dtype=torch.float64, device=DEV)
    if case["rhat"] == "inverse":
        a = torch.arange(1, ny - 1, device=DEV, dtype=torch.float64)[:, None]
        b = torch.arange(1, nx - 1, device=DEV, dtype=torch.float64)[None, :]
        s["rhat"] = (0.1 / torch.sqrt(a ** 2 + b ** 2))[None].repeat(len(s["data"]), 1, 1).contiguous()
    return s


def _morph_inputs(case, seed):
    """Smooth members, reference and displacements of up to 3 cells (squared-exponential, 20 cells)."""
    g, ny, nx, M, K = _generator(seed), case["ny"], case["nx"], case["blocks"], case["members"]
    py, px = ny + ny % 2, nx + nx % 2
    amp = _se(py, px, 20.0).sqrt().float()

    def smooth(out):
        z = torch.randn(out.shape[0], py, px, device=DEV, generator=g)
        out.copy_(_field(amp, z)[:, :ny, :nx])

    u = torch.empty(M, K, ny, nx, device=DEV)
    ext = torch.empty(M + 2, K, ny, nx, device=DEV)
    u_ref = torch.empty(M, ny, nx, device=DEV)
    smooth(u_ref)
    for k in range(K):
        smooth(u[:, k])
        smooth(ext[:2, k])
    ext[:2] *= 3.0 / ext[:2].abs().amax(dim=(2, 3), keepdim=True)
    ext[2:] = 0.0
    return {"u": u, "u_ref": u_ref, "ext": ext, "ext_ref": torch.empty(M + 2, ny, nx, device=DEV),
            "u_out": torch.empty(M, K, ny, nx, device=DEV)}


LAYERS = ((256, 64), (64, 64), (64, 64), (64, 128))


def _network(g):
    """Weights of the size a trained network has, [W1, b1, ..., W4, b4] flat."""
    parts = []
    for i, o in LAYERS:
        parts += [(torch.rand(o * i, device=DEV, generator=g) * 2 - 1) * math.sqrt(3.0 / i),
                  0.1 * torch.randn(o, device=DEV, generator=g)]
    return torch.cat(parts)


def _train_inputs(case, seed):
    """A batch of features and targets, and Adam's state some way into a training."""
    g, B = _generator(seed), case["batch"]
    p = _network(g)
    return {"params": p, "m": 1e-3 * torch.randn(p.shape, device=DEV, generator=g),
            "v": 1e-5 * (0.1 + torch.rand(p.shape, device=DEV, generator=g)),
            "x": torch.randn(B, 256, device=DEV, generator=g), "y": torch.randn(B, 128, device=DEV, generator=g),
            "grads": torch.empty_like(p), "loss": torch.empty(1, device=DEV), "step": 100}


def _learned_inputs(case, seed):
    g, ny, nx, N = _generator(seed), case["ny"], case["nx"], case["members"]
    S = _unit((1.0 + 4.0 * math.pi ** 2 * 64.0 * _xi2(ny, nx)) ** -1.5, nx)   # power law, 8 cells, slope -3
    u = _field(S.sqrt().float(), torch.randn(N + 1, ny, nx, device=DEV, generator=g))
    noise = math.sqrt(0.1) * torch.randn(N + 1, 1, ny, nx, device=DEV, generator=g)
    return {"ensemble": u[None, :N].contiguous(), "data": (u[N:] + noise[N]).contiguous(), "perturbations": noise[:N].contiguous(),
            "rhat": torch.full((1, ny, nx // 2 + 1), 0.1, dtype=torch.float64, device=DEV), "params": _network(g)}


class _Batch:
    """The batched plan's handle and workspace, released with the state."""

    def __init__(self, case):
        self.handle = abi.fftenkf_plan_batched([(ny, nx, N) for ny, nx, N, _, _ in _batched_shapes(case)],
                                               abi.FFTENKF_F32 if case["storage"] == "f32" else abi.FFTENKF_BF16)
        self.ws = torch.empty(abi.fftenkf_batch_workspace_size(self.handle), dtype=torch.uint8, device=DEV)

    def __del__(self):
        abi.fftenkf_batch_destroy(self.handle)


class _Denoiser:
    def __init__(self, case):
        self.handle = abi.fftenkf_denoiser_create(case["ny"], case["nx"], case["members"])

    def __del__(self):
        abi.fftenkf_denoiser_destroy(self.handle)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batched":
        flat, items = _batched_inputs(case, seed)
        lists = {n: [it[n] for it in items] for n in items[0]}
        return {"kind": kind, "flat": flat, "items": lists, "batch": _Batch(case)}
    if kind == "morph":
        return {"kind": kind, "case": case, **_morph_inputs(case, seed)}
    if kind == "train":
        return {"kind": kind, "batch": case["batch"], **_train_inputs(case, seed)}
    if kind == "learned":
        s = _learned_inputs(case, seed)
        plan = torch_api.Plan(case["ny"], case["nx"], 1, case["members"], torch.float32, [1])
        table = torch.empty(plan.spectrum_doubles, dtype=torch.float64, device=DEV)
        plan.workspace(DEV)
        return {"kind": kind, "case": case, "plan": plan, "denoiser": _Denoiser(case), "plain": table,
                "learned": torch.empty_like(table), **s}
    observed = [int(o) for o in case["observed"]]
    shape = (case["ny"], case["nx"], len(observed), case["members"], DTYPES[case["storage"]], observed)
    if kind == "sine":
        return {"kind": kind, "plan": torch_api.SinePlan(*shape), **_sine_inputs(case, seed)}
    s = _periodic_inputs(case, seed, case["ny"], case["nx"])
    plan = torch_api.Plan(*shape, coupled=(kind == "coupled"))
    plan.workspace(DEV)
    return {"kind": kind, "plan": plan, "seed": int(seed) + 77, **s}


# ------------------------------------------------------------------ one pass
def run(state):
    kind = state["kind"]
    if kind == "batched":
        it, b = state["items"], state["batch"]
        abi.fftenkf_analyze_batched(b.handle, it["ensemble"], it["data"], it["perturbations"], it["rhat"], b.ws, _stream())
        return state["flat"]
    if kind == "morph":
        c, s = state["case"], _stream()
        M, K, ny, nx = c["blocks"], c["members"], c["ny"], c["nx"]
        abi.fftenkf_morph_forward(state["u"], state["u_ref"], state["ext"], M, K, ny, nx, c["n_iter"], c["tol"], s)
        abi.fftenkf_morph_reference(state["ext"], state["ext_ref"], M + 2, K, ny, nx, s)
        abi.fftenkf_morph_inverse(state["ext"], state["u_ref"], state["u_out"], M, K, ny, nx, s)
        return {"ext": state["ext"], "ext_ref": state["ext_ref"], "u_out": state["u_out"]}
    if kind == "train":
        t, s = state, _stream()
        abi.fftenkf_mlp_gradient(t["params"], t["x"], t["y"], t["batch"], t["grads"], t["loss"], s)
        t["step"] += 1
        abi.fftenkf_mlp_adam(t["params"], t["m"], t["v"], t["grads"], t["step"], 1e-3, s)
        return {n: t[n] for n in ("params", "m", "v", "grads", "loss")}
    plan = state["plan"]
    if kind == "seeded":
        return plan.analyze_seeded(state["ensemble"], state["data"], state["rhat"], state["seed"])
    if kind == "learned":
        plan.estimate_spectrum(state["ensemble"], state["plain"])
        abi.fftenkf_denoise_spectrum(state["denoiser"].handle, state["params"], state["plain"], state["learned"],
                                     state["case"]["members"], _stream(), want_flag=False)
        return plan.analyze(state["ensemble"], state["data"], state["perturbations"], state["rhat"], state["learned"])
    return plan.analyze(state["ensemble"], state["data"], state["perturbations"], state["rhat"])


def _stream():
    return int(torch.cuda.current_stream().cuda_stream)


# ------------------------------------------------------------------ what a pass cannot do without
def _analysis_work(ny, nx, M, N, n_obs, s, drawn=False):
    """Ensemble in and out, perturbations, data and rhat in; forward transforms of every member and
    innovation, inverse ones of every increment (5 G log2 G / 2 each, real), 8 flops per product."""
    G, K = ny * nx, ny * (nx // 2 + 1)
    nbytes = 2 * M * N * G * s + n_obs * G * 4 + n_obs * K * 8 + (0 if drawn else N * n_obs * G * s)
    flops = (2 * M + n_obs) * N * 2.5 * G * math.log2(G) + 8.0 * K * N * n_obs * (2 * M)
    return nbytes, flops


def work(case):
    kind = case["kind"]
    if kind == "batched":
        w = [_analysis_work(ny, nx, 1, N, 1, SIZE[case["storage"]]) for ny, nx, N, _, _ in _batched_shapes(case)]
        return {"bytes": sum(x[0] for x in w), "flops": sum(x[1] for x in w)}
    if kind == "train":
        # the batch, parameters, moments in; gradients, parameters, moments out; three products per weight
        P, B = sum(i * o + o for i, o in LAYERS), case["batch"]
        return {"bytes": 4 * (7 * P + B * (256 + 128)), "flops": 6.0 * B * P}
    ny, nx, N = case["ny"], case["nx"], case["members"]
    if kind == "morph":
        # forward: T and the members in, residuals out; reference: its channels' means out; inverse: members out
        M, G = case["blocks"], ny * nx
        return {"bytes": 4 * G * (2 * N + 3 * M * N + M + M + 2), "flops": 11.0 * G * N * (2 * M + 2)}
    if kind == "learned":
        b, f = _analysis_work(ny, nx, 1, N, 1, 4)
        return {"bytes": b, "flops": f}
    M, n_obs = len(case["observed"]), case["observed"].count("1")
    b, f = _analysis_work(ny, nx, M, N, n_obs, SIZE[case["storage"]], kind == "seeded")
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ the same in 64 bits
def _update(ens, data, pert, rhat, fwd, inv, spectrum=None, coupled=False, add=None, observed=(1,)):
    """The analysis of eq. (spectral-multi-enkf) with forward and inverse transforms fwd, inv (FP64).
    spectrum: the observed auto tables in place of the estimate (one block); add(k, i): a term added
    to the innovation coefficients instead of perturbations."""
    M, N = ens.shape[:2]
    obs = [j for j in range(M) if observed[j]]
    mean = [ens[j].double().mean(0) for j in range(M)]
    auto, cross = {}, {}
    for k in range(N if spectrum is None else 0):
        A = [fwd(ens[j, k].double() - mean[j]) for j in range(M)]
        for i in obs:
            for j in range(M):
                if j == i:
                    auto[i] = auto.get(i, 0) + A[i].abs() ** 2 / (N - 1)
                elif coupled or j not in obs:
                    cross[j, i] = cross.get((j, i), 0) + A[j] * A[i].conj() / (N - 1)
    if spectrum is not None:
        auto = {i: spectrum[n] for n, i in enumerate(obs)}
    r = {i: rhat[n] for n, i in enumerate(obs)}
    gain = {}
    if coupled and len(obs) == 2:
        p, q = obs
        a, d, b = auto[p] + r[p], auto[q] + r[q], cross[q, p]
        det = a * d - b.abs() ** 2
        for j in range(M):
            cp = auto[p] if j == p else cross[j, p]
            cq = auto[q] if j == q else cross[j, q]
            gain[j, p] = (cp * d - cq * b) / det
            gain[j, q] = (cq * a - cp * b.conj()) / det
    else:
        for i in obs:
            gain[i, i] = auto[i] / (auto[i] + r[i])
            for j in range(M):
                if j not in obs:
                    gain[j, i] = cross[j, i] / (auto[i] + r[i])
    out = torch.empty(ens.shape, dtype=torch.float64, device=DEV)
    for k in range(N):
        W = {}
        for n, i in enumerate(obs):
            w = data[n].double() - ens[i, k].double()
            W[i] = fwd(w if add is not None else w + pert[k, n].double())
            if add is not None:
                W[i] = W[i] + add(k, n)
        for j in range(M):
            S = sum(gain[j, i] * W[i] for i in obs if (j, i) in gain)
            out[j, k] = ens[j, k].double() + inv(S)
    return out


def _periodic(ny, nx):
    return (lambda x: torch.fft.rfft2(x, norm="ortho")), (lambda X: torch.fft.irfft2(X, s=(ny, nx), norm="ortho"))


def _dst(x, dim):
    """Orthonormal DST-I along dim, from the DFT of the odd extension."""
    m = x.shape[dim]
    z = torch.zeros_like(x.narrow(dim, 0, 1))
    Y = torch.fft.rfft(torch.cat([z, x, z, -x.flip(dim)], dim), dim=dim)
    return Y.narrow(dim, 1, m).imag * (-0.5 * math.sqrt(2.0 / (m + 1)))


def _exact_sine(s, observed):
    full = s["ensemble"].double()
    cut = slice(1, -1)
    both = lambda x: _dst(_dst(x, 0), 1)   # noqa: E731  (its own inverse)
    full[..., cut, cut] = _update(s["ensemble"][..., cut, cut], s["data"][..., cut, cut], s["perturbations"][..., cut, cut],
                                  s["rhat"], both, both, observed=observed)
    return full


def _mulhilo(a, b):
    p = a * b
    return (p >> 32) & 0xFFFFFFFF, p & 0xFFFFFFFF


def _philox(c, seed):
    """Philox4x32-10 of the counter words c (int64 tensors below 2^32) under the 64-bit key."""
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    for _ in range(10):
        h0, l0 = _mulhilo(c[0], 0xD2511F53)
        h1, l1 = _mulhilo(c[2], 0xCD9E8D57)
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def _normals(wa, wb):
    ua, ub = (((w >> 8).double() + 0.5) * 2.0 ** -24 for w in (wa, wb))
    return torch.polar(torch.sqrt(-2.0 * torch.log(ua)), 2.0 * math.pi * ub)


def _white(ny, nx, stream, seed):
    """The half spectrum of white noise that the seeded analysis draws (counters of include/fftenkf.h)."""
    L, h = nx // 2, math.sqrt(0.5)
    ky = torch.arange(ny // 2, device=DEV)[:, None].expand(-1, L - 1)
    kx = torch.arange(1, L, device=DEV)[None, :].expand(ny // 2, -1)
    zero = torch.zeros_like(ky)
    w = _philox([ky, kx, zero + stream, zero], seed)
    out = torch.empty(ny, L + 1, dtype=torch.complex128, device=DEV)
    out[:ny // 2, 1:L] = h * _normals(w[0], w[1])
    out[ny // 2:, 1:L] = h * _normals(w[2], w[3])
    k = torch.arange(ny, device=DEV)
    m = torch.minimum(k, (ny - k) % ny)
    for c in (0, L):
        w = _philox([m, torch.full_like(m, c), torch.full_like(m, stream), torch.zeros_like(m)], seed)
        n = _normals(w[0], w[1])
        z = torch.where(2 * k > ny, n.conj(), n) * h
        out[:, c] = torch.where((k == 0) | (2 * k == ny), n.real.to(n.dtype), z)
    return out


def _interp(f, dy, dx):
    """f [ny][nx] at the nodes displaced by (dy, dx), bilinear and periodic."""
    ny, nx = f.shape
    fy, fx = torch.floor(dy), torch.floor(dx)
    wy, wx = dy - fy, dx - fx
    y0 = (torch.arange(ny, device=DEV)[:, None] + fy.long()) % ny
    x0 = (torch.arange(nx, device=DEV)[None, :] + fx.long()) % nx
    y1, x1 = (y0 + 1) % ny, (x0 + 1) % nx
    g = f.reshape(-1)
    return ((1 - wy) * ((1 - wx) * g[y0 * nx + x0] + wx * g[y0 * nx + x1])
            + wy * ((1 - wx) * g[y1 * nx + x0] + wx * g[y1 * nx + x1]))


def _exact_morph(case, s):
    M, K = case["blocks"], case["members"]
    ext, u, u_ref = s["ext"].double(), s["u"], s["u_ref"].double()
    out = torch.empty(u.shape, dtype=torch.float64, device=DEV)
    for k in range(K):
        tx, ty = ext[0, k], ext[1, k]
        dy, dx = torch.zeros_like(tx), torch.zeros_like(tx)
        moving = torch.ones_like(tx, dtype=torch.bool)
        for _ in range(case["n_iter"]):
            nx_, ny_ = -_interp(tx, dy, dx), -_interp(ty, dy, dx)
            still = ((nx_ - dx).abs() <= case["tol"]) & ((ny_ - dy).abs() <= case["tol"])
            dx, dy = torch.where(moving, nx_, dx), torch.where(moving, ny_, dy)
            moving &= ~still
        for j in range(M):
            ext[2 + j, k] = _interp(u[j, k].double(), dy, dx) - u_ref[j]
            out[j, k] = _interp(u_ref[j] + ext[2 + j, k], ty, tx)
    return {"ext": ext, "ext_ref": ext.mean(1), "u_out": out}


def _layers(flat):
    """(W, b) of every layer in FP64, the weights rounded to BF16 as the forward pass uses them."""
    out, at = [], 0
    for i, o in LAYERS:
        out += [flat[at:at + i * o].bfloat16().double().view(o, i), flat[at + i * o:at + i * o + o].double()]
        at += i * o + o
    return out


def _mlp(layers, x):
    for n in range(0, len(layers), 2):
        x = (x if n == 0 else torch.nn.functional.gelu(x)) @ layers[n].T + layers[n + 1]
    return x


def _exact_train(s):
    layers = [t.requires_grad_() for t in _layers(s["params"])]
    loss = ((_mlp(layers, s["x"].double()) - s["y"].double()) ** 2).mean()
    loss.backward()
    g = torch.cat([t.grad.reshape(-1) for t in layers])
    step = s["step"] + 1
    m = 0.9 * s["m"].double() + 0.1 * g
    v = 0.999 * s["v"].double() + 0.001 * g * g
    p = s["params"].double() - 1e-3 * (m / (1 - 0.9 ** step)) / (torch.sqrt(v / (1 - 0.999 ** step)) + 1e-8)
    return {"params": p, "m": m, "v": v, "grads": g, "loss": loss.detach().reshape(1)}


def _exact_learned(case, s):
    ny, nx, N = case["ny"], case["nx"], case["members"]
    fwd, inv = _periodic(ny, nx)
    u = s["ensemble"][0].double()
    chat = (fwd(u - u.mean(0)).abs() ** 2).sum(0) / (N - 1)
    ky = torch.fft.fftfreq(ny, device=DEV, dtype=torch.float64)[:, None] * ny
    kabs = torch.sqrt(ky ** 2 + torch.arange(nx // 2 + 1, device=DEV, dtype=torch.float64)[None, :] ** 2)
    width = math.sqrt(ny * ny + nx * nx) / 256.0
    bins = torch.clamp(torch.floor(kabs / width), max=127).long().reshape(-1)
    top = chat.max()
    logs = torch.log(torch.clamp(chat / top, min=1e-30)).reshape(-1)
    count = torch.bincount(bins, minlength=128)
    v = torch.zeros(128, dtype=torch.float64, device=DEV).index_add_(0, bins, logs) / count.clamp(min=1) + torch.log(top)
    v = torch.where(count > 0, v, torch.zeros_like(v))
    centre = torch.clamp((torch.arange(128, device=DEV, dtype=torch.float64) + 0.5) * width, min=0.5).log()
    x = _mlp(_layers(s["params"]), torch.cat([v - v.mean(), centre])[None])[0] + v.mean()
    pos = torch.clamp(kabs / width - 0.5, 0.0, 127.0)
    lo = torch.clamp(pos.long(), max=126)
    learned = torch.exp(x[lo] + (pos - lo) * (x[lo + 1] - x[lo]))
    return _update(s["ensemble"], s["data"], s["perturbations"], s["rhat"], fwd, inv, spectrum=[learned])


def exact(case, seed):
    kind = case["kind"]
    if kind == "batched":
        flat, items = _batched_inputs(case, seed)
        out, at = torch.empty(flat.shape, dtype=torch.float64, device=DEV), 0
        for it in items:
            e = it["ensemble"]
            fwd, inv = _periodic(*e.shape[-2:])
            out[at:at + e.numel()] = _update(e[None], it["data"][None], it["perturbations"][:, None], it["rhat"][None],
                                             fwd, inv).reshape(-1)
            at += e.numel()
        return out
    if kind == "morph":
        return _exact_morph(case, _morph_inputs(case, seed))
    if kind == "train":
        return _exact_train(_train_inputs(case, seed))
    if kind == "learned":
        return _exact_learned(case, _learned_inputs(case, seed))
    observed = [int(o) for o in case["observed"]]
    if kind == "sine":
        return _exact_sine(_sine_inputs(case, seed), observed)
    ny, nx = case["ny"], case["nx"]
    s = _periodic_inputs(case, seed, ny, nx)
    fwd, inv = _periodic(ny, nx)
    add = None
    if kind == "seeded":
        amp = s["rhat"].sqrt()
        add = lambda k, n: amp[n] * _white(ny, nx, k * len(amp) + n, int(seed) + 77)   # noqa: E731
    return _update(s["ensemble"], s["data"], s["perturbations"], s["rhat"], fwd, inv, coupled=(kind == "coupled"), add=add,
                   observed=observed)

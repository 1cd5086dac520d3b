"""The cases whose speed this repository is measured by, through its public entry points.

The library verifies windows of drafted diffusion steps (``api.verify``, once or as a
pipelined run, and ``api.log_ratios``) and runs whole samplers on an analytic mixture
(``api.sampler_run``, ``api.em_sample``).  The listed cases are the shapes of the
repository's own workloads and tests, single images and odd sizes among them; ``draw``
gives more of the same ranges.  Inputs follow workloads.py's recipes (means N(0, 1),
target mean sigma |Delta| away along a random direction, the draft drawn from the draft
kernel) and are made on the GPU from the seed alone.

``exact`` restates the method in 64 bits in plain torch: Philox4x32-10 and Box-Muller,
the log ratios, sample and block verification, the residual's 1-D draw by bisection, the
residual, reflection and bonus steps, the mixture score, the drafter and the round loop.
"""
import math

import torch

from paper_2606_13426_gb300 import api

DEV = "cuda"

# Sampler schedule and mixture recipe: workloads.SAMPLER_CONFIG (variance-preserving
# schedule, churn 0.5, component means N(0, 4 I), Dirichlet(1) weights, unit variance).
CHURN, BETA_MIN, BETA_MAX, T_FLOOR, COMP_VAR = 0.5, 0.1, 20.0, 1e-4, 1.0


def _verify(name, B, L, d, dtype="f32", mode="block", residual="decomposition", delta="uniform",
            schedule="cosine", ragged=False, bonus=False, omega=1.0, windows=1, kind="verify"):
    return dict(name=name, kind=kind, B=B, L=L, d=d, dtype=dtype, mode=mode, residual=residual,
                delta=delta, schedule=schedule, ragged=ragged, bonus=bonus, omega=omega,
                windows=windows)


def _sampler(name, B, L, d, K, C, mode="block", drafter="free", max_rounds=0):
    """max_rounds = 0: until every chain has reached step K."""
    return dict(name=name, kind="sampler", B=B, L=L, d=d, K=K, C=C, mode=mode, drafter=drafter,
                max_rounds=max_rounds)


def listed():
    return [
        # the smallest call: a handful of short chains, all latency and launches
        _verify("verify_tiny", 4, 4, 16),
        # one latent image at a time (4 x 64 x 64, the paper's window of 7): an interactive user
        _verify("verify_one_image", 1, 7, 16384),
        # one batch of 32 x 32 x 3 images, the verification between two network calls
        _verify("verify_pixel", 256, 8, 3072),
        # the same batches from several generators, verified as a captured pipelined run
        _verify("run_pixel", 256, 8, 3072, windows=8, kind="run"),
        # latent windows (4 x 64 x 64) in bf16, as a captured pipelined run
        _verify("run_latent", 64, 16, 16384, "bf16", delta="gamma", windows=8, kind="run"),
        # the log ratios of latent windows alone, for a caller with an acceptance rule of its own
        _verify("ratios_latent", 64, 16, 16384, "bf16", delta="gamma", kind="ratios"),
        # large images (256 x 256 x 3), a long window: the largest read
        _verify("verify_highres", 16, 32, 196608, schedule="linear"),
        # an odd image size (75 x 75 x 3 bf16: rows that start on no 16-byte boundary),
        # sample verification
        _verify("verify_odd", 24, 7, 16875, "bf16", mode="sample"),
        # a serving engine's batch: chains at different places of their schedules (shorter
        # last windows, finished chains) over 56 x 56 x 3 images, the bonus step's mean given
        _verify("verify_serving", 96, 7, 9408, ragged=True, bonus=True),
        # the speculative sampler at the repository's sampler workload, its first rounds
        # (a step budget; chains that flip at a tie stay close to each other that long)
        _sampler("sampler_rounds", 1024, 8, 1024, 1000, 8, max_rounds=8),
        # a small sampling run from start to end: short schedule, Frozen drafter, sample mode
        _sampler("sampler_small", 16, 4, 256, 50, 8, mode="sample", drafter="frozen"),
        # the plain chain that speculative sampling is compared with
        dict(name="em_chain", kind="em", B=1024, d=1024, K=100, C=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["verify", "verify", "verify", "run", "ratios", "sampler", "em"])
    if kind in ("verify", "run", "ratios"):
        dtype = rng.choice(["f32", "bf16"])
        windows = 8 if kind == "run" else 1
        most = (100_000_000 if dtype == "f32" else 130_000_000) // windows
        d = _log_int(rng, 16, 200_000)
        if rng.random() < 0.6:                    # whole images: a multiple of 64
            d = max(64, d // 64 * 64)
        if 11_500 < d <= 12_288:                  # rows that the first measured version cannot launch
            d -= 1024
        L = rng.randint(1, 32)
        while L * d > most:
            L = max(1, L // 2)
        B = _log_int(rng, 1, max(1, min(512, most // (L * d))))
        mode = "block" if kind == "ratios" else rng.choice(["block", "sample"])
        residual = "reflection" if mode == "sample" and kind != "ratios" and rng.random() < 0.3 else "decomposition"
        more = kind == "verify" and rng.random() < 0.4
        c = _verify("", B, L, d, dtype, mode, residual, rng.choice(["uniform", "gamma"]),
                    rng.choice(["cosine", "linear"]), more, more,
                    1.1 if more and rng.random() < 0.3 else 1.0, windows, kind)
    elif kind == "sampler":
        d = _log_int(rng, 32, 2048)
        if rng.random() < 0.7:
            d = max(32, d // 32 * 32)
        B = _log_int(rng, 4, max(8, min(1024, (1 << 20) // d)))
        c = _sampler("", B, rng.choice([2, 4, 5, 8]), d, rng.choice([100, 250, 1000]), rng.randint(2, 12),
                     rng.choice(["block", "sample"]), rng.choice(["free", "frozen"]), rng.randint(2, 8))
    else:
        d = _log_int(rng, 32, 2048)
        if rng.random() < 0.7:
            d = max(32, d // 32 * 32)
        B = _log_int(rng, 4, max(8, min(1024, (1 << 20) // d)))
        c = dict(kind="em", B=B, d=d, K=rng.randint(20, 100), C=rng.randint(2, 12))
    c.pop("name", None)
    return c


# ---------------------------------------------------------------- inputs

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(1_000_003 * int(seed) + 7)
    return g


def _window(case, g):
    """One window's tensors: x_draft, mu_target, mu_draft, sigma and the options."""
    B, L, d = case["B"], case["L"], case["d"]
    dt = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
    f = dict(device=DEV, generator=g)
    j = torch.arange(L, device=DEV, dtype=torch.float64) / max(L - 1, 1)
    if case["schedule"] == "cosine":
        row = 0.05 + 0.95 * 0.5 * (1.0 + torch.cos(math.pi * j))
    else:
        row = 1.0 + (0.01 - 1.0) * j
    # chains stand at places of their own in the schedule
    sigma = (row[None] * (0.75 + 0.5 * torch.rand(B, 1, **f))).float().contiguous()
    if case["delta"] == "uniform":
        dn = 3.0 * torch.rand(B, L, 1, **f)
    else:                                         # Gamma(shape 2, scale 0.5)
        dn = -0.5 * (torch.rand(2, B, L, 1, **f).clamp_min(1e-7).log().sum(0))
    w = {"sigma": sigma}
    u = torch.randn(B, L, d, **f)
    scale = sigma[:, :, None] * dn / u.norm(dim=-1, keepdim=True)
    mp = torch.randn(B, L, d, **f)
    w["mq"] = torch.addcmul(mp, u, scale, value=-1.0).to(dt)
    torch.randn(B, L, d, out=u, **f)
    w["x"] = torch.addcmul(mp, u, sigma[:, :, None]).to(dt)
    w["mp"] = mp.to(dt)
    if case["ragged"]:
        le = torch.full((B,), L, dtype=torch.int32, device=DEV)
        short = torch.rand(B, **f) < 0.25
        w["L_eff"] = torch.where(short, torch.randint(0, L + 1, (B,), dtype=torch.int32, **f), le).contiguous()
    if case["bonus"]:
        w["mqb"] = torch.randn(B, d, **f).to(dt)
        w["sgb"] = (0.05 + 0.9 * torch.rand(B, **f)).contiguous()
    return w


def _outputs(case):
    """Output buffers that a program keeps; zeroed once (a finished chain's rows are not written)."""
    B, L, d = case["B"], case["L"], case["d"]
    dt = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
    return dict(accepted_len=torch.zeros(B, dtype=torch.int32, device=DEV), y=torch.zeros(B, d, dtype=dt, device=DEV),
                status=torch.zeros(B, dtype=torch.int32, device=DEV), log_ratio=torch.zeros(B, L, device=DEV),
                delta_norm=torch.zeros(B, L, device=DEV), aux=torch.zeros(B, 4, device=DEV))


def _mixture(case, g):
    means = 2.0 * torch.randn(case["C"], case["d"], device=DEV, generator=g)
    e = -torch.rand(case["C"], device=DEV, generator=g).clamp_min(1e-7).log()
    return means, (e / e.sum()).log()


def _call(case, w, seed, ws, out, pipelined=False):
    return api.verify(w["x"], w["mq"], w["mp"], w["sigma"], seed, case["mode"], L_eff=w.get("L_eff"),
                      mu_target_bonus=w.get("mqb"), sigma_bonus=w.get("sgb"), residual=case["residual"],
                      omega=case["omega"], with_aux=True, workspace=ws, out=out, pipelined=pipelined)


def prepare(case, seed):
    g = _gen(seed)
    st = dict(case=case, seed=12345 + int(seed))
    kind = case["kind"]
    if kind in ("verify", "run", "ratios"):
        dt = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
        st["w"] = [_window(case, g) for _ in range(case["windows"])]
        st["ws"] = api.make_workspace(case["B"], case["L"], case["d"], dt)
        if kind != "ratios":
            st["out"] = [_outputs(case) for _ in range(case["windows"])]
        if kind == "run":                         # a serving loop captures its run once
            def calls():
                return [_call(case, w, st["seed"] + i, st["ws"], st["out"][i], pipelined=True)
                        for i, w in enumerate(st["w"])]
            side = torch.cuda.Stream()
            side.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(side):
                calls()
            torch.cuda.current_stream().wait_stream(side)
            torch.cuda.synchronize()
            st["graph"] = torch.cuda.CUDAGraph()
            with torch.cuda.graph(st["graph"], stream=side):
                st["res"] = calls()
    else:
        means, logw = _mixture(case, g)
        st["target"] = api.GmmTarget(means, logw, COMP_VAR, case["K"], CHURN, BETA_MIN, BETA_MAX, T_FLOOR)
        if kind == "sampler":
            n = api.B.sdv_sampler_workspace_bytes(case["B"], case["L"], case["d"])
            st["ws"] = torch.empty(n, dtype=torch.uint8, device=DEV)
    return st


def run(st):
    case, kind = st["case"], st["case"]["kind"]
    if kind == "verify":
        return _call(case, st["w"][0], st["seed"], st["ws"], st["out"][0])
    if kind == "run":
        st["graph"].replay()
        return st["res"]
    if kind == "ratios":
        w = st["w"][0]
        return api.log_ratios(w["x"], w["mq"], w["mp"], w["sigma"], workspace=st["ws"])
    if kind == "sampler":
        return api.sampler_run(case["B"], case["L"], st["target"], st["seed"], case["mode"], case["drafter"],
                               max_rounds=case["max_rounds"] or None, workspace=st["ws"])
    return api.em_sample(case["B"], st["target"], st["seed"])


def work(case):
    kind, B, d = case["kind"], case["B"], case["d"]
    if kind in ("verify", "run", "ratios"):
        L, s, n = case["L"], 4 if case["dtype"] == "f32" else 2, case["windows"]
        rows = 0.875 * L if case["ragged"] else L   # a quarter of the windows half as long
        by = 3 * B * rows * d * s + 3 * B * L * 4
        if kind != "ratios":
            by += B * d * s * (2 if case["bonus"] else 1) + 28 * B
        return {"bytes": n * by, "flops": n * 6 * B * rows * d}
    C = case["C"]
    row = d * (6 * C + 12)                        # mixture score and mean of one state
    step = 60 * d                                 # one step's Philox block and Box-Muller share, and the update
    if kind == "em":
        return {"bytes": 4 * (B * d + C * d), "flops": B * case["K"] * (row + step)}
    L = case["L"]
    rounds = case["max_rounds"] or max(1, round(case["K"] / (0.7 * L)))
    return {"bytes": 4 * (B * d + C * d) + 12 * B, "flops": B * rounds * ((L + 1) * row + L * (step + 6 * d) + step)}


def tolerance(case):
    kind = case["kind"]
    if kind == "sampler":
        # a chain with a coin at its threshold may go either way, and its state differs from
        # then on by what a few steps' noise makes (measured with one such chain of 1024
        # against 64 bits: 4.3e-3); without one the states are within 2e-6
        return {"rel": 0.02, "max": 0.9, "differ": 0.01}
    if kind == "em":
        # measured against 64 bits: 8e-7, and 8e-6 where a chain passes between two
        # components, which amplifies the rounding of its squared distances
        return {"rel": 4e-5, "max": 1.6e-3}
    if case["dtype"] == "bf16" and kind != "ratios":
        return {"rel": 1e-3, "max": 1e-2, "differ": 0.01}   # y is stored in bf16: one ulp where its rounding flips
    return {"rel": 1e-5, "max": 4e-4, "differ": 0.01}


# ---------------------------------------------------------------- the method in 64 bits

M32 = 0xFFFFFFFF
STREAM_COIN, STREAM_U, STREAM_RESID, STREAM_BONUS, STREAM_DRAFT, STREAM_INIT, STREAM_EM = range(7)


def _mul32(a, b):
    """(high, low) words of the 64-bit product of a 32-bit constant and 32-bit values held in int64."""
    pl, ph = a * (b & 0xFFFF), a * (b >> 16)
    return (ph + (pl >> 16)) >> 16, (pl + ((ph & 0xFFFF) << 16)) & M32


def _philox(seed, c0, c1, c2, c3):
    c0, c1 = torch.broadcast_tensors(c0, c1)
    c2, c3 = torch.full_like(c0, c2), torch.full_like(c0, c3)
    k0, k1 = seed & M32, (seed >> 32) & M32
    for _ in range(10):
        h0, l0 = _mul32(0xD2511F53, c0)
        h1, l1 = _mul32(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c0, c1, c2, c3


def _unif(w):
    return (w.double() + 0.5) * 2.0 ** -32


def _normals(seed, b, d, stream, sub):
    """[len(b), d] normals of chains b: counter (b, i/4, stream, sub), Box-Muller on the word pairs."""
    i = torch.arange((d + 3) // 4, device=b.device)
    w = [_unif(v) for v in _philox(seed, b[:, None], i[None], stream, sub)]
    z = []
    for p in (0, 2):
        r = torch.sqrt(-2.0 * torch.log(w[p]))
        z += [r * torch.cos(2 * math.pi * w[p + 1]), r * torch.sin(2 * math.pi * w[p + 1])]
    return torch.stack(z, -1).reshape(len(b), -1)[:, :d]


def _log1mexp(x):
    x = x.clamp_max(0.0)
    return torch.where(x > -math.log(2.0), torch.log(-torch.expm1(x)), torch.log1p(-torch.exp(x)))


_lphi = torch.special.log_ndtr


def _log_v(D, la):
    """log v = log(alpha Phi(a+) - Phi(a-)), a+- = log alpha / D +- D / 2."""
    ap = la / D + 0.5 * D
    A = la + _lphi(ap)
    return A + _log1mexp(_lphi(ap - D) - A)


def _draw_u(D, la, w):
    """U with Psi(U) = w, Psi(u) = (alpha Phi(u) - Phi(u - D)) / v, by bisection in t = a+ - u."""
    ap, lv, lw = la / D + 0.5 * D, _log_v(D, la), torch.log(w)

    def below(t):
        u = ap - t
        A = la + _lphi(u)
        return A + _log1mexp(_lphi(u - D) - A) - lv < lw

    lo, hi = torch.zeros_like(D), torch.full_like(D, 1e-3)
    for _ in range(60):
        hi = torch.where(below(hi), hi, 2 * hi)
    for _ in range(90):
        mid = 0.5 * (lo + hi)
        b = below(mid)
        lo, hi = torch.where(b, lo, mid), torch.where(b, mid, hi)
    return ap - 0.5 * (lo + hi)


def _accept(ell, dn, g, seed, mode, omega=1.0):
    """tau (1-based) and log alpha_{tau-1} of each chain; g [B] window lengths."""
    B, L = ell.shape
    dev = ell.device
    b, j = torch.arange(B, device=dev), torch.arange(L, device=dev)
    leta = torch.log(_unif(_philox(seed, b[:, None], j[None], STREAM_COIN, 0)[0]))
    live = j[None] < g[:, None]
    e = torch.where(live, ell / omega ** 2, torch.zeros_like(ell))
    if mode == "sample":
        fail = live & ~(leta < e.clamp_max(0.0))
        first = torch.where(fail, j[None], torch.full_like(live, L, dtype=torch.int64)).amin(1)
        return torch.where(fail.any(1), first + 1, g + 1), torch.zeros(B, device=dev, dtype=torch.float64)
    la = torch.zeros(B, L + 1, device=dev, dtype=torch.float64)
    for k in range(L):
        la[:, k + 1] = (la[:, k] + e[:, k]).clamp_max(0.0)
    succ = torch.zeros(B, L, dtype=torch.bool, device=dev)
    for k in range(L):
        a = la[:, k + 1]
        nxt = dn[:, k + 1] if k + 1 < L else torch.ones_like(a)
        D = torch.where(nxt > 0, nxt, torch.ones_like(nxt))
        lv = _log_v(D, a)
        lh = lv - torch.logaddexp(lv, _log1mexp(a))
        lh = torch.where((a < 0) & (nxt <= 0), torch.full_like(a, -math.inf), lh)
        lh = torch.where(a >= 0, torch.zeros_like(a), lh)
        lh = torch.where(g == k + 1, a, lh)
        succ[:, k] = leta[:, k] < lh
    last = torch.where(succ & live, j[None] + 1, torch.zeros_like(live, dtype=torch.int64)).amax(1)
    return last + 1, la.gather(1, last[:, None])[:, 0]


def _verify64(case, w, seed):
    """The outputs of one call in 64 bits, chain by chain groups (whole windows in 64 bits would not fit)."""
    B, L, d = case["B"], case["L"], case["d"]
    S1 = torch.empty(B, L, device=DEV, dtype=torch.float64)
    S2 = torch.empty_like(S1)
    for b in range(0, B, max(1, 50_000_000 // (L * d))):
        c = slice(b, b + max(1, 50_000_000 // (L * d)))
        dl = w["mp"][c].double() - w["mq"][c].double()
        S2[c] = dl.square().sum(-1)
        S1[c] = (w["x"][c].double() - w["mp"][c].double()).mul_(dl).sum(-1)
        del dl
    sg = w["sigma"].double()
    ell, dn = -(S1 + 0.5 * S2) / sg ** 2, S2.sqrt() / sg
    g = w["L_eff"].long() if "L_eff" in w else torch.full((B,), L, device=DEV)
    live = torch.arange(L, device=DEV)[None] < g[:, None]
    ell, dn = torch.where(live, ell, torch.zeros_like(ell)), torch.where(live, dn, torch.zeros_like(dn))
    if case["kind"] == "ratios":
        return ell, dn
    tau, la = _accept(ell, dn, g, seed, case["mode"], case["omega"])
    act, res = g > 0, tau <= g
    row = torch.where(res, tau - 1, (g - 1).clamp_min(0))
    at = torch.arange(B, device=DEV)
    x, mq, mp = (w[k][at, row].double() for k in ("x", "mq", "mp"))
    s, D = sg[at, row][:, None], dn[at, row]
    y = x.clone()
    nan = torch.full((B,), math.nan, device=DEV, dtype=torch.float64)
    U = nan.clone()
    if case["residual"] == "reflection":
        refl = x - (mp - mq) * (1.0 + 2.0 * S1[at, row] / S2[at, row])[:, None]
        y = torch.where(res[:, None], refl, y)
    else:
        ww = _unif(_philox(seed, at, torch.zeros_like(at), STREAM_U, 0)[0])
        Ds = torch.where(res & (D > 0), D, torch.ones_like(D))
        u = _draw_u(Ds, torch.where(res, la, torch.zeros_like(la)), ww)
        U = torch.where(res, u, nan)
        G = _normals(seed, at, d, STREAM_RESID, 0)
        e = (mp - mq) / (mp - mq).norm(dim=1, keepdim=True)
        r = mq + s * (G + e * (u - (e * G).sum(1))[:, None])
        y = torch.where(res[:, None], r, y)
    if case["bonus"]:
        yb = w["mqb"].double() + w["sgb"].double()[:, None] * _normals(seed, at, d, STREAM_BONUS, 0)
        y = torch.where(res[:, None], y, yb)
    y = torch.where(act[:, None], y, torch.zeros_like(y))
    aux = torch.stack([U, la, torch.where(res, D, nan), torch.where(res, s[:, 0], nan)], 1)
    aux = torch.where(act[:, None], aux, torch.zeros_like(aux))
    acc = torch.where(act, tau - 1, torch.zeros_like(tau)).int()
    return dict(accepted_len=acc, y=y, status=torch.zeros(B, dtype=torch.int32, device=DEV), log_ratio=ell,
                delta_norm=dn, aux=aux)


class _Target:
    """The analytic target: mean and score at generative steps k, in 64 bits."""

    def __init__(self, case, means, logw):
        self.K, self.mu, self.lw = case["K"], means.double(), logw.double()

    def beta(self, k):
        t = ((self.K - k).double() / self.K).clamp_min(T_FLOOR)
        return t, BETA_MIN + (BETA_MAX - BETA_MIN) * t

    def sigma(self, k):
        return math.sqrt(1.0 / self.K) * CHURN * self.beta(k)[1].sqrt()

    def drift(self, z, k, score):
        be = self.beta(k)[1][..., None]
        return z + (0.5 * be * z + 0.5 * (1 + CHURN ** 2) * be * score) / self.K

    def score(self, z, k):
        t, _ = self.beta(k)
        ab = torch.exp(-(BETA_MIN * t + 0.5 * (BETA_MAX - BETA_MIN) * t * t))
        v, sab = (ab * COMP_VAR + 1 - ab)[..., None], ab.sqrt()[..., None]
        d2 = torch.stack([(z - sab * m).square().sum(-1) for m in self.mu], -1)
        r = torch.softmax(self.lw - d2 / (2 * v), -1)
        return (sab * (r @ self.mu) - z) / v


def _splitmix(z):
    m = (1 << 64) - 1
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & m
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & m
    return z ^ (z >> 31)


def _sampler64(case, T, seed):
    B, L, d, K = case["B"], case["L"], case["d"], case["K"]
    b = torch.arange(B, device=DEV)
    y = _normals(seed, b, d, STREAM_INIT, 0)
    k = torch.zeros(B, dtype=torch.int64, device=DEV)
    rounds, tsum = torch.zeros_like(k), torch.zeros_like(k)
    sc = T.score(y, k)
    r = 0
    while r < (case["max_rounds"] or K) and bool((k < K).any()):
        rs = _splitmix((seed + (r + 1) * 0x9E3779B97F4A7C15) & ((1 << 64) - 1))
        g = torch.minimum(torch.full_like(k, L), K - k)
        if case["drafter"] == "frozen":
            sc = T.score(y, k)
        st, mp, mq, scs, sg = [y], [], [], [], []
        for j in range(L + 1):
            kj = torch.minimum(k + j, torch.full_like(k, K))
            scs.append(T.score(st[j], kj))
            mq.append(T.drift(st[j], kj, scs[j]))
            sg.append(T.sigma(kj))
            if j < L:
                mp.append(T.drift(st[j], kj, sc))
                st.append(mp[j] + sg[j][:, None] * _normals(rs, b, d, STREAM_DRAFT, j))
        ell, dn = [], []
        for j in range(L):
            dl = (mp[j] - mq[j]) / sg[j][:, None]
            z = (st[j + 1] - mp[j]) / sg[j][:, None]
            ell.append(-(z * dl).sum(-1) - 0.5 * dl.square().sum(-1))
            dn.append(dl.norm(dim=-1))
        live = torch.arange(L, device=DEV)[None] < g[:, None]
        ell, dn = (torch.where(live, torch.stack(v, 1), torch.zeros_like(live, dtype=torch.float64)) for v in (ell, dn))
        tau, la = _accept(ell, dn, g, rs, case["mode"])
        res = tau <= g
        st, mp, mq, scs, sg = (torch.stack(v, 1) for v in (st, mp, mq, scs, sg))
        row = torch.where(res, tau - 1, (g - 1).clamp_min(0))
        ww = _unif(_philox(rs, b, torch.zeros_like(b), STREAM_U, 0)[0])
        D = torch.where(res & (dn[b, row] > 0), dn[b, row], torch.ones_like(la))
        u = _draw_u(D, torch.where(res, la, torch.zeros_like(la)), ww)
        dl = mp[b, row] - mq[b, row]
        e = dl / dl.norm(dim=1, keepdim=True)
        G = _normals(rs, b, d, STREAM_RESID, 0)
        ny = mq[b, row] + sg[b, row][:, None] * (G + e * (u - (e * G).sum(1))[:, None])
        yb = mq[b, g] + sg[b, g][:, None] * _normals(rs, b, d, STREAM_BONUS, 0)
        end = (k + g >= K)[:, None]
        ny = torch.where(res[:, None], ny, torch.where(end, st[b, g], yb))
        act = g > 0
        y = torch.where(act[:, None], ny, y)
        sc = torch.where(act[:, None], scs[b, torch.minimum(tau, g)], sc)
        k = torch.where(act, torch.minimum(k + tau, torch.full_like(k, K)), k)
        rounds, tsum, r = rounds + act, tsum + torch.where(act, tau, torch.zeros_like(tau)), r + 1
    return dict(y=y, k=k.int(), chain_rounds=rounds.int(), tau_sum=tsum.int(), rounds=r)


def exact(case, seed):
    g, s = _gen(seed), 12345 + int(seed)
    kind = case["kind"]
    if kind == "run":
        return [_verify64(case, w, s + i) for i, w in enumerate([_window(case, g) for _ in range(case["windows"])])]
    if kind in ("verify", "ratios"):
        return _verify64(case, _window(case, g), s)
    T = _Target(case, *_mixture(case, g))
    if kind == "sampler":
        # of tens of thousands of coins one lies within rounding of its threshold in one run
        # of four, and its chain's state has no 64-bit value to be compared with
        if case["B"] * case["L"] * (case["max_rounds"] or case["K"] // case["L"] * 2) > 4000:
            return None
        return _sampler64(case, T, s)
    b = torch.arange(case["B"], device=DEV)
    y = _normals(s, b, case["d"], STREAM_INIT, 0)
    for k in range(case["K"]):
        kk = torch.full((1,), k, device=DEV)
        y = T.drift(y, kk, T.score(y, kk)) + T.sigma(kk) * _normals(s, b, case["d"], STREAM_EM, k)
    return y

"""The calls that users of this library make, as measurable cases.

A receiver trains a detector on the pilots of a frame, detects (or tracks through) its data
vectors and, where the detector sits inside a larger model, differentiates through it.  The
cases take those calls through the package's public entry points at the sizes of the test and
benchmark workloads: the smallest frame, the ordinary one, the largest blocks, ragged counts,
each contraction precision, and both directions.

Inputs follow the synthetic uplink of the package (i.i.d. Rayleigh channel, Gray QPSK, cubic power
amplifier, AWGN, one AGC gain per instance), drawn on the GPU from the seed alone.
"""
from __future__ import annotations

import math

import torch

from paper_2201_05024_gb300 import apsm

_SNR_DB = 15.0
_PAPER_SIGMA = math.sqrt(0.05)


# ---- the cases ---------------------------------------------------------------------------------

def listed():
    return [
        # the smallest frame: train on 200 pilots, detect 1000 vectors (launches and latency)
        dict(name="frame_4x2_p200_n1000", kind="frame", M=4, K=2, P=200, D=200, N=1000, W=8, sigma=0.5),
        # the paper's frame through the host-buffer call: 685 pilots, 3840 data vectors, window 20
        dict(name="host_frame_16x6_p685_n3840", kind="host_frame", M=16, K=6, P=685, D=685, N=3840, W=20,
             sigma=_PAPER_SIGMA),
        # training alone at the benchmark's block (retraining on a new channel)
        dict(name="train_16x6_p1024_w16", kind="train", M=16, K=6, P=1024, D=1024, W=16, sigma=0.5),
        # detection alone at the benchmark's block: a frozen filter over a long data block
        dict(name="detect_fp32_16x6_d1024_n65536", kind="detect", dtype="fp32", M=16, K=6, D=1024, N=65536, sigma=0.5),
        # train, then track through the data with decided targets; the dictionary slides (FIFO)
        dict(name="track_16x6_p685_n1920", kind="track", M=16, K=6, P=685, D=685, N=1920, W=20, sigma=0.5),
        # an odd user count and ragged entry and vector counts
        dict(name="detect_fp32_32x11_d1500_n10001", kind="detect", dtype="fp32", M=32, K=11, D=1500, N=10001, sigma=0.5),
        # a large array in full precision
        dict(name="detect_fp32_64x16_d4096_n100003", kind="detect", dtype="fp32", M=64, K=16, D=4096, N=100003,
             sigma=0.5),
        # the same array in the reduced-precision form, with its workspace kept
        dict(name="detect_bf16_64x16_d4096_n262144", kind="detect", dtype="bf16", M=64, K=16, D=4096, N=262144,
             sigma=0.5),
        # many uneven cells trained and detected by one graph launch
        dict(name="batch_32_uneven", kind="batch", n=32, W=16, sigma=0.5, d_lo=128, d_hi=2048, n_lo=1024, n_hi=16384),
        # adjoint of detection: fitting the coefficients over a fixed dictionary, ragged sizes
        dict(name="detect_backward_16x5_d1000_n16391", kind="detect_backward", M=16, K=5, D=1000, N=16391, sigma=0.5),
        # one differentiable train + detect with its backward, as a layer of a larger model
        dict(name="grad_step_16x6_p256_n4096", kind="grad_step", M=16, K=6, P=256, D=256, N=4096, W=8, sigma=0.5),
        # the same step for many instances that share their parameters, as one graph
        dict(name="grad_batch_64_16x6_p256_n4096", kind="grad_batch", n=64, M=16, K=6, P=256, D=256, N=4096, W=8,
             sigma=0.5),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed kinds: sizes over the logarithm of their range."""
    kind = rng.choice(["frame", "host_frame", "train", "detect", "detect", "detect", "track", "batch",
                       "detect_backward", "grad_step", "grad_batch"])
    if kind == "detect":
        dtype = rng.choice(["fp32", "fp32", "fp32", "bf16", "fp16"])
        # no more work than the largest listed case of full or of reduced precision
        limit = max(work(c)["flops"] for c in listed() if c["kind"] == kind and (c["dtype"] == "fp32") == (dtype == "fp32"))
        M = rng.choice([4, 8, 16, 32, 64] if dtype == "fp32" else [16, 32, 64])
        c = dict(kind=kind, dtype=dtype, M=M, K=rng.randint(2, min(M // 2 + 1, 16)), D=_log_int(rng, 128, 4096),
                 N=_log_int(rng, 1000, 262144), sigma=0.5)
        while work(c)["flops"] > limit:
            c["N"] = c["N"] // 2 + 1
        return c
    if kind == "batch":
        d_lo, n_lo = _log_int(rng, 64, 256), _log_int(rng, 300, 1500)
        return dict(kind=kind, n=_log_int(rng, 3, 32), W=rng.randint(4, 20), sigma=0.5, d_lo=d_lo,
                    d_hi=_log_int(rng, 512, 2048), n_lo=n_lo, n_hi=_log_int(rng, 3000, 16384))
    M = rng.choice([4, 8, 16, 32])
    K = rng.randint(2, min(M // 2 + 1, 12))
    if kind == "detect_backward":
        return dict(kind=kind, M=M, K=K, D=_log_int(rng, 100, 1024), N=_log_int(rng, 500, 20000), sigma=0.5)
    if kind in ("grad_step", "grad_batch"):
        M = rng.choice([4, 8, 16])
        K = rng.randint(2, min(M // 2 + 1, 6))
        P = _log_int(rng, 40, 256)
        c = dict(kind=kind, M=M, K=K, P=P, D=P, N=_log_int(rng, 300, 4096), W=rng.randint(4, 16), sigma=0.5)
        if kind == "grad_batch":
            c["n"] = _log_int(rng, 3, 64)
        return c
    P = _log_int(rng, 60, 1024)
    c = dict(kind=kind, M=M, K=K, P=P, D=P, W=rng.randint(4, 24), sigma=0.5)
    if kind != "train":
        c["N"] = _log_int(rng, 300, 16384) if kind != "track" else _log_int(rng, 100, 2000)
    return c


# ---- inputs --------------------------------------------------------------------------------------

def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _cn(g, *shape):
    """CN(0, 1) samples in 64 bits."""
    x = torch.randn(*shape, 2, generator=g, device=g.device, dtype=torch.float32).double()
    return torch.view_as_complex(x) * math.sqrt(0.5)


def _uplink(g, M, K, P, N):
    """(pilots [P][M], pilot symbols [P][K], data vectors [N][M], data symbols [N][K], channel
    scaled by the AGC gain [M][K], noise variance after the gain)."""
    h = _cn(g, M, K)

    def symbols(n):
        i = torch.randint(0, 2, (n, K, 2), generator=g, device=g.device)
        return torch.view_as_complex((1.0 - 2.0 * i.double()) * math.sqrt(0.5))

    sp, sd = symbols(P), symbols(N)
    n0 = 10.0 ** (-_SNR_DB / 10.0)

    def receive(s):
        return (s + 0.1 * s * s.abs().square()) @ h.T + math.sqrt(n0) * _cn(g, s.shape[0], M)

    rp, rd = receive(sp), receive(sd)
    gain = 1.0 / rp.abs().square().sum(1).mean().sqrt()
    c64 = torch.complex64
    return ((rp * gain).to(c64), sp.to(c64), (rd * gain).to(c64), sd.to(c64), 1.1 * gain * h, n0 * gain * gain)


def _filter(g, c):
    """A detector over given entries: the linear MMSE filter plus Gaussian coefficients of the size
    training leaves ([D][2][K], [M][K])."""
    rp, _, rd, sd, h, n0 = _uplink(g, c["M"], c["K"], c["D"], c["N"])
    eye = torch.eye(c["K"], dtype=h.dtype, device=h.device)
    clin = (torch.linalg.solve(h.mH @ h + n0 * eye, h.mH).mH / 0.5).to(torch.complex64).contiguous()
    gamma = 0.05 * torch.randn(c["D"], 2, c["K"], generator=g, device=g.device, dtype=torch.float32)
    return rp, gamma, clin, rd, sd


def _gen(seed):
    return torch.Generator(device=_dev()).manual_seed(int(seed))


def _params(c, **kw):
    return apsm.Params(M=c["M"], K=c["K"], window=c.get("W", 1), dict_cap=c["D"], sigma=c["sigma"], mu=0.5, eps=0.01,
                       w_L=0.5, dtype=c.get("dtype", "fp32"), **kw)


def _batch_shapes(c, seed):
    """Per-instance sizes of the uneven batch (fixed by the seed)."""
    g = torch.Generator().manual_seed(int(seed))

    def pick(lo, hi):
        return int(torch.randint(lo, hi + 1, (1,), generator=g))

    out = []
    for i in range(c["n"]):
        D = pick(c["d_lo"], c["d_hi"])
        out.append(dict(M=(8, 16, 32)[i % 3], K=2 + (5 * i) % 11 if i % 3 else 2 + i % 4, P=D, D=D,
                        N=pick(c["n_lo"], c["n_hi"]), W=c["W"], sigma=c["sigma"]))
    return out


def _shapes_seed(c):
    """The batch's sizes belong to the case, not to the seed of its inputs."""
    return 7 * c["n"] + 13 * c["d_hi"] + c["n_hi"]


# ---- one pass --------------------------------------------------------------------------------------

def prepare(case, seed):
    c, g, kind = case, _gen(seed), case["kind"]
    s = {"case": c}
    if kind == "batch":
        insts = []
        for sh in _batch_shapes(c, _shapes_seed(c)):
            rp, sp, rd, _, _, _ = _uplink(g, sh["M"], sh["K"], sh["P"], sh["N"])
            insts.append(apsm.BatchInstance(_params(sh), rp, sp, rd))
        s["batch"] = apsm.Batch(insts, lanes=16)
        return s
    p = s["p"] = _params(c)
    if kind in ("detect", "detect_backward"):
        entries, gamma, clin, rd, sd = _filter(g, c)
        s["state"] = apsm.state_set(p, apsm.State(p), entries, gamma, clin)
        s["rx"] = rd
        if kind == "detect":
            # the reduced-precision form packs its operands into a workspace that callers keep
            s["ws"] = apsm.detect_workspace(p, c["N"]) if c["dtype"] != "fp32" else None
        else:
            s["dsoft"] = (0.1 * _cn(g, c["N"], c["K"])).to(torch.complex64)
        return s
    if kind == "grad_batch":
        inst = [_uplink(g, c["M"], c["K"], c["P"], c["N"])[:4] for _ in range(c["n"])]
        clin0 = (0.05 * _cn(g, c["M"], c["K"])).to(torch.complex64)
        s["gb"] = apsm.GradBatch(p, inst, clin0, lanes=64 if c["n"] >= 64 else 16, graph=True)
        return s
    s["rp"], s["sp"], s["rd"], s["sd"], _, _ = _uplink(g, c["M"], c["K"], c["P"], c.get("N", 1))
    if kind == "grad_step":
        s["clin0"] = (0.05 * _cn(g, c["M"], c["K"])).to(torch.complex64).requires_grad_(True)
        s["theta"] = [torch.tensor(v, dtype=torch.float64, requires_grad=True) for v in (p.sigma, p.mu, p.eps, p.w_L)]
        return s
    s["state"] = apsm.State(p)
    if kind == "host_frame":
        for k in ("rp", "sp", "rd"):
            s[k] = s[k].cpu().pin_memory()
    return s


def _state_out(st):
    return {"gamma": st.gamma, "clin": st.clin, "dict": st.dict, "meta": st.meta}


def run(state):
    s = state
    c, kind = s["case"], s["case"]["kind"]
    if kind == "detect":
        soft, hard = apsm.detect(s["p"], s["state"], s["rx"], workspace=s["ws"])
        return {"soft": soft, "hard": hard}
    if kind == "train":
        return _state_out(apsm.train(s["p"], s["rp"], s["sp"], s["state"]))
    if kind == "frame":
        st = apsm.train(s["p"], s["rp"], s["sp"], s["state"])
        soft, hard = apsm.detect(s["p"], st, s["rd"])
        return {"soft": soft, "hard": hard, **_state_out(st)}
    if kind == "host_frame":
        soft, hard = apsm.train_detect_host(s["p"], s["rp"], s["sp"], s["rd"], state=s["state"])
        return {"soft": soft, "hard": hard}
    if kind == "track":
        st = apsm.train(s["p"], s["rp"], s["sp"], s["state"])
        soft, hard = apsm.train_continue(s["p"], s["rd"], st)
        return {"soft": soft, "hard": hard, **_state_out(st)}
    if kind == "batch":
        s["batch"].launch()
        return [{"soft": b.soft, "hard": b.hard} for b in s["batch"].instances]
    if kind == "detect_backward":
        dgamma, dclin, dscal = apsm.detect_backward(s["p"], s["state"], s["rx"], s["dsoft"])
        return {"dgamma": dgamma, "dclin": dclin, "dscalars": dscal}
    if kind == "grad_step":
        s["clin0"].grad = None
        for t in s["theta"]:
            t.grad = None
        soft = apsm.train_detect_autograd(s["p"], s["rp"], s["sp"], s["rd"], s["clin0"], *s["theta"])
        (soft - s["sd"]).abs().square().sum().backward()
        return {"soft": soft.detach(), "dclin0": s["clin0"].grad, "dtheta": [t.grad for t in s["theta"]]}
    gb = s["gb"]
    gb.run()
    loss, dtheta, dclin0 = gb.grads()
    return {"soft": gb.soft_all, "loss": gb.loss, "total": loss, "dtheta": dtheta, "dclin0": dclin0}


# ---- what a pass cannot do without --------------------------------------------------------------

def _detect_work(M, K, D, N):
    # per (vector, entry): the complex inner product, three exponentials, the coefficient sums
    return 8 * (N * M + N * K) + N * K + D * (8 * M + 4 + 8 * K), N * D * (8 * M + 8 * K + 9)


def _train_work(M, K, P, D, W):
    # each pilot against the entries held at its arrival, and per step the window's kernel values
    # applied to the window for every user
    pairs = sum(min(t, D) for t in range(P))
    by = P * (8 * M + 8 * K) + min(P, D) * (8 * M + 4 + 16 * K) + 8 * M * K
    return by, pairs * (8 * M + 8 * K + 9) + 2 * P * (W * (4 * M + 5) + 2 * W * W * K)


def work(case):
    c, kind = case, case["kind"]
    if kind == "batch":
        tot = [0, 0]
        for sh in _batch_shapes(c, _shapes_seed(c)):
            for b, f in (_train_work(sh["M"], sh["K"], sh["P"], sh["D"], sh["W"]),
                         _detect_work(sh["M"], sh["K"], sh["D"], sh["N"])):
                tot = [tot[0] + b, tot[1] + f]
        return {"bytes": tot[0], "flops": tot[1]}
    M, K, D = c["M"], c["K"], c["D"]
    by = fl = 0
    if kind in ("frame", "host_frame", "train", "track", "grad_step", "grad_batch"):
        by, fl = _train_work(M, K, c["P"], D, c["W"])
    if kind in ("frame", "host_frame", "detect", "grad_step", "grad_batch"):
        b, f = _detect_work(M, K, D, c["N"])
        by, fl = by + b, fl + f
    if kind == "track":
        b, f = _train_work(M, K, c["P"] + c["N"], D, c["W"])
        by, fl = b + 9 * c["N"] * K, f
    if kind in ("detect_backward", "grad_step", "grad_batch"):
        N = c["N"]
        by += 8 * (N * M + N * K) + D * (8 * M + 4 + 16 * K) + 16 * M * K
        fl += N * D * (8 * M + 16 * K + 12) + 8 * N * M * K
    if kind in ("grad_step", "grad_batch"):  # the adjoint of the recurrence: about twice the recurrence
        fl += 2 * _train_work(M, K, c["P"], D, c["W"])[1]
        by += _train_work(M, K, c["P"], D, c["W"])[0]
        by, fl = by * c.get("n", 1), fl * c.get("n", 1)
    return {"bytes": by, "flops": fl}


# ---- the same values in 64 bits -----------------------------------------------------------------

def _split(r):
    """Real-split samples of received vectors [..][P][M] -> [..][2P][2M] float64."""
    r = r.to(torch.complex128)
    x = torch.stack([torch.cat([r.real, r.imag], -1), torch.cat([r.imag, -r.real], -1)], -2)
    return x.flatten(-3, -2)


def _targets(s):
    s = s.to(torch.complex128)
    return torch.stack([s.real, s.imag], -2).flatten(-3, -2)


def _sqdist(x, y):
    return ((x * x).sum(-1)[..., :, None] + (y * y).sum(-1)[..., None, :] - 2.0 * x @ y.mT).clamp_min(0.0)


def _recurrence(x, b, W, D, sigma, w0, n_samples=None, decide_from=None, mu=0.5, eps=0.01, wl=0.5):
    """APSM over real-split samples x [B][S][2M] with targets b [B][S][K] from linear filters w0
    [B][2M][K]: (gamma [B][S][K], w [B][2M][K], outputs at arrival [B][S][K])."""
    B, S, _ = x.shape
    K = b.shape[-1]
    b = b.clone()
    gauss = torch.exp(-_sqdist(x, x) / (2.0 * sigma * sigma))
    kern = wl * (x @ x.mT) + (1.0 - wl) * gauss
    evict = S // 2 > D
    if not evict:
        gauss = None
    diag = torch.diagonal(kern, dim1=1, dim2=2)[..., None]
    p = wl * (x @ w0)
    gamma = torch.zeros(B, S, K, dtype=x.dtype, device=x.device)
    dropped = torch.zeros(S, dtype=torch.bool, device=x.device)
    arrival = torch.zeros_like(gamma)
    ends = None if n_samples is None else torch.tensor(n_samples, device=x.device)[:, None, None]
    for n in range(S):
        if evict and n % 2 == 0 and n // 2 >= D:
            o = n - 2 * D
            p = p - (1.0 - wl) * (gauss[:, :, o:o + 2] @ gamma[:, o:o + 2])
            dropped[o:o + 2] = True
        arrival[:, n] = p[:, n]
        if decide_from is not None and n >= decide_from:
            b[:, n] = torch.where(p[:, n] >= 0, 1.0, -1.0).to(x.dtype) * math.sqrt(0.5)
        lo = max(0, n - W + 1)
        pw, bw = p[:, lo:n + 1], b[:, lo:n + 1]
        step = (mu / (n + 1 - lo)) * (torch.minimum(torch.maximum(pw, bw - eps), bw + eps) - pw) / diag[:, lo:n + 1]
        if ends is not None:
            step = torch.where(n < ends, step, torch.zeros_like(step))
        gamma[:, lo:n + 1] += step
        p = p + kern[:, :, lo:n + 1] @ step
    w = w0 + x.mT @ gamma
    gamma = torch.where(dropped[None, :, None], torch.zeros_like(gamma), gamma)
    return gamma, w, arrival


def _evaluate(x, entries, gamma, w, sigma, wl=0.5):
    """f(x) for real-split samples x [S][2M]: entries' samples [E][2M], gamma [E][K], w [2M][K]."""
    return wl * (x @ w) + (1.0 - wl) * (torch.exp(-_sqdist(x, entries) / (2.0 * sigma * sigma)) @ gamma)


def _soft(rx, entries, gamma, w, sigma, rows=8192):
    out = []
    for i in range(0, rx.shape[0], rows):
        y = _evaluate(_split(rx[i:i + rows]), entries, gamma, w, sigma)
        out.append(torch.complex(y[0::2], y[1::2]))
    return torch.cat(out)


def _as_clin(w):
    M = w.shape[-2] // 2
    return torch.complex(w[..., :M, :].contiguous(), w[..., M:, :].contiguous())


def _as_w(clin):
    c = clin.to(torch.complex128)
    return torch.cat([c.real, c.imag], -2)


def _ring_gamma(gamma, n_vec, c):
    """Coefficients [2 n_vec][K] in the slots of the ring ([A][2][K], A = D rounded up to 32)."""
    A = -(-c["D"] // 32) * 32
    out = torch.zeros(A, 2, c["K"], dtype=gamma.dtype, device=gamma.device)
    t = torch.arange(max(0, n_vec - c["D"]), n_vec, device=gamma.device)
    out[t % c["D"]] = gamma.reshape(n_vec, 2, -1)[t]
    return out


def _grad_soft(x, b, rd, c, clin0, theta):
    """Differentiable train + detect of instances [B] in 64 bits: soft [B][N][K]."""
    sigma, mu, eps, wl = theta
    B, S, _ = x.shape
    K, W = c["K"], c["W"]
    d2, lin = _sqdist(x, x), x @ x.mT
    diag = wl * torch.diagonal(lin, dim1=1, dim2=2)[..., None] + (1.0 - wl)
    w0 = torch.cat([clin0.real, clin0.imag], -2)
    p = wl * (x @ w0)
    steps = []
    for n in range(S):
        lo = max(0, n - W + 1)
        pw, bw = p[:, lo:n + 1], b[:, lo:n + 1]
        beta = (torch.relu(bw - eps - pw) - torch.relu(pw - bw - eps)) / diag[:, lo:n + 1]
        step = (mu / (n + 1 - lo)) * beta
        steps.append(torch.nn.functional.pad(step, (0, 0, lo, S - 1 - n)))
        kern = wl * lin[:, :, lo:n + 1] + (1.0 - wl) * torch.exp(-d2[:, :, lo:n + 1] / (2.0 * sigma * sigma))
        p = p + kern @ step
    gamma = torch.stack(steps).sum(0)
    w = w0 + x.mT @ gamma
    xd = _split(rd)
    y = wl * (xd @ w) + (1.0 - wl) * (torch.exp(-_sqdist(xd, x) / (2.0 * sigma * sigma)) @ gamma)
    return torch.complex(y[:, 0::2].contiguous(), y[:, 1::2].contiguous())


def exact(case, seed):
    c, g, kind = case, _gen(seed), case["kind"]
    if kind == "batch":
        shapes = _batch_shapes(c, _shapes_seed(c))
        ups = [_uplink(g, sh["M"], sh["K"], sh["P"], sh["N"])[:3] for sh in shapes]
        S = max(2 * sh["P"] for sh in shapes)
        x = torch.zeros(c["n"], S, 2 * 32, dtype=torch.float64, device=g.device)
        b = torch.zeros(c["n"], S, 12, dtype=torch.float64, device=g.device)
        for i, (sh, (rp, sp, _)) in enumerate(zip(shapes, ups)):
            x[i, :2 * sh["P"], :2 * sh["M"]] = _split(rp)
            b[i, :2 * sh["P"], :sh["K"]] = _targets(sp)
        w0 = torch.zeros(c["n"], 64, 12, dtype=torch.float64, device=g.device)
        gamma, w, _ = _recurrence(x, b, c["W"], S, c["sigma"], w0, n_samples=[2 * sh["P"] for sh in shapes])
        out = []
        for i, (sh, (rp, _, rd)) in enumerate(zip(shapes, ups)):
            gi, wi = gamma[i, :2 * sh["P"], :sh["K"]], w[i, :2 * sh["M"], :sh["K"]]
            out.append({"soft": _soft(rd, _split(rp), gi, wi, c["sigma"]), "hard": None})
        return out
    if kind in ("detect", "detect_backward"):
        entries, gamma, clin, rd, sd = _filter(g, c)
        ge, we, xe = gamma.double().reshape(2 * c["D"], c["K"]), _as_w(clin), _split(entries)
        if kind == "detect":
            return {"soft": _soft(rd, xe, ge, we, c["sigma"]), "hard": None}
        dsoft = (0.1 * _cn(g, c["N"], c["K"])).to(torch.complex64)
        sigma = torch.tensor(_params(c).sigma, dtype=torch.float64, device=g.device)
        var = [ge.requires_grad_(True), we.requires_grad_(True), sigma.requires_grad_(True),
               torch.tensor(0.5, dtype=torch.float64, device=g.device, requires_grad=True)]
        tot = [torch.zeros_like(v) for v in var]
        for i in range(0, c["N"], 4096):
            y = _evaluate(_split(rd[i:i + 4096]), xe, ge, we, var[2], var[3])
            d = _targets(dsoft[i:i + 4096])
            for t, v in zip(tot, torch.autograd.grad((y * d).sum(), var)):
                t += v
        return {"dgamma": _ring_gamma(tot[0], c["D"], c), "dclin": _as_clin(tot[1]),
                "dscalars": torch.stack(tot[2:])}
    if kind in ("grad_step", "grad_batch"):
        inst = [_uplink(g, c["M"], c["K"], c["P"], c["N"])[:4] for _ in range(c.get("n", 1))]
        clin0 = (0.05 * _cn(g, c["M"], c["K"])).to(torch.complex64).to(torch.complex128).requires_grad_(True)
        theta = [torch.tensor(v, dtype=torch.float64, device=g.device, requires_grad=True)
                 for v in (c["sigma"], 0.5, 0.01, 0.5)]
        loss, soft = [], []
        tot = [torch.zeros_like(v) for v in [clin0] + theta]
        for i in range(0, len(inst), 16):  # sixteen instances at a time keep the graph small
            part = inst[i:i + 16]
            y = _grad_soft(torch.stack([_split(u[0]) for u in part]), torch.stack([_targets(u[1]) for u in part]),
                           torch.stack([u[2] for u in part]), c, clin0, theta)
            per = (y - torch.stack([u[3] for u in part]).to(torch.complex128)).abs().square().sum((1, 2))
            for t, v in zip(tot, torch.autograd.grad(per.sum(), [clin0] + theta)):
                t += v
            soft.append(y.detach())
            loss.append(per.detach())
        soft, loss = torch.cat(soft), torch.cat(loss)
        if kind == "grad_step":
            return {"soft": soft[0], "dclin0": tot[0], "dtheta": tot[1:]}
        return {"soft": soft, "loss": loss, "total": loss.sum(), "dtheta": torch.stack(tot[1:]), "dclin0": tot[0]}
    rp, sp, rd, _, _, _ = _uplink(g, c["M"], c["K"], c["P"], c.get("N", 1))
    seq, b, n_vec = rp, _targets(sp), c["P"]
    if kind == "track":
        seq, n_vec = torch.cat([rp, rd]), c["P"] + c["N"]
        b = torch.cat([b, torch.zeros(2 * c["N"], c["K"], dtype=b.dtype, device=b.device)])
    x = _split(seq)
    w0 = torch.zeros(1, 2 * c["M"], c["K"], dtype=torch.float64, device=g.device)
    gamma, w, arrival = _recurrence(x[None], b[None], c["W"], c["D"], c["sigma"], w0,
                                    decide_from=2 * c["P"] if kind == "track" else None)
    A = -(-c["D"] // 32) * 32
    held = torch.zeros(A, c["M"], dtype=torch.complex128, device=g.device)
    t = torch.arange(max(0, n_vec - c["D"]), n_vec, device=g.device)
    held[t % c["D"]] = seq[t].to(torch.complex128)
    st = {"gamma": _ring_gamma(gamma[0], n_vec, c), "clin": _as_clin(w[0]), "dict": held, "meta": None}
    if kind == "train":
        return st
    if kind == "track":
        y = arrival[0, 2 * c["P"]:]
        return {"soft": torch.complex(y[0::2].contiguous(), y[1::2].contiguous()), "hard": None, **st}
    soft = _soft(rd, x, gamma[0], w[0], c["sigma"])
    return {"soft": soft, "hard": None, **(st if kind == "frame" else {})}

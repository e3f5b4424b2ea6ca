"""Timing cases: the work that programs have this filter do, through the public
Python API (paper_1310_4624_gb300.filter).

A pass of a filter case is one whole sequence: `reset`, T frames, and the
read-back of the results.  Sizes come from the package's workloads
(paper_1310_4624_gb300/synth.py), its benchmark and its tests; `draw` spreads
over the same ranges.  Every input is made from the seed alone: frames are
Poisson images of spots at seeded positions, and the filter's own random
streams are keyed by the seed.
"""
import math

import numpy as np
import torch

from paper_1310_4624_gb300 import synth
from paper_1310_4624_gb300.filter import LogLikelihood, ParticleFilter, config_from_workload, resample

DEV = "cuda:0"


def _filter_case(name, api, **kw):
    """A filter case: one track of G groups of Np particles unless `tracks` says otherwise."""
    c = dict(name=name, kind="filter", api=api, tracks=1, G=4, Np=1024, H=64, W=64, T=20, arna=True, ex_ratio=0.1,
             radius=5, sharing=False, frame_ratio=False, ess=False, keyed=False, topology=0, size_seed=0)
    c.update(kw)
    return c


def listed():
    return [
        # A short sequence of one spot, the package's smallest workload: launches and latency count.
        _filter_case("small_rna", "step", arna=False, T=20),
        # A track started at a detection and followed into the next frame: the shortest use of a filter.
        _filter_case("new_track_pair", "step", T=2),
        # The headline workload: a million particles tracking one spot, frames already on the device.
        _filter_case("tracking_arna", "step", G=64, Np=16384, H=512, W=512, T=20),
        # The same population fed from host memory, an estimate read back every frame (online tracking).
        _filter_case("tracking_stream_host", "host", G=64, Np=16384, H=512, W=512, T=20, arna=False),
        # Information sharing: all groups but one start spread over the image and search for the spot.
        _filter_case("sharing_frame_ratio", "step", G=256, Np=4096, H=512, W=512, T=20, sharing=True,
                     frame_ratio=True),
        # Gradient of log Z, forward and backward, at the package's differentiable workload (fewer frames).
        _filter_case("gradient", "grad", G=16, Np=65536, H=512, W=512, T=20),
        # The shortest gradient: two frames of a small track, as a parameter fit on many short tracks runs it.
        _filter_case("gradient_pair", "grad", G=4, Np=4096, H=64, W=64, T=2),
        # Many independent tracks of mixed sizes in one handle, one graph launch per frame (batch serving).
        _filter_case("batched_graph", "graph", tracks=512, H=256, W=256, T=4),
        # Several objects in one sequence, one filter per object, all given the same frames.
        _filter_case("multi_object", "step", tracks=64, G=16, Np=1024, H=512, W=512, T=20),
        # Method variants on ragged sizes: threshold resampling, keyed send sets, node-aware ring.
        _filter_case("variants_ragged", "step", G=95, Np=1269, H=200, W=181, T=20, ess=True, keyed=True, topology=1),
        # A wide spot and an odd frame: the largest patch radius, ragged groups, rows off the 16-byte grid.
        _filter_case("wide_patch_odd_frame", "step", G=33, Np=3001, H=277, W=301, T=20, radius=7, arna=False,
                     ex_ratio=0.25),
        # The resampler alone on a caller's log-weights (a program with its own propagation and likelihood).
        dict(name="resample_ragged", kind="resample", G=37, Np=20011, codes=False),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "host", "grad", "graph", "multi", "resample"])
    if kind == "resample":
        g = _log_int(rng, 1, 256)
        return dict(kind="resample", G=g, Np=_log_int(rng, 64, min(1 << 20, (1 << 21) // g)), codes=rng.random() < 0.4)
    if kind == "graph":
        c = _filter_case("", "graph", tracks=_log_int(rng, 2, 384), H=rng.randint(48, 256), W=rng.randint(48, 256), T=4,
                         size_seed=rng.randint(1, 1000))
    elif kind == "multi":
        c = _filter_case("", "step", tracks=rng.randint(2, 64), G=rng.randint(4, 24), Np=_log_int(rng, 256, 2048), H=512,
                         W=512, T=rng.randint(4, 16))
    else:
        g = _log_int(rng, 2, 256)
        n = _log_int(rng, 4096, 1 << 20)
        c = _filter_case("", kind, G=g, Np=max(16, n // g), H=rng.randint(64, 512), W=rng.randint(64, 512),
                         T=rng.choice([2, rng.randint(3, 20)]), arna=rng.random() < 0.6,
                         ex_ratio=rng.choice([0.0, 0.1, 0.25, 0.5]), radius=rng.choice([3, 5, 5, 5, 7]))
        if kind == "step":
            c["sharing"] = rng.random() < 0.3
            c["frame_ratio"] = c["sharing"] or rng.random() < 0.2
            c["ess"] = rng.random() < 0.2
            c["keyed"] = rng.random() < 0.2
            c["topology"] = rng.choice([0, 0, 0, 1, 2])
    del c["name"]
    return c


def _psf(radius):
    return {3: 1.0, 5: 1.5, 7: 2.1}[radius]


def _workloads(case, seed):
    """The synthetic workloads of a filter case, one per track."""
    H, W, T = case["H"], case["W"], case["T"]
    mode = synth.ARNA if case["arna"] else synth.RNA
    if case["api"] == "graph":  # track sizes belong to the case, frames and random streams to the seed
        wls = synth.batched_tracks(case["tracks"], seed=case["size_seed"], H=H, W=W, T=T)
        return [wl.replace(seed=seed, data_seed=seed * 4096 + t) for t, wl in enumerate(wls)]
    if case["tracks"] > 1:
        return synth.multi_object(n_obj=case["tracks"], G=case["G"], Np=case["Np"], H=H, W=W, T=T, mode=mode, seed=seed,
                                  data_seed=seed)
    return [synth.Workload(name="one", G=case["G"], Np=case["Np"], H=H, W=W, T=T, mode=mode, seed=seed, data_seed=seed,
                           ex_ratio=case["ex_ratio"], patch_radius=case["radius"], sigma_psf=_psf(case["radius"]),
                           margin=min(6.0, H / 8, W / 8),
                           init=synth.INIT_SHARING if case["sharing"] else synth.INIT_POINT,
                           obs_model=1 if case["frame_ratio"] else 0, resample_rule=1 if case["ess"] else 0,
                           send_rule=1 if case["keyed"] else 0, topology=case["topology"],
                           node_groups=16 if case["topology"] == 1 else 1, truth_noise=case["api"] == "grad")]


def _sequences(case, wls, seed):
    """(frames per track, each (T, H, W) float32 on the host or the device; start state per track)."""
    if case["api"] == "graph":
        frames, truths = synth.render_batched_torch(wls, DEV, seed=seed)
        return [frames[t] for t in range(len(wls))], truths[:, 0]
    if case["tracks"] > 1:
        frames, truths = synth.make_multi_sequence(wls)
        return [frames] * len(wls), truths[:, 0]
    frames, truth = synth.make_sequence(wls[0])
    return [frames], truth[None, 0]


def _logits(case, seed):
    """Log-weights as an image likelihood leaves them (half the squared distance
    to the spot over the noise, plus pixel noise), and the groups' uniform words."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    n = case["G"] * case["Np"]
    d = torch.randn((2, n), generator=gen, device=DEV)
    lw = -2.0 * d.square().sum(0) + 0.5 * torch.randn(n, generator=gen, device=DEV) - 60.0
    u = torch.randint(-(1 << 31), (1 << 31) - 1, (case["G"],), generator=gen, device=DEV, dtype=torch.int64)
    return lw, u.to(torch.int32)


def prepare(case, seed):
    if case["kind"] == "resample":
        lw, u = _logits(case, seed)
        return dict(case=case, lw=lw, u=u)
    wls = _workloads(case, seed)
    frames, starts = _sequences(case, wls, seed)
    api = case["api"]
    cfgs = [config_from_workload(wl, starts[t], track_id=t, record_ancestors=api == "grad") for t, wl in enumerate(wls)]
    st = dict(case=case, pf=ParticleFilter(cfgs, history=max(2, case["T"]), device=DEV))
    if api == "graph":
        st["frames"] = frames
        st["table"] = st["pf"].frame_table(frames)
    elif api == "host":
        st["frames"] = torch.from_numpy(frames[0]).pin_memory()
        st["xhat"] = torch.zeros((case["T"], 1, 5)).pin_memory()
        st["log_Z"] = torch.zeros((case["T"], 1), dtype=torch.float64).pin_memory()
        st["done"] = [torch.cuda.Event() for _ in range(2)]
    else:
        st["frames"] = torch.from_numpy(frames[0]).to(DEV)
    if api == "grad":
        wl = wls[0]
        st["theta"] = torch.tensor([wl.sigma_psf, wl.amplitude, wl.background, wl.sigma_pos, wl.sigma_v],
                                   dtype=torch.float32, device=DEV, requires_grad=True)
    return st


def run(state):
    case = state["case"]
    if case["kind"] == "resample":
        out = resample(state["lw"], state["u"], case["G"], case["Np"], want_q=case["codes"])
        return dict(anc=out[0], q=out[1]) if case["codes"] else dict(anc=out)
    pf, api, T = state["pf"], case["api"], case["T"]
    if api == "grad":
        theta = state["theta"]
        theta.grad = None
        log_z = LogLikelihood.apply(theta, pf, state["frames"])
        log_z.backward()
        return dict(log_Z=log_z.detach(), grad=theta.grad)
    pf.reset()
    if api == "host":
        # the estimate of frame k - 1 is awaited while frame k runs
        frames, xhat, log_z, done = state["frames"], state["xhat"], state["log_Z"], state["done"]
        for k in range(T):
            pf.step_host(frames[k])
            pf.estimate_async(xhat[k], log_z[k])
            done[k & 1].record(pf.stream)
            if k > 0:
                done[(k - 1) & 1].synchronize()
        done[(T - 1) & 1].synchronize()
        return dict(xhat=xhat, log_Z=log_z)
    if api == "graph":
        for _ in range(T):
            pf.step_table(state["table"], graph=True)
        x, z, _ = pf.estimate()
        return dict(xhat=x, log_Z=z)
    frames, n = state["frames"], case["tracks"]
    for k in range(T):
        pf.step(frames[k] if n == 1 else [frames[k]] * n)
    x, z, _ = pf.estimate()
    out = dict(xhat=x, log_Z=z)
    if n == 1:
        p = pf.particles()
        out.update(states=p["states"], logw=p["logw"], anc=p["anc"])
    return out


def _particles(case):
    if case["api"] == "graph":
        return sum(wl.N for wl in _workloads(case, 0))
    return case["tracks"] * case["G"] * case["Np"]


def work(case):
    """Bytes and lane operations of one pass: per particle and step the parent
    state and ancestor read and the new state and ancestor written (48 B), the
    frames read once, and the method's arithmetic (a (2R+1)^2 patch at three
    operations a pixel, its Gaussians, the dynamics and their random numbers:
    610 at R = 5).  The gradient adds the recorded parent and the reverse
    sweep: state, parent and state adjoint once more, and twice the arithmetic."""
    if case["kind"] == "resample":
        n = case["G"] * case["Np"]
        return dict(bytes=n * (16 if case["codes"] else 8) + 4 * case["G"], flops=20 * n)
    D = 2 * case["radius"] + 1
    n, T = _particles(case), case["T"]
    ops = 3 * D * D + 5 * D + 192
    frames = T * case["H"] * case["W"] * 4 * (case["tracks"] if case["api"] == "graph" else 1)
    if case["api"] == "grad":
        return dict(bytes=n * T * (52 + 64) + 2 * frames, flops=3 * n * T * ops)
    return dict(bytes=n * T * 48 + frames, flops=n * T * ops)


# ---------------------------------------------------------------- 64-bit values
def _philox(key, c):
    """Philox4x32-10 of counters c (four uint64 arrays holding 32-bit words)."""
    m32 = np.uint64(0xFFFFFFFF)
    k0, k1 = key & 0xFFFFFFFF, key >> 32
    c = [x.astype(np.uint64) for x in c]
    for r in range(10):
        p0, p1 = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        a, b = np.uint64((k0 + r * 0x9E3779B9) & 0xFFFFFFFF), np.uint64((k1 + r * 0xBB67AE85) & 0xFFFFFFFF)
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ a, p1 & m32, (p0 >> np.uint64(32)) ^ c[3] ^ b, p0 & m32]
    return c


def _normals(seed, G, Np, k):
    """The five process-noise normals (5, G Np) of track 0 at step k."""
    g, j = np.divmod(np.arange(G * Np, dtype=np.uint64), np.uint64(Np))
    kk = np.full(G * Np, k, np.uint64)
    w = [x for call in (0, 1) for x in _philox(seed, [j, g, kk, np.full(G * Np, (1 << 4) | call, np.uint64)])]
    u = [((x >> np.uint64(9)).astype(np.float64) + 0.5) * 2.0 ** -23 for x in w]
    e = []
    for a in range(0, 6, 2):
        rho = np.sqrt(-2.0 * np.log(u[a]))
        e += [rho * np.cos(2 * math.pi * u[a + 1]), rho * np.sin(2 * math.pi * u[a + 1])]
    return torch.from_numpy(np.stack(e[:5])).to(DEV)


def _loglik(case, z, s, theta):
    """Patch log-likelihoods (sigma_obs = 1) of states s (5, n) under frame z (H, W), float64."""
    R, (H, W) = case["radius"], z.shape
    psf, bg = theta[0], theta[2]
    x, y, amp = s[0], s[1], s[4]
    cx, cy = torch.floor(x + 0.5).detach(), torch.floor(y + 0.5).detach()
    out = 0.0
    for b in range(-R, R + 1):
        gy = torch.exp(-(cy + b - y) ** 2 / (2 * psf ** 2))
        for a in range(-R, R + 1):
            u, v = (cx + a).long(), (cy + b).long()
            inside = (u >= 0) & (u < W) & (v >= 0) & (v < H)
            pix = torch.where(inside, z[v.clamp(0, H - 1), u.clamp(0, W - 1)] - bg, torch.zeros_like(x))
            m = amp * torch.exp(-(cx + a - x) ** 2 / (2 * psf ** 2)) * gy
            out = out - 0.5 * ((pix - m) ** 2 - (pix ** 2 if case["frame_ratio"] else 0.0))
    return out


def exact(case, seed):
    """The first two frames of one track started at a point have a closed
    form: every particle scores the first frame alike, so resampling keeps all
    of them in place, and the second step is one draw of the dynamics.  Longer
    runs follow their own resampling, whose choices a different rounding
    changes: no value is given for them, nor for whole-number outputs."""
    if case["kind"] == "resample" or case["T"] != 2 or case["tracks"] != 1 or case["sharing"]:
        return None
    wl = _workloads(case, seed)[0]
    frames, starts = _sequences(case, [wl], seed)
    f = torch.from_numpy(frames[0]).to(DEV).double()
    n = case["G"] * case["Np"]
    start = torch.from_numpy(np.float32(starts[0])).to(DEV).double()
    f32 = [float(np.float32(v)) for v in (wl.sigma_psf, wl.amplitude, wl.background, wl.sigma_pos, wl.sigma_v)]
    e = _normals(seed, case["G"], case["Np"], 1)
    grad = case["api"] == "grad"

    def states(theta, lo, hi):
        s0 = torch.cat([start[:4], theta[1:2]]) if grad else start
        x = e[:, lo:hi]
        return torch.stack([s0[0] + s0[2] + theta[3] * x[0], s0[1] + s0[3] + theta[3] * x[1], s0[2] + theta[4] * x[2],
                            s0[3] + theta[4] * x[3], s0[4] + wl.sigma_I * x[4]])

    def first(theta):
        s0 = torch.cat([start[:4], theta[1:2]]) if grad else start
        return _loglik(case, f[0], s0[:, None], theta)[0]

    spans = [(lo, min(n, lo + (1 << 16))) for lo in range(0, n, 1 << 16)]
    theta = torch.tensor(f32, dtype=torch.float64, device=DEV)
    with torch.no_grad():
        s = torch.cat([states(theta, *p) for p in spans], 1)
        lik = torch.cat([_loglik(case, f[1], s[:, lo:hi], theta) for lo, hi in spans])
        l0 = float(first(theta))
        log_c = float(torch.logsumexp(lik, 0)) - math.log(n)
    if not grad:
        w = torch.softmax(lik, 0)
        x0, x1 = start.float().cpu().numpy().astype(np.float64), (s @ w).cpu().numpy()
        if case["api"] == "host":
            return dict(xhat=np.stack([x0, x1])[:, None, :], log_Z=np.array([[l0], [l0 + log_c]]))
        return dict(xhat=x1[None], log_Z=np.array([l0 + log_c]), states=s, logw=lik - math.log(n), anc=None)
    total = torch.zeros(5, dtype=torch.float64, device=DEV)
    w = torch.softmax(lik, 0)
    for part in [None] + spans:  # d log Z = d l_0 + sum_i w_i d l_1(i)
        th = theta.clone().requires_grad_(True)
        v = first(th) if part is None else (w[part[0]:part[1]] * _loglik(case, f[1], states(th, *part), th)).sum()
        v.backward()
        total += th.grad
    return dict(log_Z=l0 + log_c, grad=total)

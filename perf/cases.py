"""Performance cases of the power Doppler hot path.

Each case is one call (or the short run of calls that a program makes
together) through the package's public entry points: the five stages of the
path in the forms that the 2D and 3D workloads use, the learned clutter
filter, and two whole calls (one ensemble, a batch of uneven ensembles).

  listed()             the cases
  draw(rng)            one more case of the same ranges
  prepare(case, seed)  inputs on the GPU, made from the seed, and the plans,
                       weights and output buffers that a program keeps
  run(state)           one pass; returns its outputs
  work(case)           bytes and operations that a pass cannot do without
  exact(case, seed)    the outputs in 64 bits by plain torch, or None
"""
import math

import numpy as np
import torch

from paper_2509_05464_gb300 import fq
from paper_2509_05464_gb300 import learned
from paper_2509_05464_gb300 import workload as W
from paper_2509_05464_gb300.pipeline import Pipeline

DEV = "cuda"
DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
GRAM = {"f32": fq.FQ_GRAM_F32, "tf32": fq.FQ_GRAM_TF32, "bf16": fq.FQ_GRAM_BF16}
FILTER_CH = (2, 32, 32, 32, 2)


def listed():
    return [
        # Smallest call: the blood echo of the 64-element single-angle
        # workload added to the static tissue RF (what a program with still
        # tissue calls for each ensemble): launch and latency bound.
        {"name": "rf_blood_small", "kind": "rf", "probe": "linear64", "scatterers": 200, "frames": 10,
         "base": True, "rf": "f32"},
        # RF synthesis of the 2D compounded workload's medium in FP32: the
        # linear probe, 5 angles, float-float delays.
        {"name": "rf_2d", "kind": "rf", "probe": "linear128", "scatterers": 100_000, "frames": 16,
         "base": False, "rf": "f32"},
        # RF synthesis of the 3D volumetric workload's medium, BF16 records:
        # the matrix probe, 9 tilts.  The largest part of a 3D ensemble.
        {"name": "rf_3d", "kind": "rf", "probe": "matrix32", "scatterers": 500_000, "frames": 12,
         "base": False, "rf": "bf16"},
        # Beamforming of the whole 2D compounded ensemble, FP32.
        {"name": "beamform_2d", "kind": "beamform", "probe": "linear128", "frames": 200, "nx": 256, "ny": 1,
         "nz": 256, "rf": "f32", "ch": "f32"},
        # Beamforming of the 3D volumetric ensemble, BF16 RF and channel IQ.
        {"name": "beamform_3d", "kind": "beamform", "probe": "matrix32", "frames": 100, "nx": 128, "ny": 128,
         "nz": 128, "rf": "bf16", "ch": "bf16"},
        # SVD clutter filter and power Doppler of the 2D ensemble: two
        # components removed, the filtered IQ kept.
        {"name": "clutter_2d", "kind": "clutter", "pixels": 256 * 256, "frames": 200, "k": 2, "iq": "f32",
         "gram": "f32", "want_iq": True},
        # The same of the 3D ensemble with the energy cutoff, power Doppler
        # alone.
        {"name": "clutter_3d", "kind": "clutter", "pixels": 128 ** 3, "frames": 100, "k": -1, "iq": "f32",
         "gram": "f32", "want_iq": False},
        # Vessel membership and the trajectories of the 3D medium: 500k
        # scatterers, a tree of 63 vessels, 100 frames.
        {"name": "motion_3d", "kind": "motion", "medium": "tree", "scatterers": 500_000, "frames": 100},
        # One training step of the learned filter on four patches of 64
        # frames x 32 x 32 pixels (the size the trainer uses): forward, loss,
        # gradients.
        {"name": "filter_train", "kind": "train", "volumes": 4, "frames": 64, "nz": 32, "nx": 32},
        # The learned filter applied to the whole 2D ensemble.
        {"name": "filter_apply", "kind": "filter", "frames": 200, "nz": 256, "nx": 256},
        # One whole ensemble of the smallest workload (still tissue, 2000
        # scatterers), scatterers to power Doppler: many short launches.
        {"name": "ensemble_small", "kind": "ensemble", "medium": "still", "scatterers": 2000, "frames": 48,
         "nx": 64, "nz": 128},
        # A batch of uneven ensembles through the persistent kernels and the
        # CUDA graph.
        {"name": "batch_uneven", "kind": "batch", "members": 8, "s_lo": 10_000, "s_hi": 60_000, "f_lo": 50,
         "f_hi": 120},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["rf", "rf", "beamform", "beamform", "clutter", "clutter", "motion", "train", "filter",
                       "ensemble", "batch"])
    if kind == "rf":
        probe = rng.choice(["linear64", "linear128", "matrix32"])
        s = _log_int(rng, 150, 500_000)
        lines = len(_tilts(probe)[0]) * _probe(probe).n_elements
        # at most the pairs of the 3D listed case, at most 100 frames
        f = max(1, min(100, int(5.5e10 / (lines * s)), _log_int(rng, 2, 128)))
        if probe == "matrix32":
            f = min(f, 12)
        return {"kind": "rf", "probe": probe, "scatterers": s, "frames": f,
                "base": rng.random() < 0.25, "rf": rng.choice(["f32", "f32", "bf16", "f16"])}
    if kind == "beamform":
        probe = rng.choice(["linear64", "linear128", "linear128", "matrix32"])
        dt = rng.choice(["f32", "bf16", "f16"])
        f = _log_int(rng, 12, 200 if probe != "matrix32" else 100)
        if probe == "matrix32":
            n = [_log_int(rng, 24, 96) for _ in range(3)]
        else:
            n = [_log_int(rng, 48, 256), 1, _log_int(rng, 64, 320)]
        return {"kind": "beamform", "probe": probe, "frames": f, "nx": n[0], "ny": n[1], "nz": n[2], "rf": dt,
                "ch": dt}
    if kind == "clutter":
        return {"kind": "clutter", "pixels": _log_int(rng, 8192, 1_500_000), "frames": _log_int(rng, 40, 200),
                "k": rng.choice([2, 3, -1]), "iq": rng.choice(["f32", "f32", "bf16"]), "gram": "f32",
                "want_iq": rng.random() < 0.5}
    if kind == "motion":
        return {"kind": "motion", "medium": rng.choice(["tree", "arcs", "arcs"]),
                "scatterers": _log_int(rng, 2000, 500_000), "frames": _log_int(rng, 8, 100)}
    if kind == "train":
        return {"kind": "train", "volumes": rng.randint(1, 4), "frames": rng.randint(17, 64),
                "nz": 4 * rng.randint(4, 8), "nx": 32 * rng.randint(1, 2)}
    if kind == "filter":
        if rng.random() < 0.5:
            return {"kind": "filter", "frames": _log_int(rng, 24, 200), "nz": rng.randint(32, 256),
                    "nx": 128 * rng.randint(1, 2)}
        return {"kind": "filter", "frames": _log_int(rng, 24, 200), "nz": 4 * rng.randint(8, 64),
                "nx": 32 * rng.randint(1, 7)}
    if kind == "ensemble":
        if rng.random() < 0.25:
            return {"kind": "ensemble", "medium": "still", "scatterers": 2000, "frames": rng.randint(40, 100),
                    "nx": 64, "nz": 128}
        return {"kind": "ensemble", "medium": rng.choice(["moving", "compounded"]),
                "scatterers": _log_int(rng, 1000, 20_000), "frames": rng.randint(40, 100),
                "nx": rng.randint(40, 128), "nz": rng.randint(64, 160)}
    s_lo = _log_int(rng, 2000, 10_000)
    f_lo = rng.randint(40, 60)
    return {"kind": "batch", "members": rng.randint(2, 8), "s_lo": s_lo, "s_hi": s_lo * rng.randint(2, 6),
            "f_lo": f_lo, "f_hi": f_lo + rng.randint(10, 60)}


# ------------------------------------------------------------------ inputs --
def _probe(name):
    """The probes of the 2D plain, 2D compounded and 3D workloads."""
    if name == "linear64":
        return W.Probe(64, 1, 0.3e-3, 0.3e-3, 0.3e-3, 0.3e-3, 5e6, 20e6, 1540.0, 0.5, 2, 1024)
    if name == "linear128":
        return W.Probe(128, 1, 0.1e-3, 0.1e-3, 0.1e-3, 0.1e-3, 15.6e6, 62.5e6, 1540.0, 0.5, 2, 2048)
    return W.Probe(32, 32, 0.3e-3, 0.3e-3, 0.3e-3, 0.3e-3, 7.8e6, 31.25e6, 1540.0, 0.5, 2, 1536)


def _tilts(name):
    if name == "linear64":
        return np.zeros(1), np.zeros(1)
    if name == "linear128":
        return np.radians(np.linspace(-6.0, 6.0, 5)), np.zeros(5)
    t = np.radians(np.array([-5.0, 0.0, 5.0]))
    return np.repeat(t, 3), np.tile(t, 3)


def _field(name):
    """Field of view: x half-width, y half-width, z from, z to (m)."""
    return {"linear64": (10e-3, 0.0, 2e-3, 32e-3), "linear128": (6.4e-3, 0.0, 1e-3, 21e-3),
            "matrix32": (7.5e-3, 7.5e-3, 5e-3, 20e-3)}[name]


def _grid(probe, nx, ny, nz):
    xh, yh, z0, z1 = _field(probe)
    return W.Grid(nx, ny, nz, -xh, -yh if ny > 1 else 0.0, z0, 2 * xh / (nx - 1), 2 * yh / (ny - 1) if ny > 1 else 0.0,
                  (z1 - z0) / (nz - 1), 1.0)


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 7919 + 13)


def _uniform(g, n, lo, hi):
    return lo + (hi - lo) * torch.rand(n, generator=g, device=DEV, dtype=torch.float64)


def _inputs_rf(c, seed):
    """Scatterers uniform over the field of view, one in ten of them blood
    (20 dB weaker, moving 10 um a frame in a common direction); the tissue
    moves 50 um at 1 Hz, frames at 1 kHz."""
    g = _gen(seed)
    S, F = c["scatterers"], c["frames"]
    xh, yh, z0, z1 = _field(c["probe"])
    x = _uniform(g, S, -1.1 * xh, 1.1 * xh)
    y = _uniform(g, S, -yh, yh)
    z = _uniform(g, S, 0.9 * z0, z1 + 0.5e-3)
    amp = math.sqrt(2.0 / math.pi) * torch.sqrt(-2.0 * torch.log(1.0 - 0.999999 * _uniform(g, S, 0.0, 1.0)))
    blood = torch.arange(S, device=DEV) >= S - S // 10
    if c["base"]:
        blood[:] = True  # the tissue is in the base
    amp = torch.where(blood, 0.1 * amp, amp).float()
    t = torch.arange(F, device=DEV, dtype=torch.float64)[:, None] * 1e-3
    pos = torch.empty((F, 3, S), dtype=torch.float32, device=DEV)
    b = blood.double()[None, :]
    pos[:, 0] = (x[None] + b * 8e-3 * t).float()
    pos[:, 1] = y.float()[None]
    pos[:, 2] = (z[None] + 50e-6 * torch.sin(2 * math.pi * t) + b * 6e-3 * t).float()
    base = None
    if c["base"]:
        p = _probe(c["probe"])
        base = _speckle(g, len(_tilts(c["probe"])[0]) * p.n_elements, p) * 30.0
        base = base.reshape(1, -1, p.n_elements, p.n_samples)
    return pos, amp, base


def _speckle(g, lines, p):
    """Band-limited Gaussian noise about the carrier, [lines][samples]."""
    n = torch.arange(p.n_samples, device=DEV, dtype=torch.float64)
    ph = 2 * math.pi * p.f0 / p.fs * n
    w = torch.randn((2, lines, p.n_samples + 7), generator=g, device=DEV)
    env = sum(w[:, :, i:i + p.n_samples] for i in range(8)) / math.sqrt(8.0)
    return (env[0] * torch.cos(ph).float() + env[1] * torch.sin(ph).float()).contiguous()


def _inputs_beamform(c, seed):
    """RF [F][A][M][Ns]: two fixed speckle patterns whose mixture turns
    slowly from frame to frame (moving tissue) and 20 dB weaker patterns
    that change with every frame (blood)."""
    g = _gen(seed)
    p = _probe(c["probe"])
    A, M, F = len(_tilts(c["probe"])[0]), p.n_elements, c["frames"]
    s0, s1 = _speckle(g, A * M, p), _speckle(g, A * M, p)
    rf = torch.empty((F, A, M, p.n_samples), dtype=DTYPES[c["rf"]], device=DEV)
    for f in range(F):
        a = 0.5 * math.sin(2 * math.pi * 1e-3 * f)
        v = 10.0 * (math.cos(a) * s0 + math.sin(a) * s1) + torch.randn(s0.shape, generator=g, device=DEV)
        rf[f] = v.reshape(A, M, p.n_samples)
    return rf


def _inputs_clutter(c, seed):
    """Casorati matrix [P][F][2]: three slowly turning clutter components
    (20, 14 and 6 dB over the blood), blood of random Doppler shift and
    noise 26 dB below it."""
    g = _gen(seed)
    P, F = c["pixels"], c["frames"]
    out = torch.empty((P, F, 2), dtype=DTYPES[c["iq"]], device=DEV)
    t = torch.arange(F, device=DEV, dtype=torch.float32)[None]
    # temporal patterns of the clutter: nearly still, and two that turn
    basis = [torch.polar(1.0 + 0.05 * torch.sin(0.03 * (j + 1) * t), w * t + 0.4 * torch.sin(0.02 * (j + 1) * t))
             for j, w in enumerate((0.004, 0.09, -0.17))]
    step = 1 << 17
    for b in range(0, P, step):
        n = min(step, P - b)
        s = torch.zeros((n, F), dtype=torch.complex64, device=DEV)
        for lev, tb in zip((10.0, 5.0, 2.0), basis):
            s += lev * torch.randn((n, 1), generator=g, device=DEV, dtype=torch.complex64) * tb
        shift = 0.3 + 1.2 * torch.rand((n, 1), generator=g, device=DEV)
        amp = torch.randn((n, 1), generator=g, device=DEV, dtype=torch.complex64)
        s += amp * torch.polar(torch.ones_like(shift * t), shift * t)
        s += 0.05 * torch.randn((n, F), generator=g, device=DEV, dtype=torch.complex64)
        out[b:b + n] = torch.view_as_real(s)
    return out


def _inputs_motion(c, seed):
    if c["medium"] == "tree":
        return W.config3(seed=seed, n_frames=c["frames"], n_scat=c["scatterers"])
    return W.config2(seed=seed, n_frames=c["frames"], n_scat=c["scatterers"])


def _filter_layers(seed):
    """Weights as after training: He-normal hidden layers, a smaller last one."""
    rng = np.random.default_rng(seed)
    out = []
    for i, (a, b) in enumerate(zip(FILTER_CH[:-1], FILTER_CH[1:])):
        w = rng.standard_normal((45, a, b)) * np.sqrt(2.0 / (45 * a)) * (0.3 if i == 3 else 1.0)
        out.append((w.astype(np.float32), (0.05 * rng.standard_normal(b)).astype(np.float32)))
    return out


def _inputs_train(c, seed):
    """Normalised two-channel volumes (BF16, zero-padded to 32 channels) and
    FP32 targets that follow them in part."""
    g = _gen(seed)
    shape = (c["volumes"], c["frames"], c["nz"], c["nx"])
    x = torch.randn(shape + (2,), generator=g, device=DEV)
    x = (x + torch.roll(x, 1, 1) + torch.roll(x, 2, 1)) / math.sqrt(3.0)
    vol = torch.zeros(shape + (32,), dtype=torch.bfloat16, device=DEV)
    vol[..., :2] = x.bfloat16()
    tgt = (0.6 * x + 0.5 * torch.randn(shape + (2,), generator=g, device=DEV)).contiguous()
    return vol, tgt


def _compounded(seed, scatterers, frames, nx, nz):
    w = W.config2(seed=seed, n_frames=frames, n_scat=scatterers)
    w.grid = _grid("linear128", nx, 1, nz)
    return w


def _inputs_ensemble(c, seed):
    """The smallest workload (still tissue), its probe over moving tissue, or
    a small 2D compounded ensemble."""
    if c["medium"] == "still":
        return W.config1(seed=seed, n_frames=c["frames"])
    if c["medium"] == "moving":
        return learned.member(seed, c["frames"], c["nz"], c["nx"], c["scatterers"])
    return _compounded(seed, c["scatterers"], c["frames"], c["nx"], c["nz"])


def _inputs_batch(c, seed):
    """Members of both 2D probes; scatterers, frames and grids spread over
    the case's ranges."""
    n, out = c["members"], []
    for i in range(n):
        u, v = (i + 0.5) / n, ((7 * i + 3) % n + 0.5) / n
        s = int(round(math.exp(math.log(c["s_lo"]) * (1 - u) + math.log(c["s_hi"]) * u)))
        f = int(round(c["f_lo"] + v * (c["f_hi"] - c["f_lo"])))
        nx, nz = ((64, 64), (96, 80), (128, 128))[i % 3]
        out.append(_compounded(100 * seed + i, s, f, nx, nz) if i % 2 else
                   learned.member(100 * seed + i, f, nz, nx, s))
    return out


# ------------------------------------------------------------ prepare, run --
def prepare(case, seed):
    c, k = case, case["kind"]
    st = {"case": c}
    if k == "rf":
        p = _probe(c["probe"])
        st["probe"], st["tilts"] = p, _tilts(c["probe"])
        st["pos"], st["amp"], st["base"] = _inputs_rf(c, seed)
        st["rf"] = torch.empty((c["frames"], len(st["tilts"][0]), p.n_elements, p.n_samples),
                               dtype=DTYPES[c["rf"]], device=DEV)
    elif k == "beamform":
        p = _probe(c["probe"])
        st["probe"], st["tilts"] = p, _tilts(c["probe"])
        st["grid"] = _grid(c["probe"], c["nx"], c["ny"], c["nz"])
        st["rf"] = _inputs_beamform(c, seed)
        st["iq"] = torch.empty((st["grid"].n_pixels, c["frames"], 2), device=DEV)
        st["ws"] = fq.workspace(fq.fq_beamform_das_workspace_size(p, *st["tilts"], c["frames"], DTYPES[c["ch"]]))
    elif k == "clutter":
        st["iq"] = _inputs_clutter(c, seed)
        P, F = c["pixels"], c["frames"]
        st["out"] = {"iq_f": torch.empty_like(st["iq"]) if c["want_iq"] else None,
                     "pd": torch.empty(P, device=DEV),
                     "eigvals": torch.empty(F, dtype=torch.float64, device=DEV),
                     "k_used": torch.empty(1, dtype=torch.int32, device=DEV),
                     "ws": fq.workspace(fq.fq_clutter_svd_workspace_size(P, F, GRAM[c["gram"]]))}
    elif k == "motion":
        w = st["w"] = _inputs_motion(c, seed)
        st["in"] = [torch.from_numpy(np.ascontiguousarray(a)).to(DEV) for a in (w.p0, w.seg, w.flow, w.amp)]
        st["pos"] = torch.empty((c["frames"], 3, w.S), device=DEV)
        st["vessel"] = torch.empty(w.S, dtype=torch.int32, device=DEV)
        st["amp_eff"] = torch.empty(w.S, device=DEV)
    elif k == "train":
        st["net"] = fq.CNN(seed)
        st["net"].set_weights(_filter_layers(seed))
        st["vol"], st["tgt"] = _inputs_train(c, seed)
        st["acts"] = fq.cnn_act_workspace(c["volumes"], c["frames"], c["nz"], c["nx"])
        st["grads"] = st["net"].grads_buffer()
        st["loss"] = torch.zeros(1, device=DEV)
    elif k == "filter":
        F, Z, X = c["frames"], c["nz"], c["nx"]
        st["net"] = fq.CNN(seed)
        st["net"].set_weights(_filter_layers(seed))
        st["iq"] = _inputs_clutter({"pixels": Z * X, "frames": F, "iq": "f32"}, seed)
        st["vol"] = torch.empty((1, F, Z, X, 32), dtype=torch.bfloat16, device=DEV)
        st["acts"] = fq.cnn_act_workspace(1, F, Z, X)
        st["ws"] = fq.workspace(fq.lib().fq_cnn_prep_bytes(Z, X))
        st["scale"] = torch.empty(1, device=DEV)
        st["pd"] = torch.empty(Z * X, device=DEV)
    elif k == "ensemble":
        st["pl"] = Pipeline(_inputs_ensemble(c, seed))
        st["pl"].upload()
    else:
        st["batch"] = fq.Batch(_inputs_batch(c, seed))
        st["batch"].capture()
    return st


def run(state):
    c = state["case"]
    k = c["kind"]
    if k == "rf":
        return fq.fq_simulate_rf(state["probe"], *state["tilts"], state["pos"], state["amp"], c["frames"],
                                 rf_base=state["base"], rf=state["rf"])
    if k == "beamform":
        return fq.fq_beamform_das(state["probe"], *state["tilts"], state["rf"], c["frames"], state["grid"],
                                  ch_dtype=DTYPES[c["ch"]], iq=state["iq"], ws=state["ws"])
    if k == "clutter":
        o = state["out"]
        fq.fq_clutter_svd(state["iq"], c["k"], 0.9, GRAM[c["gram"]], want_iq_f=c["want_iq"], **o)
        out = {"pd": o["pd"], "k": o["k_used"]}
        if c["want_iq"]:
            out["iq_f"] = o["iq_f"]
        return out
    if k == "motion":
        w, (p0, seg, flow, amp) = state["w"], state["in"]
        fq.fq_classify_scatterers(p0, seg, w.segments, amp, state["vessel"], state["amp_eff"])
        fq.fq_advect_scatterers(p0, seg, flow, w.segments, w.motion, 0.0, 1.0 / w.prf, c["frames"], state["pos"])
        return {"vessel": state["vessel"], "amp": state["amp_eff"], "pos": state["pos"]}
    if k == "train":
        fq.fq_cnn_forward(state["net"], state["vol"], state["acts"])
        fq.fq_cnn_backward(state["net"], state["vol"], state["tgt"], state["acts"], state["grads"], state["loss"])
        y = fq.cnn_output(state["acts"], c["volumes"], c["frames"], c["nz"], c["nx"])
        return {"loss": state["loss"], "grads": state["grads"], "y": y[..., :2]}
    if k == "filter":
        F, Z, X = c["frames"], c["nz"], c["nx"]
        fq.fq_cnn_from_casorati(state["iq"], F, Z, X, scale_out=state["scale"], vol=state["vol"], ws=state["ws"])
        fq.fq_cnn_forward(state["net"], state["vol"], state["acts"])
        y = fq.cnn_output(state["acts"], 1, F, Z, X)[0]
        fq.fq_cnn_power_doppler(y, float(state["scale"].item()), pd=state["pd"])
        return {"y": y[..., :2], "pd": state["pd"]}
    if k == "ensemble":
        pl = state["pl"]
        pl.step()
        return {"rf": pl.rf, "iq": pl.iq, "pd": pl.pd, "k": pl.k_used}
    b = state["batch"]
    b.graph_launch()
    return {"pd": b.pd, "k": b.k_used}


# -------------------------------------------------------------------- work --
def _rf_flops(p, pairs):
    return pairs * (17.0 + 10.0 * p.n_cycles * p.fs / p.f0 + (5.0 if p.ny > 1 else 0.0))


def _das_terms(p, g, A):
    """Active (pixel, transmit, element) triples: the receive aperture
    |x - x_m| <= z / (2 f#), |y - y_m| <= z / (2 f#)."""
    z = g.z0 + g.dz * np.arange(g.nz)

    def active(n, pitch, lo, d, m):
        e = (np.arange(m) - 0.5 * (m - 1)) * pitch
        v = lo + d * np.arange(n)
        return (np.abs(v[:, None, None] - e[None, None, :]) <= (z / (2 * g.fnumber))[None, :, None]).sum(2)  # [n][nz]

    ax = active(g.nx, p.pitch_x, g.x0, g.dx, p.nx).sum(0)
    ay = active(g.ny, p.pitch_y, g.y0, g.dy, p.ny).sum(0) if p.ny > 1 else np.full(g.nz, g.ny)
    return float(A * (ax.astype(np.float64) * ay).sum())


def _work_rf(p, A, S, F, esz, base):
    return {"bytes": 12.0 * F * S + 4.0 * S + esz * F * A * p.n_elements * p.n_samples
            + (4.0 * A * p.n_elements * p.n_samples if base else 0.0),
            "flops": _rf_flops(p, float(S) * p.n_elements * A * F)}


def _work_beamform(p, A, g, F, esz):
    n = float(F) * A * p.n_elements * p.n_samples
    return {"bytes": esz * n + 8.0 * g.n_pixels * F,
            "flops": n * (2 + 4 * (4 * round(p.fs / p.f0) + 1)) + _das_terms(p, g, A) * (20.0 + 14.0 * F)}


def _work_clutter(P, F, esz, want, k=2):
    return {"bytes": esz * 2.0 * P * F * (2 if want else 1) + 4.0 * P,
            "flops": 4.0 * P * F * F + 16.0 * P * F * k}


def _work_motion(S, F, n_seg):
    return {"bytes": 12.0 * S * F + 28.0 * S + 12.0 * S, "flops": 20.0 * S * F + 20.0 * S * n_seg}


def _work_filter(V, pixels, train):
    macs = sum(45.0 * a * b for a, b in zip(FILTER_CH[:-1], FILTER_CH[1:]))
    if train:
        back = macs + 45.0 * (32 * 32 * 2 + 32 * 2)  # weight gradients, data gradients of three layers
        return {"bytes": V * (64.0 * 1 + 3 * 64 * 2 + 2 * 4 * 2), "flops": 2.0 * V * (macs + back)}
    return {"bytes": V * (8.0 + 8.0) + 4.0 * pixels, "flops": 2.0 * V * macs}


def _work_ensemble(w, esz=4):
    g, A, F = w.grid, w.A, w.n_frames
    parts = [_work_motion(w.S, F, len(w.segments)), _work_rf(w.probe, A, w.S, F, esz, False),
             _work_beamform(w.probe, A, g, F, esz), _work_clutter(g.n_pixels, F, 4, False)]
    return {"bytes": 28.0 * w.S + 4.0 * g.n_pixels, "flops": sum(p["flops"] for p in parts)}


def work(case):
    c, k = case, case["kind"]
    size = {"f32": 4.0, "bf16": 2.0, "f16": 2.0}
    if k == "rf":
        return _work_rf(_probe(c["probe"]), len(_tilts(c["probe"])[0]), c["scatterers"], c["frames"],
                        size[c["rf"]], c["base"])
    if k == "beamform":
        return _work_beamform(_probe(c["probe"]), len(_tilts(c["probe"])[0]),
                              _grid(c["probe"], c["nx"], c["ny"], c["nz"]), c["frames"], size[c["rf"]])
    if k == "clutter":
        return _work_clutter(c["pixels"], c["frames"], size[c["iq"]], c["want_iq"])
    if k == "motion":
        return _work_motion(c["scatterers"], c["frames"], 63 if c["medium"] == "tree" else 3)
    if k == "train":
        return _work_filter(float(c["volumes"]) * c["frames"] * c["nz"] * c["nx"], 0, True)
    if k == "filter":
        return _work_filter(float(c["frames"]) * c["nz"] * c["nx"], c["nz"] * c["nx"], False)
    ws = [_inputs_ensemble(c, 1)] if k == "ensemble" else _inputs_batch(c, 1)
    parts = [_work_ensemble(w) for w in ws]
    return {"bytes": sum(p["bytes"] for p in parts), "flops": sum(p["flops"] for p in parts)}


# ------------------------------------------------------------------- exact --
# The definitions in float64 (plain torch on the GPU).  Integer decisions
# that the path takes in binary32 (the receive aperture) are taken so here;
# positions are rounded to binary32 between the stages, as the path stores
# them.
F64 = torch.float64


def _elements(p):
    ex = (torch.arange(p.nx, device=DEV, dtype=F64) - 0.5 * (p.nx - 1)) * p.pitch_x
    ey = (torch.arange(p.ny, device=DEV, dtype=F64) - 0.5 * (p.ny - 1)) * p.pitch_y
    return ex.repeat(p.ny), ey.repeat_interleave(p.nx)


def _directions(p, tilts):
    ex, ey = _elements(p)
    out = []
    for tx, ty in zip(*tilts):
        ux, uy = math.sin(tx), math.sin(ty)
        out.append((ux, uy, math.sqrt(1.0 - ux * ux - uy * uy), float((ux * ex + uy * ey).min())))
    return out


def _exact_rf(p, tilts, pos, amp, base):
    F, _, S = pos.shape
    ex, ey = _elements(p)
    dirs = _directions(p, tilts)
    M, ns = p.n_elements, p.n_samples
    T, k0 = p.n_cycles / p.f0, 2 * math.pi * p.f0 / p.c
    alpha = p.alpha_db_cm_mhz * 100.0 / (20.0 / math.log(10.0)) * p.f0 * 1e-6
    rf = torch.zeros((F, len(dirs), M * ns + 1), dtype=F64, device=DEV)
    half = 0.5 * T * p.fs
    taps = int(math.floor(2 * half)) + 1
    step = max(1, min(S, int(4e6 // M)))

    def sinc(v):
        return torch.where(v == 0, torch.ones_like(v), torch.sin(v) / torch.where(v == 0, torch.ones_like(v), v))

    for f in range(F):
        for b in range(0, S, step):
            x, y, z = (pos[f, d, b:b + step].to(F64)[:, None] for d in range(3))
            a0 = amp[b:b + step].to(F64)[:, None]
            dx, dy = x - ex[None], y - ey[None]
            r = torch.sqrt(dx * dx + dy * dy + z * z)
            D = sinc(k0 * 0.5 * p.width_x * dx / r)
            if p.ny > 1:
                D = D * sinc(k0 * 0.5 * p.width_y * dy / r)
            for i, (ux, uy, uz, org) in enumerate(dirs):
                path = ux * x + uy * y + uz * z - org + r
                A = a0 * D * torch.exp(-alpha * path) / r
                u = path / p.c * p.fs
                first = torch.ceil(u - half)
                line = torch.arange(M, device=DEV)[None] * ns
                for j in range(taps):
                    k = first + j
                    t = (k - u) / p.fs
                    v = A * 0.5 * (1 + torch.cos(2 * math.pi * t / T)) * torch.cos(2 * math.pi * p.f0 * t)
                    ok = (k >= 0) & (k <= ns - 1) & (t.abs() < 0.5 * T)
                    idx = torch.where(ok, line + k.long().clamp(0, ns - 1), M * ns)
                    rf[f, i].index_add_(0, idx.reshape(-1), torch.where(ok, v, torch.zeros_like(v)).reshape(-1))
    rf = rf[:, :, :-1].reshape(F, len(dirs), M, ns)
    return rf + base.to(F64) if base is not None else rf


def _exact_channel_iq(p, rf):
    """[F][A][M][Ns] -> complex128 [A M][Ns][F]"""
    F = rf.shape[0]
    ns = p.n_samples
    J = 2 * int(round(p.fs / p.f0))
    j = torch.arange(-J, J + 1, device=DEV, dtype=F64)
    fc = 2.0 * p.f0 / p.fs
    h = fc * torch.sinc(fc * j) * 0.5 * (1 + torch.cos(math.pi * j / (J + 1)))
    h = h / h.sum()
    n = torch.arange(ns, device=DEV, dtype=F64)
    mix = torch.polar(torch.ones_like(n), -2 * math.pi * p.f0 * n / p.fs)
    lines = rf.shape[1] * rf.shape[2]
    out = torch.empty((lines, ns, F), dtype=torch.complex128, device=DEV)
    for f in range(F):
        m = torch.nn.functional.pad(rf[f].to(F64).reshape(lines, ns) * mix, (J, J))
        acc = torch.zeros((lines, ns), dtype=torch.complex128, device=DEV)
        for i in range(2 * J + 1):  # sample k - j sits at k - j + J of the padded row
            acc += h[i] * m[:, 2 * J - i:2 * J - i + ns]
        out[:, :, f] = 2 * acc
    return out


def _exact_das(p, tilts, ch, g, F):
    ex, ey = _elements(p)
    dirs = _directions(p, tilts)
    M, ns = p.n_elements, p.n_samples
    ix = torch.arange(g.nx, device=DEV, dtype=F64)
    iy = torch.arange(g.ny, device=DEV, dtype=F64)
    iz = torch.arange(g.nz, device=DEV, dtype=F64)
    y, z, x = torch.meshgrid(g.y0 + iy * g.dy, g.z0 + iz * g.dz, g.x0 + ix * g.dx, indexing="ij")
    x, y, z = x.reshape(-1), y.reshape(-1), z.reshape(-1)
    half = z.float() * torch.tensor(0.5 / g.fnumber, dtype=torch.float32, device=DEV)
    out = torch.zeros((x.numel(), F), dtype=torch.complex128, device=DEV)
    for m in range(M):
        ok = (x.float() - ex[m].float()).abs() <= half
        if p.ny > 1:
            ok &= (y.float() - ey[m].float()).abs() <= half
        sel = ok.nonzero().reshape(-1)
        if not sel.numel():
            continue
        xs, ys, zs = x[sel], y[sel], z[sel]
        r = torch.sqrt((xs - ex[m]) ** 2 + (ys - ey[m]) ** 2 + zs * zs)
        for a, (ux, uy, uz, org) in enumerate(dirs):
            tau = (ux * xs + uy * ys + uz * zs - org + r) / p.c
            u = tau * p.fs
            i = torch.floor(u)
            phi = (u - i)[:, None]
            il = i.long()
            inside = (il >= 0) & (il + 1 < ns)
            il = il.clamp(0, ns - 2)
            rows = ch[a * M + m]
            v = (1 - phi) * rows[il] + phi * rows[il + 1]
            rot = torch.polar(inside.to(F64), 2 * math.pi * p.f0 * tau)
            out.index_add_(0, sel, v * rot[:, None])
    return out / len(dirs)


def _exact_pd(s, k, thresh=0.9):
    """(power Doppler, filtered matrix, k) of the complex128 matrix s [P][F]."""
    G = s.mH @ s
    lam, V = torch.linalg.eigh(G)
    lam, V = lam.flip(0).clamp(min=0), V.flip(1)
    if k < 0:
        k = int((torch.cumsum(lam, 0) < thresh * lam.sum()).sum()) + 1
    V = V[:, :k]
    sf = s - (s @ V) @ V.mH
    return (sf.real ** 2 + sf.imag ** 2).mean(1), sf, k


def _exact_motion(w, F):
    """(positions [F][3][S], vessel [S], amplitude [S])"""
    t = (torch.arange(F, device=DEV, dtype=F64) / w.prf)[:, None, None]
    p0, flow = (torch.from_numpy(np.ascontiguousarray(a)).to(DEV).to(F64) for a in (w.p0, w.flow))
    seg = torch.from_numpy(np.ascontiguousarray(w.seg)).to(DEV).long()
    pos = p0[None].expand(F, 3, w.S).clone()
    vessel = seg.clone()
    for i, s in enumerate(w.segments):
        a1, a2, a3, c0 = (torch.tensor(v, device=DEV, dtype=F64)[:, None] for v in (s.a1, s.a2, s.a3, s.p0))
        q, x1, x2 = flow
        idx = (seg == i).nonzero().reshape(-1)
        q, x1, x2 = q[idx][None], x1[idx][None], x2[idx][None]
        v = s.vmax * (1.0 - (x1 * x1 + x2 * x2) / s.radius ** 2)
        if s.kind == W.SEG_LINE:
            a = torch.remainder(q + v * t[:, 0], s.length)
            pos[:, :, idx] = c0[None] + a[:, None] * a1[None] + x1[None] * a2[None] + x2[None] * a3[None]
        else:
            a = torch.remainder(q + v * t[:, 0] / s.arc_radius, s.phi1)
            rr = (s.arc_radius + x1)[:, None]
            pos[:, :, idx] = (c0[None] + rr * (torch.cos(a)[:, None] * a1[None] + torch.sin(a)[:, None] * a2[None])
                              + x2[None] * a3[None])
        d = p0 - c0
        u1, u2, u3 = (d * a1).sum(0), (d * a2).sum(0), (d * a3).sum(0)
        if s.kind == W.SEG_LINE:
            inside = (u1 >= 0) & (u1 <= s.length) & (u2 * u2 + u3 * u3 < s.radius ** 2)
        else:
            rin = torch.sqrt(u1 * u1 + u2 * u2) - s.arc_radius
            inside = (u2 >= 0) & (u1 * s.arc_end[1] - u2 * s.arc_end[0] >= 0) & (rin * rin + u3 * u3 < s.radius ** 2)
        vessel = torch.where((vessel < 0) & inside, torch.full_like(vessel, i), vessel)
    m = w.motion
    gain = 1.0 + ((pos - torch.tensor(m.elastic_center, device=DEV, dtype=F64)[None, :, None])
                  * torch.tensor(m.elastic_grad, device=DEV, dtype=F64)[None, :, None]).sum(1, keepdim=True)
    assert not any(m.omega)
    disp = sum((a * torch.sin(2 * math.pi * f * t + ph) * torch.tensor(d, device=DEV, dtype=F64)[None, :, None]
                for a, f, ph, d in zip(m.amp, m.freq, m.phase, m.dir)), torch.zeros_like(t))
    pos = pos + t * torch.tensor(m.vel, device=DEV, dtype=F64)[None, :, None] + gain * disp
    amp = torch.from_numpy(np.ascontiguousarray(w.amp)).to(DEV).to(F64)
    return pos, vessel, torch.where((seg < 0) & (vessel >= 0), torch.zeros_like(amp), amp)


TAPS = [(dt, dz, dx) for dt in range(-2, 3) for dz in range(-1, 2) for dx in range(-1, 2)]


def _shift(x, d):
    """y[v] = x[v + d], zero outside the volume (x [N][F][Z][X][C])"""
    for axis, n in zip((1, 2, 3), d):
        if n:
            y = torch.zeros_like(x)
            m = x.shape[axis] - abs(n)
            if m > 0:
                y.narrow(axis, max(0, -n), m).copy_(x.narrow(axis, max(0, n), m))
            x = y
    return x


def _exact_forward(layers, x):
    acts = [x]
    for i, (w, b) in enumerate(layers):
        y = torch.zeros(x.shape[:-1] + (w.shape[2],), dtype=F64, device=DEV) + b
        for t, d in enumerate(TAPS):
            y += _shift(acts[-1], d) @ w[t]
        acts.append(y if i == 3 else y.clamp(min=0))
    return acts


def _exact_train(case, seed):
    layers = [(torch.from_numpy(w).to(DEV).to(F64), torch.from_numpy(b).to(DEV).to(F64))
              for w, b in _filter_layers(seed)]
    vol, tgt = _inputs_train(case, seed)
    acts = _exact_forward(layers, vol[..., :2].to(F64))
    e = acts[4] - tgt.to(F64)
    loss = (e * e).mean().reshape(1)
    dy = 2 * e / e.numel()
    gw = torch.zeros((4, 45, 32, 32), dtype=F64, device=DEV)
    gb = torch.zeros((4, 32), dtype=F64, device=DEV)
    for i in (3, 2, 1, 0):
        w, _ = layers[i]
        a, b = w.shape[1:]
        flat = dy.reshape(-1, b)
        gb[i, :b] = flat.sum(0)
        dx = torch.zeros_like(acts[i]) if i else None
        for t, d in enumerate(TAPS):
            gw[i, t, :a, :b] = _shift(acts[i], d).reshape(-1, a).T @ flat
            if i:
                dx += _shift(dy, tuple(-v for v in d)) @ w[t].T
        if i:
            dy = dx * (acts[i] > 0)
    return {"loss": loss, "grads": torch.cat([gw.reshape(-1), gb.reshape(-1)]), "y": acts[4]}


def _exact_filter(case, seed):
    layers = [(torch.from_numpy(w).to(DEV).to(F64), torch.from_numpy(b).to(DEV).to(F64))
              for w, b in _filter_layers(seed)]
    F, Z, X = case["frames"], case["nz"], case["nx"]
    s = _inputs_clutter({"pixels": Z * X, "frames": F, "iq": "f32"}, seed).to(F64)
    s = s - s.mean(1, keepdim=True)
    scale = 1.0 / torch.sqrt((s * s).mean())
    x = (s * scale).permute(1, 0, 2).reshape(1, F, Z, X, 2).contiguous()
    y = _exact_forward(layers, x)[4][0]
    pd = (y * y).sum(3).mean(0).reshape(-1) / (scale * scale)
    return {"y": y, "pd": pd}


def exact(case, seed):
    c, k = case, case["kind"]
    if k == "rf":
        p = _probe(c["probe"])
        if float(c["scatterers"]) * p.n_elements * len(_tilts(c["probe"])[0]) * c["frames"] > 1.5e9:
            return None
        pos, amp, base = _inputs_rf(c, seed)
        return _exact_rf(p, _tilts(c["probe"]), pos, amp, base)
    if k == "beamform":
        p, tilts = _probe(c["probe"]), _tilts(c["probe"])
        g = _grid(c["probe"], c["nx"], c["ny"], c["nz"])
        if _das_terms(p, g, len(tilts[0])) * c["frames"] > 1.5e10:
            return None
        rf = _inputs_beamform(c, seed)
        return torch.view_as_real(_exact_das(p, tilts, _exact_channel_iq(p, rf), g, c["frames"]))
    if k == "clutter":
        s = torch.view_as_complex(_inputs_clutter(c, seed).to(F64))
        pd, sf, _ = _exact_pd(s, c["k"])
        out = {"pd": pd, "k": None}
        if c["want_iq"]:
            out["iq_f"] = torch.view_as_real(sf)
        return out
    if k == "motion":
        pos, _, amp = _exact_motion(_inputs_motion(c, seed), c["frames"])
        return {"vessel": None, "amp": amp, "pos": pos}
    if k == "train":
        return _exact_train(c, seed)
    if k == "filter":
        return _exact_filter(c, seed)
    if k == "ensemble":
        w = _inputs_ensemble(c, seed)
        tilts = (w.tilt_x, w.tilt_y)
        if float(w.S) * w.M * w.A * w.n_frames > 1.5e9:
            return None
        pos, _, amp = _exact_motion(w, w.n_frames)
        rf = _exact_rf(w.probe, tilts, pos.float(), amp, None)
        iq = _exact_das(w.probe, tilts, _exact_channel_iq(w.probe, rf), w.grid, w.n_frames)
        return {"rf": rf, "iq": torch.view_as_real(iq), "pd": _exact_pd(iq, w.k_cut)[0], "k": None}
    return None

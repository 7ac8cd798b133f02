"""The hot kernels at the edges of their layouts: angle blocks and record
segments of the RF kernel, pixel panels and column blocks of the FP32 Gram,
register blocks of the tridiagonalisation, frame groups and voxel pairs of
the 16-bit delay-and-sum, accumulator runs of the convolution."""
import threading

import numpy as np
import pytest
import torch

import oracle
from oracle import cnn as ocnn
from paper_2509_05464_gb300 import build as fqbuild
from paper_2509_05464_gb300 import fq
from paper_2509_05464_gb300 import workload as W
from paper_2509_05464_gb300.pipeline import Pipeline

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    fqbuild.build()
    fq.lib()


def rel_l2(a, b):
    return float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(b.ravel()))


# blocks of 8, 4, 2 and 1 angles and their sums; record lengths around whole
# segments (the shortest: segments of their least 8 samples), aligned and not;
# echoes from before the record to past its end.  Bars as for the other RF
# routes: 1e-5 in FP32, the storage rounding in 16 bits.
@pytest.mark.parametrize("A", [1, 2, 3, 5, 7, 8, 9, 11])
@pytest.mark.parametrize("ns,dt", [(40, "f32"), (301, "f32"), (1000, "f32"), (1000, "bf16"), (999, "f16")])
def test_rf_angle_blocks_and_segments(A, ns, dt):
    p = W.Probe(8, 1, 0.1e-3, 0.1e-3, 0.1e-3, 0.1e-3, 15.6e6, 62.5e6, 1540.0, 0.5, 2, ns)
    rng = np.random.default_rng(100 * A + ns)
    S, z1 = 517, 1.15 * ns * 1540.0 / 62.5e6 / 2
    pos = np.stack([rng.uniform(-1e-3, 1e-3, S), np.zeros(S), rng.uniform(0.02e-3, z1, S)]).astype(np.float32)
    amp = rng.standard_normal(S).astype(np.float32)
    tx = list(np.radians(np.linspace(-6.0, 6.0, A))) if A > 1 else [0.0]
    base = rng.standard_normal((A, 8, ns)).astype(np.float32)
    t = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}[dt]
    for b in (None, base):
        got = fq.fq_simulate_rf(p, tx, [0.0] * A, torch.from_numpy(pos[None]).cuda(), torch.from_numpy(amp).cuda(), 1,
                                rf_base=None if b is None else torch.from_numpy(b).cuda(), out_dtype=t)
        want = oracle.simulate_rf(p, tx, [0.0] * A, pos, amp, rf=None if b is None else b.astype(np.float64),
                                  accumulate=b is not None)
        err = rel_l2(got[0].float().cpu().numpy().astype(np.float64), want)
        assert err <= {"f32": 1e-5, "bf16": 1e-2, "f16": 1e-3}[dt], (b is None, err)


# products of a sum of 2 P terms in binary32, any order: within gamma_2P of
# the sum of magnitudes
@pytest.mark.parametrize("F", [2, 3, 4, 5, 31, 100, 130, 201, 260])
@pytest.mark.parametrize("P,dt", [(1, "f32"), (15, "f32"), (33, "f32"), (1000, "f32"), (5003, "f32"), (1000, "bf16")])
def test_gram_panels(F, P, dt):
    g = torch.Generator(device="cuda").manual_seed(F * 1000 + P)
    S = torch.randn((P, F, 2), generator=g, device="cuda").to(torch.float32 if dt == "f32" else torch.bfloat16)
    G = torch.view_as_complex(fq.fq_casorati_gram(S).double().contiguous())
    s = torch.view_as_complex(S.double().contiguous())
    mag = (S.double().abs().sum(2)).mT @ S.double().abs().sum(2)
    err = (G - s.mH @ s).abs()
    assert bool((err <= 2.0 ** -24 * (2 * P + 16) * mag).all())


# register blocks of 32 columns, the shared-memory limit (220) and beyond;
# eigenvalues within 2 F 2^-24 of the largest, and with them the filtered
# energy of the pixels
@pytest.mark.parametrize("F", [2, 3, 5, 32, 33, 65, 128, 129, 200, 221, 300])
def test_eigen_blocks(F):
    g = torch.Generator(device="cuda").manual_seed(F)
    P, k = 700, min(3, F - 1)
    lev = torch.tensor([100.0, 40.0, 20.0], device="cuda")[:k]
    U = torch.randn((P, k), generator=g, device="cuda", dtype=torch.complex64)
    V = torch.linalg.qr(torch.randn((F, k), generator=g, device="cuda", dtype=torch.complex64))[0]
    s = (U * lev) @ V.mH + 0.3 * torch.randn((P, F), generator=g, device="cuda", dtype=torch.complex64)
    pd, ev = torch.empty(P, device="cuda"), torch.empty(F, dtype=torch.float64, device="cuda")
    S = torch.view_as_real(s).contiguous()
    fq.fq_clutter_svd(S, k_cut=k, want_iq_f=False, pd=pd, eigvals=ev)
    s64 = s.to(torch.complex128)
    lam, vec = torch.linalg.eigh(s64.mH @ s64)
    lam, vec = lam.flip(0), vec.flip(1)[:, :k]
    assert float((ev - lam).abs().max()) <= (2 * F * 2.0 ** -24 + 2.0 ** -22) * float(lam[0])
    sf = s64 - (s64 @ vec) @ vec.mH
    want = (sf.real ** 2 + sf.imag ** 2).mean(1)
    assert rel_l2(pd.double().cpu().numpy(), want.cpu().numpy()) <= 1e-3


# 16-bit channel data against the FP32 kernel on the same values: the
# interpolation rounds b - a, its weight and the result to u, so a term is
# within u (2 |b - a| + |v|), at most ~4 u of it on white data
@pytest.mark.parametrize("dt,u", [(torch.bfloat16, 2.0 ** -8), (torch.float16, 2.0 ** -11)])
@pytest.mark.parametrize("F", [1, 17, 64, 65, 100, 129, 200])
@pytest.mark.parametrize("nx,matrix", [(1, False), (17, False), (37, False), (19, True)])
def test_das_frame_groups_and_voxel_pairs(dt, u, F, nx, matrix):
    p = (W.Probe(8, 6, 0.3e-3, 0.3e-3, 0.3e-3, 0.3e-3, 7.8e6, 31.25e6, 1540.0, 0.5, 2, 500) if matrix else
         W.Probe(40, 1, 0.1e-3, 0.1e-3, 0.1e-3, 0.1e-3, 15.6e6, 62.5e6, 1540.0, 0.5, 2, 500))
    ny = 3 if matrix else 1
    grid = W.Grid(nx, ny, 9, -1.9e-3, -0.4e-3 if matrix else 0.0, 1e-3, 0.11e-3, 0.4e-3 if matrix else 0.0, 0.55e-3, 1.0)
    tx = [-0.06, 0.0, 0.06]
    g = torch.Generator(device="cuda").manual_seed(F + nx)
    ch = torch.randn((3 * p.nx * p.ny, p.n_samples, fq.frame_pad(F), 2), generator=g, device="cuda").to(dt)
    got = fq.fq_das(p, tx, [0.0] * 3, ch, F, grid)
    want = fq.fq_das(p, tx, [0.0] * 3, ch.float(), F, grid)
    assert rel_l2(got.double().cpu().numpy(), want.double().cpu().numpy()) <= 4 * u
    for f in {0, F // 2, F - 1}:
        assert rel_l2(got[:, f].double().cpu().numpy(), want[:, f].double().cpu().numpy()) <= 8 * u


# runs of one to many frames (every number of new and finished outputs), both
# tiles (a depth that is not a multiple of 4 takes the 128-pixel rows)
@pytest.mark.parametrize("shape", [(1, 1, 4, 32), (1, 2, 4, 32), (1, 3, 3, 128), (2, 4, 1, 128), (1, 5, 8, 96),
                                   (1, 9, 4, 160), (1, 33, 2, 128), (3, 17, 4, 32)])
def test_conv_frame_runs(shape):
    n, F, Z, X = shape
    rng = np.random.default_rng(sum(shape))
    layers = [(rng.standard_normal((45, 32, 32)) * np.sqrt(2.0 / 1440), rng.standard_normal(32) * 0.1) for _ in range(4)]
    net = fq.CNN(3)
    net.set_weights(layers)
    x = torch.from_numpy(rng.standard_normal(shape + (32,)).astype(np.float32)).bfloat16().cuda()
    w = torch.from_numpy(layers[1][0].astype(np.float32)).bfloat16().double().numpy()
    b = layers[1][1].astype(np.float32).astype(np.float64)
    x64 = x.double().cpu().numpy()
    ref = np.stack([ocnn.conv3d(x64[i], w, b) for i in range(n)])
    out = torch.empty(shape + (32,), dtype=torch.float32, device="cuda")
    fq.fq_cnn_conv(fq.CNN_MODE_LINEAR, x, net, 1, 0, out)
    torch.cuda.synchronize()
    assert int(net.status.item()) == 0
    # FP32 sums of at most 1440 exact products of BF16 values
    assert np.abs(out.double().cpu().numpy() - ref).max() <= 1e-5 * np.abs(ref).max()


def test_batch_of_small_and_large_eigen_problems():
    """Members on both sides of the shared-memory limit of the eigen step in one
    wave: each gives exactly what its single call gives."""
    ms = [w for i, F in enumerate((240, 100, 222, 40))
          for w in W.config4(seed=80 + i, n=1, s_range=(300, 800), f_range=(F, F), grids=((16, 1, 24),))]
    b = fq.Batch(ms)
    b.launch()
    b.status()
    torch.cuda.synchronize()
    for i, w in enumerate(ms):
        pl = Pipeline(w)
        pl.upload()
        pl.step()
        fq.fq_clutter_status(pl.ws_svd)
        torch.cuda.synchronize()
        assert int(b.k_used[i].cpu()[0]) == int(pl.k_used.cpu()[0]), i
        assert torch.equal(b.eigvals[i], pl.eigvals), i
        assert torch.equal(b.pd[i], pl.pd), i


@pytest.mark.parametrize("F,Z,X", [(1, 1, 1), (15, 3, 5), (16, 5, 7), (33, 2, 33), (48, 9, 29), (65, 4, 16)])
@pytest.mark.parametrize("remove_mean", [True, False])
def test_filter_volume_frame_batches(F, Z, X, remove_mean):
    """The learned filter's volume, target and power Doppler for frame counts
    around the batches of loads: elementwise FP32 sums against FP64."""
    g = torch.Generator(device="cuda").manual_seed(F)
    iq = torch.randn((Z * X, F, 2), generator=g, device="cuda") + 0.5
    vol = torch.full((F, Z, X, 32), 7.0, device="cuda", dtype=torch.bfloat16)
    tgt = torch.empty((F, Z, X, 2), device="cuda")
    _, _, sc = fq.fq_cnn_from_casorati(iq, F, Z, X, remove_mean, gain=2.0, vol=vol, target=tgt)
    d = iq.double()
    d = d - d.mean(1, keepdim=True) if remove_mean else d
    sc_ref = 1.0 / d.square().mean().sqrt() if (F > 1 or not remove_mean) else sc.double()
    eps = 2.0 ** -23
    assert torch.allclose(sc.double().reshape(()), sc_ref.reshape(()), rtol=(F + 8) * eps, atol=0)
    ref = (d * sc.double() * 2.0).permute(1, 0, 2).reshape(F, Z, X, 2)
    # the mean of F values of size <= 6 and three roundings of the product
    tol = ((F + 4) * eps * 6 * 2.0 * sc.double()).item()
    assert (tgt.double() - ref).abs().max().item() <= tol
    assert torch.equal(vol[..., :2], tgt.to(torch.bfloat16)) and not vol[..., 2:].any()
    y = torch.randn((F, Z, X, 32), generator=g, device="cuda")
    pd = fq.fq_cnn_power_doppler(y, 0.5)
    pd_ref = y[..., :2].double().square().sum(-1).mean(0) / 0.25
    assert ((pd.double().reshape(Z, X) - pd_ref).abs() <= (F + 6) * eps * pd_ref).all()


# records too short for echoes clear of both ends (at most 2 dmax + 9 samples,
# dmax = ceil(3 pitch fs / c) + 2: 39 at 0.1 mm, 257 at 1 mm) up to the first
# length that has them, in blocks of 1, 4 + 1, 8 and 8 + 1 angles.  FP32 bar:
# 5e-6 and the phase of four roundings (of the difference of squares, the
# root, the reciprocal, the product) of an element's delay offset from its
# quad's first, at most 3 pitches
@pytest.mark.parametrize("A", [1, 5, 8, 9])
@pytest.mark.parametrize("ns,pitch", [(9, 0.1e-3), (16, 0.1e-3), (38, 0.1e-3), (39, 0.1e-3), (40, 0.1e-3),
                                      (128, 1e-3), (256, 1e-3), (257, 1e-3), (258, 1e-3)])
@pytest.mark.parametrize("dt", ["f32", "bf16", "f16"])
def test_rf_short_records(A, ns, pitch, dt):
    p = W.Probe(8, 1, pitch, pitch, 0.1e-3, 0.1e-3, 15.6e6, 62.5e6, 1540.0, 0.5, 2, ns)
    rng = np.random.default_rng(100 * A + ns)
    S, z1 = 517, 1.15 * ns * 1540.0 / 62.5e6 / 2
    pos = np.stack([rng.uniform(-5 * pitch, 5 * pitch, S), np.zeros(S), rng.uniform(0.02e-3, z1, S)]).astype(np.float32)
    amp = 1e-3 * rng.standard_normal(S).astype(np.float32)  # (1 / r is up to 5e4 here)
    tx = list(np.radians(np.linspace(-6.0, 6.0, A))) if A > 1 else [0.0]
    base = rng.standard_normal((A, 8, ns)).astype(np.float32)
    t = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}[dt]
    for b in (None, base):
        got = fq.fq_simulate_rf(p, tx, [0.0] * A, torch.from_numpy(pos[None]).cuda(), torch.from_numpy(amp).cuda(), 1,
                                rf_base=None if b is None else torch.from_numpy(b).cuda(), out_dtype=t)
        want = oracle.simulate_rf(p, tx, [0.0] * A, pos, amp, rf=None if b is None else b.astype(np.float64),
                                  accumulate=b is not None)
        err = rel_l2(got[0].float().cpu().numpy().astype(np.float64), want)
        f32 = 5e-6 + 2 * np.pi * p.f0 * 3 * pitch / p.c * 2.0 ** -22
        assert err <= {"f32": f32, "bf16": 1e-2, "f16": 1e-3}[dt], (b is None, err)


# every step of the filter scales by powers of two exactly, so an ensemble times
# 2^n gives the same result times 2^n, bit for bit (eigenvalues and power
# Doppler times 4^n); at 2^40 the largest eigenvalue is ~5e31
@pytest.mark.parametrize("F,k", [(100, 1), (100, 2), (100, 8), (240, 2)])
@pytest.mark.parametrize("form", ["f32", "bf16", "tf32 gram", "bf16 gram", "noalloc"])
def test_clutter_filter_at_any_amplitude(F, k, form):
    g = torch.Generator(device="cuda").manual_seed(F + k)
    lev = 100.0 * 0.8 ** torch.arange(k, device="cuda")
    U = torch.randn((4096, k), generator=g, device="cuda", dtype=torch.complex64)
    V = torch.linalg.qr(torch.randn((F, k), generator=g, device="cuda", dtype=torch.complex64))[0]
    s = (U * lev) @ V.mH + 0.3 * torch.randn((4096, F), generator=g, device="cuda", dtype=torch.complex64)
    S = torch.view_as_real(s).to(torch.bfloat16 if form == "bf16" else torch.float32).contiguous()
    mode = {"tf32 gram": fq.FQ_GRAM_TF32, "bf16 gram": fq.FQ_GRAM_BF16}.get(form, fq.FQ_GRAM_F32)

    def run(n):
        x = S * 2.0 ** n
        o = fq.fq_clutter_svd_noalloc(x, k) if form == "noalloc" else fq.fq_clutter_svd(x, k, gram_mode=mode)
        return o["iq_f"].double() * 2.0 ** -n, o["pd"].double() * 4.0 ** -n, o["eigvals"] * 4.0 ** -n

    want = run(0)
    assert float(want[1].mean()) < 2.0 * 2 * 0.3 ** 2  # the components are gone, the noise is left
    for n in (-40, -20, 20, 40):
        for a, b in zip(run(n), want):
            assert torch.equal(a, b), n


def test_batch_at_any_amplitude():
    ms = W.config4(seed=90, n=2, s_range=(300, 800), f_range=(60, 80), grids=((32, 1, 48),))
    out = []
    for n in (0, -40, 24):
        for w in ms:
            w.amp = (w.amp * np.float32(2.0 ** n)).astype(np.float32)
        b = fq.Batch(ms)
        b.launch()
        b.status()
        out.append([p.double() * 4.0 ** -n for p in b.pd])
        for w in ms:
            w.amp = (w.amp * np.float32(2.0 ** -n)).astype(np.float32)
    for o in out[1:]:
        for a, b in zip(o, out[0]):
            assert torch.equal(a, b)


def test_threads_with_different_frame_counts():
    """Gram matrices of 40 and 200 frames (less and more than 48 KB of shared
    memory) from threads on their own streams: no call takes back what
    another is about to launch with (a race: seen in one of 40000 launches)."""
    errors = []

    def work(F):
        try:
            g = torch.Generator(device="cuda").manual_seed(F)
            S = torch.randn((8, F, 2), generator=g, device="cuda")
            want, G = fq.fq_casorati_gram(S), torch.empty((F, F, 2), device="cuda")
            torch.cuda.synchronize()
            ws, st = fq.workspace(fq.fq_gram_workspace_size(8, F)), torch.cuda.Stream()
            for _ in range(20000):
                fq.fq_casorati_gram(S, G=G, ws=ws, stream=st)
            st.synchronize()
            assert torch.equal(G, want), F
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    ts = [threading.Thread(target=work, args=(F,)) for F in (40, 200, 40, 200, 40)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errors, errors


# F reflectors, each unitary to its rounding, and unit vectors at the end: V^H V
# within (F + 8) 2^-24 of the identity
@pytest.mark.parametrize("F", [2, 3, 5, 40, 100, 128, 160, 220, 221, 300])
def test_eigenvectors_are_orthonormal(F):
    g = torch.Generator(device="cuda").manual_seed(F)
    A = torch.randn((2 * F, F), generator=g, device="cuda", dtype=torch.complex128)
    G = torch.view_as_real((A.mH @ A).to(torch.complex64)).contiguous()
    lam, V, ws = fq.fq_hermitian_eig(G)
    fq.fq_clutter_status(ws)
    V = torch.view_as_complex(V.double())
    G64 = torch.view_as_complex(G.double())
    assert float((V.mH @ V - torch.eye(F, device="cuda")).abs().max()) <= (F + 8) * 2.0 ** -24
    assert float((G64 @ V - V * lam).norm()) <= 2 * F * 2.0 ** -24 * float(G64.norm())


# components removed without the subspace step (more than 8), with the solves'
# scratch in and beyond the matrix's storage; eigenvalues within 2 F 2^-24 of
# the largest turn the subspace by that over the gap
@pytest.mark.parametrize("F", [60, 130, 160, 220, 240])
@pytest.mark.parametrize("k", [0, 1, 8, 9, 24, 48])
def test_filtered_iq_of_many_components(F, k):
    g = torch.Generator(device="cuda").manual_seed(1000 * k + F)
    lev = torch.linspace(100.0, 50.0, max(k, 1), device="cuda")[:k]
    U = torch.randn((4096, k), generator=g, device="cuda", dtype=torch.complex64)
    V = torch.linalg.qr(torch.randn((F, max(k, 1)), generator=g, device="cuda", dtype=torch.complex64))[0][:, :k]
    s = (U * lev) @ V.mH + 0.3 * torch.randn((4096, F), generator=g, device="cuda", dtype=torch.complex64)
    S = torch.view_as_real(s).contiguous()
    got = torch.view_as_complex(fq.fq_clutter_svd(S, k)["iq_f"].double())
    s64 = torch.view_as_complex(S.double())
    lam, vec = torch.linalg.eigh(s64.mH @ s64)
    lam, vec = lam.flip(0), vec.flip(1)[:, :k]
    want = s64 - (s64 @ vec) @ vec.mH
    turn = (2 * F * 2.0 ** -24 + 2.0 ** -22) * float(lam[0] / (lam[k - 1] - lam[k])) if k else 0.0
    assert float((got - want).norm()) <= (turn + (F + 8) * 2.0 ** -24) * float(s64.norm())


# matrices of a few large eigenvalues over many near the rounding of the largest
# (slowly turning clutter, blood, noise 46 dB below), all vectors: converges,
# and the eigenvalues are within 2 F 2^-24 of the largest
@pytest.mark.parametrize("F", [100, 160, 220, 300])
def test_all_eigenvectors_of_clutter(F):
    t = torch.arange(F, device="cuda", dtype=torch.float32)[None]
    for seed in range(8):
        g = torch.Generator(device="cuda").manual_seed(seed)

        def randn(*n):
            return torch.randn(n, generator=g, device="cuda", dtype=torch.complex64)

        s = 0.05 * randn(4096, F)
        for j, (lev, w) in enumerate(((10.0, 0.004), (5.0, 0.09), (2.0, -0.17))):
            s = s + lev * randn(4096, 1) * torch.polar(1.0 + 0.05 * torch.sin(0.03 * (j + 1) * t),
                                                       w * t + 0.4 * torch.sin(0.02 * (j + 1) * t))
        shift = 0.3 + 1.2 * torch.rand((4096, 1), generator=g, device="cuda")
        s = s + randn(4096, 1) * torch.polar(torch.ones_like(shift * t), shift * t)
        G = torch.view_as_real((s.to(torch.complex128).mH @ s.to(torch.complex128)).to(torch.complex64)).contiguous()
        lam, V, ws = fq.fq_hermitian_eig(G)
        fq.fq_clutter_status(ws)
        G64 = torch.view_as_complex(G.double())
        want = torch.linalg.eigvalsh(torch.tril(G64) + torch.tril(G64, -1).mH).flip(0)
        assert float((lam - want).abs().max()) <= (2 * F * 2.0 ** -24 + 2.0 ** -22) * float(want[0]), seed
        o = fq.fq_clutter_svd(torch.view_as_real(s).contiguous(), 50, want_iq_f=False)
        fq.fq_clutter_status(o["ws"])


# the Gram matrix of orthogonal frames is diagonal, exactly: its eigenvalues, over
# nine decades, to the last bits of binary32
@pytest.mark.parametrize("F", [2, 10, 40, 100, 200, 260])
def test_eigenvalues_of_graded_frames(F):
    a = torch.tensor([10.0 ** (-4.5 * i / (F - 1)) for i in range(F)], device="cuda")
    S = torch.zeros((F, F, 2), device="cuda")
    S[torch.arange(F), torch.arange(F).flip(0), 0] = a
    lam = fq.fq_clutter_svd(S, 1)["eigvals"]
    want = (a * a).double()
    assert float(((lam - want).abs() / want).max()) <= 4 * 2.0 ** -24


def test_weight_gradient_sums_over_many_voxels():
    """Weight gradients of the last two layers over 2^20 voxels against 64 bits
    on the same BF16 operands: a running sum of n = V / (152 x 32) rounded
    additions per CTA, so sqrt(n) 2^-24 of them and a few for the products and
    the sum of the CTAs."""
    n, F, Z, X = 1, 64, 128, 128
    V = n * F * Z * X
    g = torch.Generator(device="cuda").manual_seed(4)
    rng = np.random.default_rng(4)
    net = fq.CNN(4)
    net.set_weights([(rng.standard_normal((45, a, b)) * np.sqrt(2.0 / (45 * a)), 0.05 * rng.standard_normal(b))
                     for a, b in ((2, 32), (32, 32), (32, 32), (32, 2))])
    x = torch.zeros((n, F, Z, X, 32), dtype=torch.bfloat16, device="cuda")
    x[..., :2] = torch.randn((n, F, Z, X, 2), generator=g, device="cuda").bfloat16()
    tgt = torch.randn((n, F, Z, X, 2), generator=g, device="cuda")
    acts = fq.fq_cnn_forward(net, x)
    y = fq.cnn_output(acts, n, F, Z, X)
    dy3 = torch.zeros_like(x)
    dy3[..., :2] = (2.0 * (y[..., :2] - tgt) * (1.0 / (2 * V))).bfloat16()
    hid = [fq.cnn_hidden(acts, k, n, F, Z, X).clone() for k in (1, 2)]
    dy2 = torch.empty_like(x)
    fq.fq_cnn_conv(fq.CNN_MODE_MASK, dy3, net, 3, 1, dy2, mask=hid[1])
    grads, _ = fq.fq_cnn_backward(net, x, tgt, acts)
    torch.cuda.synchronize()
    assert int(net.status.item()) == 0
    for layer, a, d in ((3, hid[1], dy3), (2, hid[0], dy2)):
        o = fq.lib().fq_cnn_param_offset(0, layer) // 4
        gw = grads[o:o + 45 * 1024].view(45, 32, 32).double()
        pad = torch.nn.functional.pad(a[0].double(), (0, 0, 1, 1, 1, 1, 2, 2))
        num = den = 0.0
        for t in (0, 13, 22, 44):
            dt, dz, dx = t // 9, t // 3 % 3, t % 3
            want = pad[dt:dt + F, dz:dz + Z, dx:dx + X].reshape(-1, 32).T @ d[0].double().reshape(-1, 32)
            num += float(((gw[t] - want) ** 2).sum())
            den += float((want ** 2).sum())
        assert (num / den) ** 0.5 <= ((V / (152 * 32)) ** 0.5 + 4) * 2.0 ** -24, layer


# panels of 16 and 8 pixels at their limit (272 frames) and the most frames, even
# and odd counts, whole panels and remainders, rows of whole and of half 16-byte
# units; the bar of test_gram_panels
@pytest.mark.parametrize("F", [271, 272, 273, 300, 385, 511, 512])
@pytest.mark.parametrize("P", [1, 7, 8, 33, 1001])
@pytest.mark.parametrize("dt,shift", [("f32", 0), ("f32", 2), ("bf16", 0), ("bf16", 4)])
def test_gram_wide_panels(F, P, dt, shift):
    g = torch.Generator(device="cuda").manual_seed(F * 1000 + P)
    buf = torch.randn(2 * P * F + shift, generator=g, device="cuda").to(torch.float32 if dt == "f32" else torch.bfloat16)
    S = buf[shift:].view(P, F, 2)
    G = torch.view_as_complex(fq.fq_casorati_gram(S).double().contiguous())
    s = torch.view_as_complex(S.double().contiguous())
    mag = (S.double().abs().sum(2)).mT @ S.double().abs().sum(2)
    err = (G - s.mH @ s).abs()
    assert bool((err <= 2.0 ** -24 * (2 * P + 16) * mag).all())


def test_graph_of_small_and_large_eigen_problems():
    """As above by a replayed graph, with more members: the two kinds run in
    launches that overlap, and the stages after them see both."""
    ms = [w for i, F in enumerate((230, 60, 222, 200, 41, 256, 100, 225, 220, 221))
          for w in W.config4(seed=120 + i, n=1, s_range=(300, 800), f_range=(F, F), grids=((16, 1, 24),))]
    b = fq.Batch(ms)
    b.capture()
    for _ in range(3):
        b.graph_launch()
    b.status()
    torch.cuda.synchronize()
    for i, w in enumerate(ms):
        pl = Pipeline(w)
        pl.upload()
        pl.step()
        torch.cuda.synchronize()
        assert torch.equal(b.eigvals[i], pl.eigvals), i
        assert torch.equal(b.pd[i], pl.pd), i


@pytest.mark.parametrize("dt", ["f32", "bf16"])
def test_rf_echoes_near_the_record_end(dt):
    """Echoes wholly inside the record within 3 pitches of its end, where the
    kernel takes per-tap bounds, are the same bits as in the middle of a longer
    record (the correction of the taps' mean error, 2.6e-7 of an echo's
    amplitude, among them: it adds up over the echoes)."""
    rng = np.random.default_rng(11)
    S, t = 4000, torch.float32 if dt == "f32" else torch.bfloat16
    z = rng.uniform(282.0, 293.0, S) * 1540.0 / 62.5e6 / 2
    pos = np.stack([rng.uniform(-0.3e-3, 0.3e-3, S), np.zeros(S), z]).astype(np.float32)
    amp = torch.from_numpy(rng.uniform(0.5e-3, 1.5e-3, S).astype(np.float32)).cuda()
    out = []
    for ns in (300, 400):
        p = W.Probe(8, 1, 0.1e-3, 0.1e-3, 0.1e-3, 0.1e-3, 15.6e6, 62.5e6, 1540.0, 0.5, 2, ns)
        out.append(fq.fq_simulate_rf(p, [0.0], [0.0], torch.from_numpy(pos[None]).cuda(), amp, 1, out_dtype=t)[..., :300])
    assert float(out[0].float().abs().max()) > 0
    assert torch.equal(out[0], out[1])


def test_weight_gradients_of_an_unaligned_volume():
    """The backward pass takes a volume at any element's address."""
    n, F, Z, X = 2, 5, 8, 32
    g = torch.Generator(device="cuda").manual_seed(9)
    net = fq.CNN(9, zero_last=False)
    buf = torch.zeros(n * F * Z * X * 32 + 1, dtype=torch.bfloat16, device="cuda")
    x = buf[1:].view(n, F, Z, X, 32)
    x[..., :2] = torch.randn((n, F, Z, X, 2), generator=g, device="cuda").bfloat16()
    tgt = torch.randn((n, F, Z, X, 2), generator=g, device="cuda")
    aligned = x.clone()
    acts = fq.fq_cnn_forward(net, aligned)
    want, loss = fq.fq_cnn_backward(net, aligned, tgt, acts)
    got, loss2 = fq.fq_cnn_backward(net, x, tgt, acts)
    assert torch.equal(got, want) and torch.equal(loss, loss2)


def test_overlapping_eigen_launches_see_new_inputs():
    """The launch that starts beside the large matrices' reads this launch's
    Gram matrices, not what the caches hold of the last one's: a plan launched
    again on other amplitudes gives what a fresh plan gives."""
    ms = [w for i, F in enumerate((230, 60, 240, 200, 41))
          for w in W.config4(seed=140 + i, n=1, s_range=(300, 800), f_range=(F, F), grids=((16, 1, 24),))]
    b = fq.Batch(ms)
    b.capture()
    amps = [w.amp.copy() for w in ms]
    rng = np.random.default_rng(2)
    for _ in range(3):
        for w, a, d in zip(ms, amps, b.inputs):
            w.amp = (a * rng.uniform(0.5, 2.0, a.shape)).astype(np.float32)
            d[3].copy_(torch.from_numpy(w.amp))
        b.graph_launch()
        b.status()
        c = fq.Batch(ms)
        c.launch()
        c.status()
        torch.cuda.synchronize()
        for i in range(len(ms)):
            assert torch.equal(b.eigvals[i], c.eigvals[i]) and torch.equal(b.pd[i], c.pd[i]), i

"""The float-float trajectories at the edges of their dispatch: block frame
groups and their remainders, many wraps along lines and arcs in both flow
directions, elastic motion with drift, and the FP64 kernel that rotations
keep, against the oracle.  Bar: both sides round a position of ~48 or 53
bits once to binary32, so a result may differ by one ulp where the value is
within the float pair's error (~2^-22 ulp) of a rounding tie: at most 0.1%
of them."""
import numpy as np
import pytest
import torch

import oracle
from paper_2509_05464_gb300 import build as fqbuild
from paper_2509_05464_gb300 import fq
from paper_2509_05464_gb300 import workload as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    fqbuild.build()
    fq.lib()


def motion(kind):
    m = W.Motion(amp=[100e-6, 300e-6], freq=[1.2, 0.25], phase=[0.1, 0.5], dir=[(0.0, 0.0, 1.0), (0.6, 0.0, 0.8)])
    if kind == "elastic":
        m.elastic_grad, m.elastic_center, m.vel = (5.0, -3.0, 20.0), (1e-3, 0.0, 12e-3), (1e-3, -2e-3, 5e-4)
    if kind == "rotation":
        m.omega, m.rot_center = (0.1, 0.2, -0.3), (0.0, 0.0, 10e-3)
    return m


@pytest.mark.parametrize("medium,kind", [("tree", "rigid"), ("tree", "elastic"), ("arcs", "rigid"),
                                         ("arcs", "elastic"), ("arcs", "rotation")])
@pytest.mark.parametrize("S,F,dt,sign", [(2000, 1, 1e-3, 1), (2000, 17, 0.11, 1), (60_000, 100, 0.013, -1),
                                         (257, 33, 1.7, -1)])
def test_trajectories(medium, kind, S, F, dt, sign):
    w = W.config3(seed=5, n_scat=S, n_frames=F) if medium == "tree" else W.config2(seed=5, n_scat=S, n_frames=F)
    for s in w.segments:
        s.vmax *= sign
    m = motion(kind)
    t0 = 0.37
    d = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (w.p0, w.seg, w.flow)]
    pos = fq.fq_advect_scatterers(*d, w.segments, m, t0, dt, F).cpu().numpy()
    st, mt = W.segment_table(w), W.motion_table(m)
    same = 0
    frames = sorted({0, F - 1, F // 2, min(15, F - 1), min(16, F - 1)})
    for f in frames:
        want = oracle.advect(w.p0, w.seg, w.flow, st, mt, t0 + f * dt)
        ulp = np.spacing(np.abs(want).astype(np.float32))
        diff = np.abs(pos[f].astype(np.float64) - want.astype(np.float64))
        assert np.all(diff <= ulp), (f, float((diff / ulp).max()))
        same += np.mean(diff == 0) / len(frames)
    assert same > 0.999


@pytest.mark.parametrize("medium", ["tree", "arcs"])
@pytest.mark.parametrize("t0", [1e3, 1e5, 1e6, 1e7])
def test_trajectories_after_many_wraps(medium, t0):
    """10^4 to 10^8 wraps: the path coordinate of IEEE double, the bars above."""
    F, dt = 5, 1e-3
    w = W.config3(seed=6, n_scat=20_000, n_frames=F) if medium == "tree" else W.config2(seed=6, n_scat=20_000, n_frames=F)
    m = motion("rigid")
    d = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (w.p0, w.seg, w.flow)]
    pos = fq.fq_advect_scatterers(*d, w.segments, m, t0, dt, F).cpu().numpy()
    st, mt = W.segment_table(w), W.motion_table(m)
    blood = w.seg >= 0
    same = 0
    for f in range(F):
        want = oracle.advect(w.p0, w.seg, w.flow, st, mt, t0 + f * dt)
        ulp = np.spacing(np.abs(want).astype(np.float32))
        diff = np.abs(pos[f].astype(np.float64) - want.astype(np.float64))
        assert np.all(diff <= ulp), (f, float((diff / ulp).max()))
        same += np.mean(diff[:, blood] == 0) / F
    assert same > 0.999

"""The double-precision step (KF_FP64) where its own arithmetic can go wrong,
against the FP64 oracle: azimuths of many turns (the table's sin and cos, and
the library's from 64 rad on) and at +-pi (the wrap), curvatures from none to
strong (the series and the quotient forms, the straight line), zero
covariance entries (conversions by shifts).

Tolerance, element by element: half an FP32 ulp for the rounding of the
result, and 1e-10 of the element's scale (1 for parameters, sqrt(C_ii C_jj) for
covariances) for the double arithmetic of both sides, 1e-16 times a condition
of up to 1e6.  The oracle is given the field as FP32, which the call takes."""
import numpy as np
import pytest
import torch

import oracle
from paper_2401_14221_gb300 import build as kbuild
from paper_2401_14221_gb300 import kf
from paper_2401_14221_gb300 import workload as W

pytestmark = pytest.mark.gpu
HALF_ULP, DOUBLE = 2.0 ** -24 * 1.001, 1e-10


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    kbuild.build()
    yield
    kf.kf_set_step_kernel(kf.KF_STEP_AUTO)


def edge_workload(kind, bz):
    w = W.make_p2z(4099, seed=21) if kind == kf.KF_P2Z else W.make_p2r(1, 4099, seed=21)
    rng = np.random.default_rng(22)
    turns = rng.integers(-16, 17, w.n)  # up to 100 rad
    w.state[4] += (2 * np.pi * turns).astype(np.float32)
    w.state[4, :400] = np.float32(np.pi) * np.where(rng.random(400) < 0.5, 1, -1)
    w.state[4, 100:400] += rng.uniform(-2e-6, 2e-6, 300).astype(np.float32)
    w.state[3, 200:1200] = 10.0 ** rng.uniform(-13, 0.3, 1000)
    w.cov[np.array([1, 3, 6, 10]), 1200:1600] = 0.0  # no correlation with x
    w.bz = bz
    return w


@pytest.mark.parametrize("kernel", [kf.KF_STEP_DIRECT, kf.KF_STEP_STAGED], ids=["direct", "staged"])
@pytest.mark.parametrize("bz", [3.8, 0.0, -3.8])
@pytest.mark.parametrize("kind", [kf.KF_P2Z, kf.KF_P2R], ids=["p2z", "p2r"])
def test_fp64_step_at_its_edges(kind, bz, kernel):
    w = edge_workload(kind, bz)
    kf.kf_set_step_kernel(kernel)
    b = kf.upload(w, kf.KF_AOSOA, 32, "cuda:0")
    b.run(kf.KF_FP64)
    torch.cuda.synchronize()
    st, cv, stat = b.download()
    o_st, o_cv, o_stat, _ = oracle.step_batch(w.kind, w.state.T, w.cov.T, w.charge, w.hit.T,
                                              w.hitcov.T, w.surf, float(np.float32(w.bz)))
    assert np.array_equal(stat, o_stat)
    d = np.abs(st.T - o_st)
    d[:, 4] = np.minimum(d[:, 4], np.abs(d[:, 4] - 2 * np.pi))  # +-pi is one azimuth
    assert np.all(d <= HALF_ULP * np.abs(o_st) + DOUBLE), d.max(axis=0)
    diag = np.sqrt(o_cv[:, [0, 2, 5, 9, 14, 20]])
    scale = np.stack([diag[:, i] * diag[:, j] for i in range(6) for j in range(i + 1)], axis=1)
    d = np.abs(cv.T - o_cv)
    assert np.all(d <= HALF_ULP * np.abs(o_cv) + DOUBLE * scale), d.max(axis=0)

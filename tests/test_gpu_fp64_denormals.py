"""Covariances in FP32's denormal range under the double-arithmetic variants.

A double holds every denormal float exactly, so KF_FP64 has to take them as
they are and return the rounded double, denormal or not, on every path: one
thread per track, the staged kernel, arrays in host memory, the chain, the
second pass of KF_ADAPTIVE.  Tolerance against the FP64 oracle, element by
element: half an ulp of the result (a denormal's ulp is 2^-149) and 1e-10 of
its scale for the double arithmetic of both sides.

KF_FP64_UPDATE transports in FP32 and updates in double.  Its single step keeps
denormals in both: every kernel gives the same bits, and the variances of k and
theta, which the transport hands on as they are and hits this much wider change
by less than one part in 2^60, come back within half an ulp."""
import numpy as np
import pytest
import torch

import oracle
from paper_2401_14221_gb300 import build as kbuild
from paper_2401_14221_gb300 import kf
from paper_2401_14221_gb300 import workload as W

pytestmark = pytest.mark.gpu
HALF_ULP, HALF_TINY, DOUBLE = 2.0 ** -24 * 1.001, 2.0 ** -150 * 1.001, 1e-10
VARIANCES = [0, 2, 5, 9, 14, 20]


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    kbuild.build()
    yield
    kf.kf_set_step_kernel(kf.KF_STEP_AUTO)
    kf.kf_set_host_path(kf.KF_HOST_AUTO)


def tiny_workload(kind):
    w = W.make_p2z(4099, seed=81) if kind == kf.KF_P2Z else W.make_p2r(1, 4099, seed=81)
    w.cov = (w.cov * 1e-35).astype(np.float32)
    assert np.mean((w.cov != 0) & (np.abs(w.cov) < 2.0 ** -126)) > 0.9
    return w


def expected(w):
    o_st, o_cv, o_stat, _ = oracle.step_batch(w.kind, w.state.T, w.cov.T, w.charge, w.hit.T,
                                              w.hitcov.T, w.surf, float(np.float32(w.bz)))
    return o_st, o_cv, o_stat


def check_fp64(got, w):
    st, cv, stat = got
    o_st, o_cv, o_stat = expected(w)
    assert np.array_equal(stat, o_stat)
    d = np.abs(st.T - o_st)
    d[:, 4] = np.minimum(d[:, 4], np.abs(d[:, 4] - 2 * np.pi))
    assert np.all(d <= HALF_ULP * np.abs(o_st) + DOUBLE), d.max(axis=0)
    diag = np.sqrt(o_cv[:, VARIANCES])
    scale = np.stack([diag[:, i] * diag[:, j] for i in range(6) for j in range(i + 1)], axis=1)
    d = np.abs(cv.T - o_cv)
    assert np.all(d <= HALF_ULP * np.abs(o_cv) + HALF_TINY + DOUBLE * scale), d.max(axis=0)


def run_step(w, path, precision):
    kf.kf_set_step_kernel(kf.KF_STEP_STAGED if path == "staged" else
                          kf.KF_STEP_DIRECT if path == "direct" else kf.KF_STEP_AUTO)
    kf.kf_set_host_path(kf.KF_HOST_DIRECT)
    if path == "host":
        b = kf.host_upload(w, kf.KF_AOSOA, 32, "cuda:0")
    elif path == "soa":
        b = kf.upload(w, kf.KF_SOA, 0, "cuda:0")
    else:
        b = kf.upload(w, kf.KF_AOSOA, 32, "cuda:0")
    b.run(precision)
    torch.cuda.synchronize()
    return b.download()


PATHS = ["auto", "direct", "staged", "soa", "host"]
KINDS = pytest.mark.parametrize("kind", [kf.KF_P2Z, kf.KF_P2R], ids=["p2z", "p2r"])


@pytest.mark.parametrize("path", PATHS)
@KINDS
def test_fp64_step(kind, path):
    w = tiny_workload(kind)
    check_fp64(run_step(w, path, kf.KF_FP64), w)


@KINDS
def test_adaptive_second_pass(kind):
    w = tiny_workload(kind)
    w.state[3] = -w.state[3]  # 1/pT <= 0 marks every track
    check_fp64(run_step(w, "auto", kf.KF_ADAPTIVE), w)


@pytest.mark.parametrize("precision", [kf.KF_FP64, kf.KF_ADAPTIVE], ids=["fp64", "adaptive"])
@KINDS
def test_chain(kind, precision):
    w = tiny_workload(kind)
    if precision == kf.KF_ADAPTIVE:
        w.state[3] = -w.state[3]
    cw = W.ChainWorkload(n=w.n, bz=w.bz, kinds=np.array([kind]), pos=np.array([w.surf]),
                         event_sizes=np.array([w.n]), state=w.state, cov=w.cov, charge=w.charge,
                         hit=w.hit[None], hitcov=w.hitcov[None], truth_pool_layers=None,
                         truth_index=None)
    dc = kf.chain_upload(cw, kf.KF_SOA, 0, "cuda:0")
    dc.run(precision)
    torch.cuda.synchronize()
    check_fp64(dc.download(), w)


@KINDS
def test_fp64_update_step(kind):
    w = tiny_workload(kind)
    _, o_cv, o_stat = expected(w)
    ref = run_step(w, "staged", kf.KF_FP64_UPDATE)
    for path in PATHS:
        for got, want in zip(run_step(w, path, kf.KF_FP64_UPDATE), ref):
            assert np.array_equal(got, want), path
    hit = (o_stat & oracle.NO_INTERSECT) == 0
    for e in (9, 20):
        o, got = o_cv[hit, e], ref[1][e, hit]
        assert np.all(np.abs(got - o) <= HALF_ULP * o + HALF_TINY)

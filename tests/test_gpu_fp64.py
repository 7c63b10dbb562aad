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


# ------------------------------------------------------------ four warps to 32
# tracks (small FP64 chains, the redo of marked tracks): the arithmetic is the
# thread-per-track kernel's, so the results are equal bit for bit.

def chain_on(cw, n, layout, width, precision):
    sub = W.ChainWorkload(n=n, bz=cw.bz, kinds=cw.kinds, pos=cw.pos, event_sizes=np.array([n]),
                          state=cw.state[:, :n], cov=cw.cov[:, :n], charge=cw.charge[:n],
                          hit=cw.hit[:, :, :n], hitcov=cw.hitcov[:, :, :n],
                          truth_pool_layers=cw.truth_pool_layers,
                          truth_index=cw.truth_index[:n])
    dc = kf.chain_upload(sub, layout, width, "cuda:0")
    dc.run(precision)
    torch.cuda.synchronize()
    return dc.download()


@pytest.fixture(scope="module")
def big_chain():
    """One track more than the sharing kernel takes, and its thread-per-track
    FP64 result."""
    n = 96 * torch.cuda.get_device_properties(0).multi_processor_count + 1
    cw = W.make_chain(events=1, seed=31, sizes=np.array([n]), pool=4096)
    cw.hitcov[0] *= 1e-6  # every hit of the first layer shrinks the variance: all marked
    return cw, chain_on(cw, n, kf.KF_SOA, 0, kf.KF_FP64)


@pytest.mark.parametrize("layout,width", [(kf.KF_SOA, 0), (kf.KF_AOSOA, 32)], ids=["soa", "aosoa"])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 4865, -1], ids=str)
def test_shared_fp64_chain_equals_thread_per_track(big_chain, n, layout, width):
    cw, ref = big_chain
    n = cw.n - 1 if n < 0 else n
    for got, want in zip(chain_on(cw, n, layout, width, kf.KF_FP64), ref):
        assert np.array_equal(got, want[..., :n])


@pytest.mark.parametrize("redo", [kf.KF_CHAIN_REDO_LIST, kf.KF_CHAIN_REDO_SPAN], ids=["list", "span"])
@pytest.mark.parametrize("n", [1, 33, 64, 65, 3000, 0], ids=str)
def test_redo_of_every_track_equals_fp64(big_chain, n, redo):
    cw, ref = big_chain
    n = n or cw.n
    kf.kf_set_chain_redo(redo)
    try:
        got = chain_on(cw, n, kf.KF_AOSOA, 32, kf.KF_ADAPTIVE)
    finally:
        kf.kf_set_chain_redo(kf.KF_CHAIN_REDO_LIST)
    for g, want in zip(got, ref):
        assert np.array_equal(g, want[..., :n])


@pytest.mark.parametrize("sizes", [[5], [64, 1, 65], [1025, 700]], ids=str)
def test_server_redo_of_every_track_equals_fp64(big_chain, sizes):
    cw, ref = big_chain
    arena = torch.empty(64 << 20, dtype=torch.uint8, device="cuda:0")
    srv = kf.Server(cw.bz, cw.kinds, cw.pos, arena, precision=kf.KF_ADAPTIVE)
    try:
        srv.pause()  # one batch of all events
        jobs, lo = [], 0
        for n in sizes:
            pin = lambda a: torch.from_numpy(np.ascontiguousarray(a)).pin_memory()
            s = slice(lo, lo + n)
            out = (torch.empty((6, n), pin_memory=True), torch.empty((21, n), pin_memory=True),
                   torch.empty(n, dtype=torch.uint8, pin_memory=True))
            t = srv.submit(pin(cw.state[:, s]), pin(cw.cov[:, s]), pin(cw.charge[s]),
                           pin(cw.hit[:, :, s]), pin(cw.hitcov[:, :, s]), *out)
            jobs.append((t, s, out))
            lo += n
        srv.pause(False)
        for t, s, out in jobs:
            srv.wait(t, 60.0)
            for g, want in zip(out, ref):
                assert np.array_equal(g.numpy(), want[..., s])
    finally:
        srv.close()

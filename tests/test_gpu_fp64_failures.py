"""The double-precision chain's outcomes other than a clean update -- S not
positive definite, 1/pT <= 0, a surface not reached, non-finite input -- in its
two forms: the one-thread form returns early or runs on, the four-warp form
selects, so both must give the same bits, and the oracle's status."""
import numpy as np
import pytest
import torch

import oracle
from paper_2401_14221_gb300 import build as kbuild
from paper_2401_14221_gb300 import kf
from paper_2401_14221_gb300 import workload as W

pytestmark = pytest.mark.gpu
MARKED = 12  # tracks 0 .. MARKED-1 fail in ways that KF_ADAPTIVE leaves to the double chain


def select(cw, n):
    return W.ChainWorkload(n=n, bz=cw.bz, kinds=cw.kinds, pos=cw.pos, event_sizes=np.array([n]),
                           state=cw.state[:, :n], cov=cw.cov[:, :n], charge=cw.charge[:n],
                           hit=cw.hit[:, :, :n], hitcov=cw.hitcov[:, :, :n],
                           truth_pool_layers=cw.truth_pool_layers, truth_index=cw.truth_index[:n])


def run(cw, n, precision, layout=kf.KF_SOA, width=0):
    dc = kf.chain_upload(select(cw, n), layout, width, "cuda:0")
    dc.run(precision)
    torch.cuda.synchronize()
    return dc.download()


def same(got, want, tracks):
    for g, w in zip(got, want):
        assert np.array_equal(g[..., tracks], w[..., tracks], equal_nan=True)


@pytest.fixture(scope="module")
def failing():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    kbuild.build()
    n = 96 * torch.cuda.get_device_properties(0).multi_processor_count + 1
    cw = W.make_chain(events=1, seed=32, sizes=np.array([n]), pool=4096)
    cw.hitcov[0] *= 1e-6  # the first layer marks every track it reaches
    planes, cylinders = np.flatnonzero(cw.kinds == W.P2Z), np.flatnonzero(cw.kinds == W.P2R)
    bad = [planes[3], cylinders[4], planes[-1], cylinders[-1]]
    for t, l in enumerate(bad):  # negative hit variances: S not positive definite
        cw.hitcov[l][[0, 2, 5], t] = -1e3
    cw.hitcov[:, [0, 2, 5], 4] = -1e3                       # in every layer
    cw.hitcov[bad[0]][[0, 2], 5], cw.hitcov[bad[0]][1, 5] = 1e-4, 1.0  # det < 0
    cw.state[3, 6] = -cw.state[3, 6]
    cw.state[3, 7] = 0.0
    cw.hit[planes[2], :2, 8] += 3e4                          # a hit far off: k may turn negative
    cw.hit[cylinders[2], 2, 9] += 3e4
    cw.hitcov[bad[1]][:, 10] = 0.0                           # a hit without spread
    cw.hitcov[bad[0]][:, 11] = 0.0
    cw.state[5, 12] = np.float32(np.pi / 2)                  # parallel to the planes, and stays so
    cw.cov[:, 12] = 0.0
    cw.state[0, 13] = 500.0                                  # outside every cylinder
    cw.state[5, 14] = 0.0                                    # along the field
    cw.state[0, 15] = np.nan
    cw.state[3, 16] = np.inf
    cw.cov[:, 17] = np.nan
    cw.hit[:, :, 18] = 0.0                                   # no azimuth
    cw.cov[:, 19], cw.hitcov[:, :, 19] = 0.0, 0.0            # S = 0
    return cw, run(cw, n, kf.KF_FP64)


def test_status_of_failing_tracks(failing):
    cw, (_, _, stat) = failing
    n = 64
    _, _, o_stat = oracle.chain_batch(cw.kinds, cw.pos, cw.state[:, :n].T, cw.cov[:, :n].T,
                                      cw.charge[:n], cw.hit[:, :, :n].transpose(0, 2, 1),
                                      cw.hitcov[:, :, :n].transpose(0, 2, 1),
                                      float(np.float32(cw.bz)))
    tracks = np.r_[0:8, 12, 13, 20:n]  # without the ill-posed ones, whose sign rounding decides
    assert np.array_equal(stat[tracks], o_stat[tracks])
    assert all(stat[:5] & oracle.S_NOT_PD) and stat[6] & oracle.BAD_K
    assert stat[12] & oracle.NO_INTERSECT and stat[13] & oracle.NO_INTERSECT


@pytest.mark.parametrize("layout,width", [(kf.KF_SOA, 0), (kf.KF_AOSOA, 32)], ids=["soa", "aosoa"])
@pytest.mark.parametrize("n", [20, 33, -1], ids=str)
def test_shared_form_equals_thread_per_track(failing, n, layout, width):
    cw, ref = failing
    n = cw.n - 1 if n < 0 else n
    same(run(cw, n, kf.KF_FP64, layout, width), ref, slice(0, n))


@pytest.mark.parametrize("redo", [kf.KF_CHAIN_REDO_LIST, kf.KF_CHAIN_REDO_SPAN], ids=["list", "span"])
@pytest.mark.parametrize("n", [33, 5000], ids=str)
def test_second_pass_of_failing_tracks(failing, n, redo):
    cw, ref = failing
    kf.kf_set_chain_redo(redo)
    try:
        got = run(cw, n, kf.KF_ADAPTIVE)
    finally:
        kf.kf_set_chain_redo(kf.KF_CHAIN_REDO_LIST)
    same(got, ref, np.r_[0:MARKED, 20:n])


def test_server_second_pass_of_failing_tracks(failing):
    cw, ref = failing
    n = 33
    arena = torch.empty(8 << 20, dtype=torch.uint8, device="cuda:0")
    srv = kf.Server(cw.bz, cw.kinds, cw.pos, arena, precision=kf.KF_ADAPTIVE)
    pin = lambda a: torch.from_numpy(np.ascontiguousarray(a)).pin_memory()
    out = (torch.empty((6, n), pin_memory=True), torch.empty((21, n), pin_memory=True),
           torch.empty(n, dtype=torch.uint8, pin_memory=True))
    try:
        srv.wait(srv.submit(pin(cw.state[:, :n]), pin(cw.cov[:, :n]), pin(cw.charge[:n]),
                            pin(cw.hit[:, :, :n]), pin(cw.hitcov[:, :, :n]), *out), 60.0)
    finally:
        srv.close()
    same([o.numpy() for o in out], ref, np.r_[0:MARKED, 20:n])


@pytest.mark.parametrize("kind", [kf.KF_P2Z, kf.KF_P2R], ids=["p2z", "p2r"])
def test_single_step_status_equals_the_oracle(failing, kind):
    w = W.make_p2z(64, seed=33) if kind == kf.KF_P2Z else W.make_p2r(1, 64, seed=33)
    w.hitcov[:, 0] = [-1e3, 0, -1e3, 0, 0, -1e3]
    w.hitcov[1, 1] = 1.0
    w.state[3, 2] = -w.state[3, 2]
    w.state[3, 3] = 0.0
    w.state[5, 4] = np.float32(np.pi / 2)
    w.state[0, 5] = 500.0
    w.cov[:, 6], w.hitcov[:, 6] = 0.0, 0.0
    b = kf.upload(w, kf.KF_SOA, 0, "cuda:0")
    b.run(kf.KF_FP64)
    torch.cuda.synchronize()
    st, cv, stat = b.download()
    o_st, o_cv, o_stat, _ = oracle.step_batch(w.kind, w.state.T, w.cov.T, w.charge, w.hit.T,
                                              w.hitcov.T, w.surf, float(np.float32(w.bz)))
    assert np.array_equal(stat, o_stat) and stat[0] & oracle.S_NOT_PD and stat[2] & oracle.BAD_K
    d = np.abs(st.T - o_st)
    d[:, 4] = np.minimum(d[:, 4], np.abs(d[:, 4] - 2 * np.pi))
    assert np.all(d <= 2.0 ** -24 * 1.001 * np.abs(o_st) + 1e-10)

"""Batches of KF_ADAPTIVE events side by side on the server's compute streams
(the next batch starts when the previous one's first pass is done).  Every
event's result must equal, bit for bit, that of the event alone through
kf_kalman_chain, in an arena small enough that freed space is used again while
other batches' second passes run.  Every third event has its first layer's hits
so precise that all its tracks go through the second pass."""
import threading

import numpy as np
import pytest
import torch

from paper_2401_14221_gb300 import build as kbuild
from paper_2401_14221_gb300 import kf
from paper_2401_14221_gb300 import workload as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def events():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    kbuild.build()
    rng = np.random.default_rng(15)
    sizes = np.concatenate([[1, 33, 6000, 64, 1025],
                            W.lognormal_event_sizes(rng, 55, median=800.0, lo=50, hi=6000)])
    cw = W.make_chain(events=len(sizes), seed=52, sizes=sizes, pool=20000)
    ends = np.cumsum(sizes)
    slices = [slice(int(hi - n), int(hi)) for hi, n in zip(ends, sizes)]
    for s in slices[::3]:
        cw.hitcov[0][:, s] *= 1e-6
    refs = []
    for s in slices:
        n = s.stop - s.start
        sub = W.ChainWorkload(n=n, bz=cw.bz, kinds=cw.kinds, pos=cw.pos, event_sizes=np.array([n]),
                              state=cw.state[:, s], cov=cw.cov[:, s], charge=cw.charge[s],
                              hit=cw.hit[:, :, s], hitcov=cw.hitcov[:, :, s],
                              truth_pool_layers=cw.truth_pool_layers, truth_index=cw.truth_index[s])
        dc = kf.chain_upload(sub, kf.KF_SOA, 0, "cuda:0")
        dc.run(kf.KF_ADAPTIVE)
        refs.append(dc.download())
    return cw, slices, refs


@pytest.mark.parametrize("mode", ["copy", "direct", "mixed"])
def test_overlapping_adaptive_batches_equal_the_events_alone(events, mode):
    cw, slices, refs = events
    pin = lambda a: torch.from_numpy(np.ascontiguousarray(a)).pin_memory()
    ins = [(pin(cw.state[:, s]), pin(cw.cov[:, s]), pin(cw.charge[s]), pin(cw.hit[:, :, s]),
            pin(cw.hitcov[:, :, s])) for s in slices]
    outs = [(torch.empty(x[0].shape, pin_memory=True), torch.empty(x[1].shape, pin_memory=True),
             torch.empty(x[2].shape, dtype=torch.uint8, pin_memory=True)) for x in ins]
    biggest = max(kf.kf_server_event_bytes(s.stop - s.start, cw.L) for s in slices)
    arena = torch.empty(3 * biggest, dtype=torch.uint8, device="cuda:0")
    srv = kf.Server(cw.bz, cw.kinds, cw.pos, arena, precision=kf.KF_ADAPTIVE)
    lock = threading.Lock()
    tickets = [None] * len(slices)

    def submit(k):
        for e in range(k, len(slices), 2):
            copied = mode == "copy" or (mode == "mixed" and e % 2)
            with lock:  # the host-path mode is process-wide
                kf.kf_set_host_path(kf.KF_HOST_COPY if copied else kf.KF_HOST_DIRECT)
                tickets[e] = srv.submit(*ins[e], *outs[e])

    try:
        for _ in range(3):  # lanes and arena space of an earlier burst again
            for o in outs:
                for t in o:
                    t.fill_(77)
            threads = [threading.Thread(target=submit, args=(k,)) for k in (0, 1)]
            for t in threads:
                t.start()
            for t in threads:
                t.join()
            for t in tickets:
                srv.wait(t, 60.0)
            for o, ref in zip(outs, refs):
                for got, want in zip(o, ref):
                    assert np.array_equal(got.numpy(), want)
        assert srv.stats()["batches"] > 3 * 4  # more than one batch to a lane each time
    finally:
        kf.kf_set_host_path(kf.KF_HOST_AUTO)
        srv.close()

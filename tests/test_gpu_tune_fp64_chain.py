"""The tuner and a KF_FP64 chain small enough for four warps to 32 tracks: that
form has one shape, so the tuner reports it and stores no entry that a larger
batch of the same bucket, one thread per track, would take; beyond the line the
candidates are timed and stored as for the other variants."""
import numpy as np
import pytest
import torch

from paper_2401_14221_gb300 import build as kbuild
from paper_2401_14221_gb300 import kf
from paper_2401_14221_gb300 import workload as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("past", [0, 1], ids=["shared", "thread per track"])
def test_chain_autotune_fp64(past):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    kbuild.build()
    kf.autotune_clear()
    n = 96 * torch.cuda.get_device_properties(0).multi_processor_count + past
    cw = W.make_chain(events=1, seed=64, sizes=np.array([n]), pool=2048)
    dc = kf.chain_upload(cw, kf.KF_AOSOA, 32, "cuda:0")
    dc.run(kf.KF_FP64)
    plain = dc.download()
    dc.reset()
    try:
        t = kf.autotune_chain(dc, kf.KF_FP64)
        assert t["ms"] > 0 and t["step_kernel"] == "direct"
        entries = kf.autotune_export().splitlines()
        if past:
            assert t["threads"] in (64, 128, 256) and len(entries) == 1
        else:
            assert t["threads"] == 128 and entries == []
        dc.run(kf.KF_FP64)
        for got, want in zip(dc.download(), plain):
            assert np.array_equal(got, want)
    finally:
        kf.autotune_clear()

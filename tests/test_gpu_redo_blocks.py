"""KF_ADAPTIVE's second pass of a single step in its two block sizes, and with
the next kernel let in before and after its wait: a batch beyond the line
between the block sizes (three blocks to each of 152 SMs, 4,096 tracks a block;
192 blocks on the compressed store) must give, for its first AoSoA blocks, the
bits of batches of only those, below either line."""
import numpy as np
import pytest
import torch

from paper_2401_14221_gb300 import build as kbuild
from paper_2401_14221_gb300 import kf
from paper_2401_14221_gb300 import workload as W

pytestmark = pytest.mark.gpu
KINDS = pytest.mark.parametrize("kind", [kf.KF_P2Z, kf.KF_P2R], ids=["p2z", "p2r"])
SHARES = pytest.mark.parametrize("share", [0.001, 0.05], ids=["one round", "two rounds"])


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    kbuild.build()
    kf.autotune_clear()


def tiled(kind, n, share):
    """n tracks from 8,192 distinct ones, a share of them with hits so precise
    that they are marked: layout, arrays of the workload, common arguments."""
    w = W.make_p2z(8192, seed=91) if kind == kf.KF_P2Z else W.make_p2r(1, 8192, seed=91)
    rep = lambda a: np.tile(a, (1, n // w.n + 1))[:, :n]
    lay = kf.make_layout(kf.KF_AOSOA, 32, n)
    hitcov = rep(w.hitcov).copy()
    hitcov[:, np.random.default_rng(92).random(n) < share] *= 1e-6
    args = (torch.from_numpy(np.tile(w.charge, n // w.n + 1)[:n]).cuda(),
            kf.to_device(rep(w.hit), lay, "cuda"), kf.to_device(hitcov, lay, "cuda"),
            torch.tensor([w.surf], dtype=torch.float32, device="cuda"), 0)
    return w, rep, lay, args


def compare(call, ins, n, prefixes):
    def run(m):
        outs = [torch.zeros_like(t) for t in ins]
        status = torch.zeros(n, dtype=torch.uint8, device="cuda")
        for _ in range(3):  # steps in a row, each let in by the one before
            call(kf.make_layout(kf.KF_AOSOA, 32, m), outs, status)
        torch.cuda.synchronize()
        blocks = -(-n // 32)
        return [o[:o.numel() // blocks * (m // 32)].cpu() for o in outs] + [status[:m].cpu()]

    big = run(n)
    assert not (big[-1] & 0x80).any()
    for m in prefixes:
        for x, y in zip(run(m), big):
            assert torch.equal(x, y[:x.numel()]), m


@SHARES
@KINDS
def test_step(kind, share):
    n = 3 * 152 * 4096 + 33
    w, rep, lay, args = tiled(kind, n, share)
    ins = (kf.to_device(rep(w.state), lay, "cuda"), kf.to_device(rep(w.cov), lay, "cuda"))
    fn = kf.kf_p2z_propagate_update if kind == kf.KF_P2Z else kf.kf_p2r_propagate_update
    params = kf.make_params(w.bz, kf.KF_ADAPTIVE)
    compare(lambda lay, outs, status: fn(params, lay, *ins, *outs, *args, status), ins, n,
            (n - 33 - 4096, 1 << 17))


@SHARES
@KINDS
def test_compressed_step(kind, share):
    n = 192 * 4096 + 33
    w, rep, lay, args = tiled(kind, n, share)
    sig, rho = W.compress_cov(w.cov)
    ins = (kf.to_device(rep(w.state), lay, "cuda"), kf.to_device(rep(sig), lay, "cuda"),
           kf.to_device_rho(rep(rho), lay, "cuda"))
    params = kf.make_params(w.bz, kf.KF_ADAPTIVE)
    compare(lambda lay, outs, status: kf.kf_propagate_update_compressed(
        kind, params, lay, *ins, *outs, *args, status), ins, n, (n - 33 - 4096, 1 << 17))

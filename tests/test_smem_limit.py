"""Launches of one kernel with different amounts of dynamic shared memory, all
above the 48 KB that need a raised limit: bands of one call that were prepared
in another order than their sizes, and calls of several threads.  No launch may
lose the limit that it needs to another one's; results equal the plain call's,
bit for bit."""
import threading

import numpy as np
import pytest

from paper_2604_06602_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 118000


@pytest.fixture(scope="module")
def umi():
    from paper_2604_06602_gb300 import umi as u
    u.load(build_if_missing=True)
    return u


@pytest.fixture(scope="module")
def curve():
    return torch.from_numpy(synth.random_curve(77, N, nan_runs=3, run_len=(1, 4000))).cuda()


def batch(curve, windows):
    off = np.arange(len(windows) + 1, dtype=np.int64) * N
    return curve.repeat(len(windows)), off, np.array(windows, np.int32)


@pytest.mark.parametrize("call", ["batched", "noalloc", "segmented"])
def test_a_tuned_band_beside_a_longer_untuned_one(umi, tmp_path, curve, call):
    # (32,68,2) at 256 threads: 70,368 bytes at the tuned chain of 24, 71,392 at
    # the 56 that 32 untuned curves are fitted to.
    flux, off, W = batch(curve, [2161] * 8 + [2101] * 32)
    f = tmp_path / "t.txt"
    f.write_text("%s|2161|throughput|32|68|2|24|256\n" % torch.cuda.get_device_name())
    umi.clear_tuning()
    want = {w: umi.detrend(curve, w)[0] for w in (2161, 2101)}
    try:
        umi.load_tuning(str(f))
        if call == "segmented":
            tr = umi.detrend_segmented(flux, off, W, gap_min=N)[0]
        else:
            tr = {"batched": umi.detrend_batched, "noalloc": umi.detrend_batched_noalloc}[call](flux, off, W)[0]
        torch.cuda.synchronize()
    finally:
        umi.clear_tuning()
    for k, w in enumerate(W):
        assert torch.equal(tr[off[k]:off[k + 1]].view(torch.int32), want[int(w)].view(torch.int32)), k


def test_threads_with_batches_of_several_sizes(umi, curve):
    umi.clear_tuning()
    sizes = (10, 32, 64)                      # 70,624, 71,392 and 72,160 bytes
    want = umi.detrend_batched(*batch(curve, [2161] * 10))[0][:N].cpu().view(torch.int32)
    inputs = [batch(curve, [2161] * B) for B in sizes]
    hosts = [x.cpu().numpy() for x, _, _ in inputs]
    errors = []

    def work(k, host):
        try:
            x, off, W = inputs[k]
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                tr, de = torch.empty_like(x), torch.empty_like(x)
                for _ in range(4):
                    if host:
                        got = torch.from_numpy(umi.detrend_batched_host(hosts[k], off, W)[0])
                    else:
                        got = umi.detrend_segmented(x, off, W, gap_min=N, trend=tr, detr=de, stream=s)[0]
                        s.synchronize()
                    assert torch.equal(got[off[-2]:].cpu().view(torch.int32), want)
        except Exception as e:  # noqa: BLE001 - reported below
            errors.append((sizes[k], host, e))

    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=(k, host)) for k in range(len(sizes)) for host in (True, False)]
    for t in threads:
        t.start()
    for t in threads:
        t.join(120)
    assert not errors, errors

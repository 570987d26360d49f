"""Two host threads with a context and stream each, calling the library with different sizes at the same time:
every call succeeds and gives what it gives alone.  (Each kernel's limit of dynamic shared memory belongs
to the kernel, not to the launch that sets it.)"""
import threading

import numpy as np
import pytest

from test_gpu_parity import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


def _catalogue(torch, n=60):
    rng = np.random.default_rng(4)
    return [torch.tensor(a, device="cuda:0") for a in (rng.uniform(0, 6, (n, 2)), rng.normal(0, 0.3, (n, 2)), np.ones(n))]


def _records(torch, ext4pcf, est, nb, nmax):
    edges, cat = np.geomspace(0.3, 4.0, nb + 1), _catalogue(torch)
    rec = torch.zeros((8, ext4pcf.record_layout(nb, nmax)["rec"], 2), dtype=torch.float64, device="cuda:0")
    ext4pcf.ext4pcf_multipoles(est.ctx, *cat, 60, edges, nb, nmax, np.arange(8, dtype=np.int64), 8, rec)
    return rec


def _third(torch, ext4pcf, est, nb, nmax):
    edges, cat = np.geomspace(0.3, 4.0, nb + 1), _catalogue(torch)
    ups = torch.zeros((5, 2 * nmax + 1, nb, nb, 2), dtype=torch.float64, device="cuda:0")
    ext4pcf.ext4pcf_measure3(est.ctx, *cat, 60, edges, nb, nmax, ups)
    return ups


def _measure(torch, ext4pcf, est, nb, nmax):
    return est.measure(*_catalogue(torch), np.geomspace(0.3, 4.0, nb + 1), nmax)


def _map4(torch, ext4pcf, est, nb, n_ap):
    ups = torch.ones(est.ups_shape(nb, 2)[1:], dtype=torch.float64, device="cuda:0")
    return torch.tensor(est.to_map4(ups, np.geomspace(1.0, 9.0, nb + 1), 9, np.geomspace(1.0, 5.0, n_ap))[1])


@pytest.mark.parametrize("prec,call,sizes", [
    ("f16x3", _records, ((1, 0), (16, 20))), ("fp64", _records, ((1, 0), (16, 9))), ("fp32", _third, ((2, 1), (12, 3))),
    ("f16x3", _measure, ((3, 1), (12, 2))), ("3xtf32", _measure, ((3, 1), (9, 2))), ("fp32", _measure, ((2, 1), (16, 1))),
    ("f16x3", _map4, ((2, 1), (2, 64)))])
def test_calls_of_two_threads_do_not_disturb_each_other(torch_cuda, prec, call, sizes):  # noqa: F811
    from paper_2509_07974_gb300 import ext4pcf
    torch, errors, results = torch_cuda, [], {}
    start = threading.Barrier(2)

    def work(k):
        stream = torch.cuda.Stream()
        try:
            with torch.cuda.stream(stream):
                est = ext4pcf.Estimator(0, prec, stream=stream)
                alone = call(torch, ext4pcf, est, *sizes[k])
                stream.synchronize()
                start.wait(timeout=60)
                for _ in range(300):
                    got = call(torch, ext4pcf, est, *sizes[k])
                stream.synchronize()
                results[k] = torch.equal(alone, got)
                est.close()
        except Exception as e:  # noqa: BLE001  (reported by the test's thread)
            errors.append("%s: %s" % (sizes[k], e))
            start.abort()

    threads = [threading.Thread(target=work, args=(k,)) for k in (0, 1)]
    for t in threads:
        t.start()
    for t in threads:
        t.join(timeout=120)
    assert not errors and results == {0: True, 1: True}, (errors, results)

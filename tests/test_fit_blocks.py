"""The fit's row blocks: row counts around the block and merge sizes against numpy's
least squares, the rank check, and the same bits whatever the thread count."""
import os
import subprocess
import sys

import numpy as np
import pytest

from oracle import basis as obasis
from workloads import data

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    from paper_1906_02318_gb300 import build, mpmi
    build.build()
    return mpmi


# blocks of 256 rows, merged eight at a time
@pytest.mark.parametrize("kind,m", [("bot", 12), ("bot", 255), ("bot", 256), ("bot", 257),
                                    ("bot", 2049), ("car", 32), ("car", 257), ("car", 288),
                                    ("car", 2048), ("car", 2305), ("car", 16385)])
def test_fit_around_the_blocks(lib, kind, m):
    x, u, xn = data.transitions(kind, 17, m)
    K, res = lib.fit_operator(kind, x, u, xn)
    X, Y = obasis.lift(kind, x, u), obasis.lift(kind, xn, u)
    ref = np.linalg.lstsq(X, Y, rcond=None)[0].T
    # both solve to rounding times the conditioning (8e3 for the race car's features)
    assert np.max(np.abs(K - ref)) <= 1e-9 * np.max(np.abs(ref))
    want = np.linalg.norm(X @ K.T - Y) / np.linalg.norm(Y)
    assert abs(res - want) <= 1e-9 * want + 1e-13


def test_rank_deficient_data_is_refused_at_any_size(lib):
    for m in (40, 300, 5000):
        x, u, xn = data.transitions("car", 18, m)
        x[:, 3] = 0.0  # vx = 0: several features vanish
        with pytest.raises(lib.MpmiError) as e:
            lib.fit_operator("car", x, u, xn)
        assert e.value.code == -1


def test_same_bits_for_any_thread_count(lib):
    code = ("import sys; sys.path.insert(0, %r); import numpy as np;"
            "from paper_1906_02318_gb300 import mpmi; from workloads import data;"
            "K, r = mpmi.fit_operator('car', *data.transitions('car', 19, 9000));"
            "sys.stdout.write(K.tobytes().hex() + r.hex())" % ROOT)
    cpus = sorted(os.sched_getaffinity(0))
    out = [subprocess.run([sys.executable, "-c", code], capture_output=True, text=True,
                          timeout=300, check=True,
                          preexec_fn=lambda c=c: os.sched_setaffinity(0, c)).stdout
           for c in (cpus, cpus[:1])]
    assert out[0] == out[1]


def test_threads_stay_within_the_callers_cpus(lib):
    """A fit starts no more threads than the CPUs that the calling thread may run on, and
    gives the same bits."""
    import os
    import threading
    import time
    if not hasattr(os, "sched_setaffinity") or len(os.sched_getaffinity(0)) < 2:
        pytest.skip("needs two CPUs and an affinity call")
    x, u, xn = data.transitions("car", 4, 60000)
    want = lib.fit_operator("car", x, u, xn)
    out, go = [], threading.Event()

    def fit_on_one_cpu():
        os.sched_setaffinity(0, {min(os.sched_getaffinity(0))})  # this thread alone
        go.wait()
        for _ in range(5):
            out.append(lib.fit_operator("car", x, u, xn))

    t = threading.Thread(target=fit_on_one_cpu)
    t.start()
    time.sleep(0.05)
    before = most = len(os.listdir("/proc/self/task"))
    go.set()
    while t.is_alive():
        most = max(most, len(os.listdir("/proc/self/task")))
        time.sleep(0.001)
    t.join()
    assert most == before
    for K, res in out:
        assert np.array_equal(K, want[0]) and res == want[1]

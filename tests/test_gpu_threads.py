"""Host threads with a stream each, every one with its own systems and hierarchies: the
calls succeed and give the bits they give alone.  The setups meet kernels whose
shared memory differs from size to size."""
import threading

import numpy as np
import pytest

from paper_2311_13914_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SIZES = [(8, 7, 4), (13, 9, 5), (18, 11, 6), (23, 13, 7), (28, 15, 8), (33, 17, 9)]


@pytest.fixture(scope="module")
def B():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2311_13914_gb300 import _build, binding

    _build.build()
    return binding


def _in_threads(job, reps):
    """job(k) once alone and `reps` times in threads that start together."""
    alone = [job(k) for k in range(len(SIZES))]
    failures = []

    def work(k, gate):
        gate.wait()
        for _ in range(reps):
            try:
                got = job(k)
                if not all(np.array_equal(a, b) for a, b in zip(alone[k], got)):
                    failures.append(f"{k}: other bits")
            except Exception as e:  # noqa: BLE001
                failures.append(f"{k}: {e}")

    gate = threading.Barrier(len(SIZES))
    threads = [threading.Thread(target=work, args=(k, gate)) for k in range(len(SIZES))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failures, failures[:5]


def test_setups_in_threads(B):
    import torch

    streams = [torch.cuda.Stream() for _ in SIZES]

    def job(k):
        m = W.mesh(*SIZES[k])
        s = B.bd_assemble(m, W.DEFAULT_PARAMS, W.fibre_table(m), stream=streams[k])
        h = B.amg_setup(s, B.amg_options_default(precision=k & 1, coarse_eq_limit=100), stream=streams[k])
        out = [np.array([B.amg_level_info(h, l)["lam"] for l in range(B.amg_num_levels(h))])]
        out.append(B.amg_export_level(h, 1, stream=streams[k])["A"][2])
        h.close()
        s.close()
        return out

    _in_threads(job, 80)

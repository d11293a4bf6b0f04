"""Host threads with a context and a stream each: SVDs with left vectors of long
columns (200 KB of shared memory a CTA) beside ones of short columns.  A
kernel's shared-memory limit belongs to the process, so a limit set by the size
of each call would refuse the other thread's launches.
"""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import seeded_inputs as si  # noqa: E402


def test_svd_of_different_heights_in_threads():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1501_05504_gb300 import binding as b
    b.slib()
    rng = si.rng_for(950)
    mats = [rng.standard_normal((m, 1)) for m in (6000, 1700, 1800, 1900)]
    errors = []
    start = threading.Barrier(len(mats))

    def work(X):
        try:
            torch.cuda.set_device(0)
            ctx = b.dmrg3s_create(0, 1 << 26)
            with torch.cuda.stream(torch.cuda.Stream()):
                d = torch.from_numpy(X).cuda()
                start.wait()
                for k in range(2000):
                    u, s, vt = b.dmrg3s_svd(ctx, [d])[0]
                    if k % 200 == 0:
                        u, s, vt = u.cpu().numpy(), s.cpu().numpy(), vt.cpu().numpy()
                        assert np.abs((u * s) @ vt - X).max() <= 1e-13 * s[0]
                torch.cuda.current_stream().synchronize()
            ctx.close()
        except Exception as e:   # noqa: BLE001 (reported by the main thread)
            errors.append(repr(e))

    threads = [threading.Thread(target=work, args=(X,)) for X in mats]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors

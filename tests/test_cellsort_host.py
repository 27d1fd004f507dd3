"""The sort of a source cell's rays (csrc/cellsort.cuh) run by host threads as
a warp or a CTA: every length around powers of two and around the thread
counts, orders from sorted to reversed.  One build checks indexes
(AddressSanitizer), the other that no two threads touch an element between
barriers (ThreadSanitizer)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
LENGTHS = [0, 1, 2, 3, 4, 5, 7, 8, 9, 31, 32, 33, 34, 63, 64, 65, 100, 127, 129, 255, 257, 1000, 1023, 1024, 1025, 2500]


@pytest.mark.parametrize("sanitizer", ["address,undefined", "thread"])
@pytest.mark.parametrize("nt", [1, 5, 32, 64])
def test_cells_are_sorted(tmp_path, sanitizer, nt):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    exe = str(tmp_path / "cellsort_host")
    r = subprocess.run([gxx, "-std=c++20", "-O1", "-g", "-fsanitize=" + sanitizer, "-fno-sanitize-recover=all",
                        os.path.join(HERE, "fft_host", "cellsort_host.cpp"), "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-600:]
    rng = np.random.default_rng(nt)
    lists = []
    for n in LENGTHS if nt < 64 else LENGTHS[-8:]:
        v = rng.choice(10 * n + 1, n, replace=False)
        lists += [v, np.sort(v)[::-1]] + ([np.sort(v)] if n < 200 else [])
    data = b"".join(np.int32(len(v)).tobytes() + np.asarray(v, np.int32).tobytes() for v in lists)
    r = subprocess.run([exe, str(nt)], input=data, capture_output=True, timeout=600)
    if r.returncode != 0 and sanitizer == "thread" and b"data race" not in r.stderr:
        pytest.skip("ThreadSanitizer cannot run here: " + r.stderr.decode()[-300:])
    assert r.returncode == 0, r.stderr.decode()[-2000:]
    out = np.frombuffer(r.stdout, np.int32)
    np.testing.assert_array_equal(out, np.concatenate([np.sort(v) for v in lists]))

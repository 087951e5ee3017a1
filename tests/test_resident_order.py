"""The order of loads and stores of the resident kernel's strips, whatever order
its CTAs start and run in (no GPU needed)."""
import ctypes
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def flips(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = tmp_path_factory.mktemp("ro") / "libresident_order.so"
    subprocess.run([nvcc, "-shared", "-Xcompiler", "-fPIC", "-std=c++17", "-o", str(out),
                    os.path.join(HERE, "csrc", "resident_order.cu")], check=True)
    return ctypes.CDLL(str(out)).resident_flips


@pytest.mark.parametrize("gh", [1, 2, 4])
def test_no_strip_overwrites_rows_a_late_neighbour_has_yet_to_load(flips, gh):
    """A strip loads its rows and its neighbours' edge rows from the first
    buffer, posts its edge rows after every gh-th step but the last, waits there
    for its neighbours' rows, and stores its result.  One strip starts last: the
    others run until they wait for it."""
    for strips in (2, 3, 6):
        for n in range(1, 14):
            exchanges = [s for s in range(n) if s % gh == gh - 1 and s + 1 < n]
            for late in range(strips):
                posted = [0] * strips          # exchanges posted by each strip
                stored = set()
                progress = True
                while progress:
                    progress = False
                    for b in range(strips):
                        if b == late or b in stored:
                            continue
                        around = [posted[(b - 1) % strips], posted[(b + 1) % strips]]
                        if posted[b] < len(exchanges) and min(around + [posted[b]]) == posted[b]:
                            posted[b] += 1
                            progress = True
                        elif posted[b] == len(exchanges) and min(around) >= posted[b]:
                            stored.add(b)
                            progress = True
                if {(late - 1) % strips, (late + 1) % strips} & stored:
                    assert flips(n, gh), f"{n} steps: stored into the rows that strip {late} of {strips} still reads"
    assert all(flips(n, gh) == 1 for n in range(1, 40, 2))      # an odd count always ends in the other buffer

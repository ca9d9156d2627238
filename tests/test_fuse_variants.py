"""The fusion's variant numbers: every compiled bundle shape stays selectable, the autotuner
times only distinct kernels, and forgets its choices when the library is rebuilt.  No GPU."""
import json
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")
SIZES = [(320 * 240, 320 * 240), (640 * 360, 1280 * 720), (640 * 360 - 1, 1280 * 720), (1, 1), (97 * 33, 61 * 47),
         (24 * 18, 61 * 47)]


@pytest.fixture(scope="module")
def effective(tmp_path_factory):
    """{(variant, views, target pixels, view pixels): the variant whose kernel runs}, from the library's rule."""
    d = tmp_path_factory.mktemp("variants")
    (d / "a.cpp").write_text("""#include <cstdio>
#include "paper_2505_18932_gb300/csrc/gvs_internal.cuh"
int main() {
    long v, k, t, p;
    while (std::scanf("%ld %ld %ld %ld", &v, &k, &t, &p) == 4)
        std::printf("%d\\n", gvs::shaped_variant((int)v, (int)k, t, p));
}
""")
    cxx = shutil.which("g++") or "g++"
    subprocess.run([cxx, "-std=c++17", "-I", ROOT, "-I", os.path.join(CUDA, "include"), "-o", str(d / "a"),
                    str(d / "a.cpp")], check=True)
    keys = [(v, k, t, p) for v in range(7) for k in range(1, 33) for t, p in SIZES]
    out = subprocess.run([str(d / "a")], input="".join("%d %d %d %d\n" % q for q in keys), capture_output=True,
                         text=True, check=True).stdout.split()
    return dict(zip(keys, map(int, out)))


def test_every_bundle_shape_can_be_chosen(effective):
    """For 5 to 16 views, where all are compiled: the plain 8 x 4 and 4 x 8 bundles (0 and 3) at every size."""
    for k in range(5, 17):
        for t, p in SIZES:
            assert {0, 2, 3, 4, 5, 6} <= {effective[v, k, t, p] for v in range(7)}, (k, t, p)
            assert effective[3, k, t, p] == 3
    for k in list(range(1, 5)):  # one choice, whatever the number
        for t, p in SIZES:
            assert len({effective[v, k, t, p] for v in range(7)}) == 1


def test_candidates_are_distinct_kernels(effective):
    from paper_2505_18932_gb300 import autotune
    for k in range(1, 33):
        for t, p in SIZES:
            c = autotune.variants_for(k, t, p)
            e = [effective[v, k, t, p] for v in c]
            assert c[0] == 0 and len(set(e)) == len(e), (k, t, p, c, e)
            if 5 <= k <= 16:
                assert set(e) == {effective[v, k, t, p] for v in range(7)}


def test_choice_is_forgotten_with_the_library(tmp_path, monkeypatch):
    """A cached choice holds for the library it was timed with."""
    from paper_2505_18932_gb300 import autotune, gvs
    lib = tmp_path / "libgvs.so"
    lib.write_bytes(b"one build")
    monkeypatch.setattr(gvs, "LIB_PATH", str(lib))
    monkeypatch.setattr(autotune, "CACHE_PATH", str(tmp_path / "autotune.json"))
    monkeypatch.setattr(autotune, "device_key", lambda: "device")
    monkeypatch.setattr(autotune, "time_ms", lambda fn: fn())
    timed = []

    def choose(ms):
        def runner(v):
            timed.append(v)
            return lambda: ms[v]
        return autotune.choose({"views": 8}, runner, candidates=(0, 1, 2))[0]

    assert choose([3.0, 1.0, 2.0]) == 1 and timed == [0, 1, 2]
    assert choose([1.0, 3.0, 2.0]) == 1 and timed == [0, 1, 2]       # from the cache
    lib.write_bytes(b"another build")
    assert choose([3.0, 2.0, 1.0]) == 2 and timed == [0, 1, 2] * 2   # timed again
    assert len(json.load(open(autotune.CACHE_PATH))) == 2

"""Host logic: work items as mm_layout.cpp packs them with the values that the
library gives it -- the device's SMs, the items' fixed cost, a supplied order --
checked by tests/layout_budget_check.cpp (no GPU)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2005_06332_gb300 import netgen
from test_layout_paths import CSRC, ROOT


@pytest.fixture(scope="module")
def packed(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    inc = [os.path.join(c, "include") for c in (os.environ.get("CUDA_HOME"), "/usr/local/cuda")
           if c and os.path.exists(os.path.join(c, "include", "vector_types.h"))]
    if not inc:
        pytest.skip("CUDA headers not available")
    d = tmp_path_factory.mktemp("budget")
    out = str(d / "layout_budget_check")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I" + CSRC, "-I" + os.path.join(ROOT, "include"), "-I" + inc[0],
                    os.path.join(ROOT, "tests", "layout_budget_check.cpp"), os.path.join(CSRC, "mm_layout.cpp"), "-o", out],
                   check=True, capture_output=True)

    def run(sizes, p_branch=0.1, group_comps=0, sms=152, cost=None, fp64=False):
        rng = np.random.default_rng(5)
        with open(d / "net.bin", "wb") as f:
            np.array([len(sizes)], np.int32).tofile(f)
            np.array([sum(sizes)], np.int64).tofile(f)
            np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64).tofile(f)
            np.concatenate([netgen.random_tree(rng, n, p_branch) for n in sizes]).astype(np.int32).tofile(f)
            np.array([cost is not None], np.int32).tofile(f)
            np.asarray(cost if cost is not None else np.zeros(len(sizes)), np.float32).tofile(f)
        r = subprocess.run([out, str(d / "net.bin"), str(group_comps), str(sms), str(int(fp64))], capture_output=True, text=True)
        fields = dict(kv.split("=") for kv in r.stdout.split())
        assert r.returncode == 0 and fields["bad"] == "0", r.stdout
        giants = [int(v) for v in fields.pop("giants").split(",") if v]
        return {k: int(v) for k, v in fields.items()}, giants

    return run


def test_giants_that_get_clusters(packed):
    """In a supplied order with small giants ahead of the huge ones and between them, the huge ones come first, the others
    in their order; giants of under 0.6 of the largest, too many giants, smaller ones, or much else in the network: none."""
    sizes, cost = [12000, 100000, 11000, 100000, 9900, 40], [9.0, 8.0, 7.0, 6.0, 5.0, 4.0]
    f, giants = packed(sizes, cost=cost)
    assert f["huge"] == 2 and giants == [100000, 100000, 12000, 11000, 9900]
    assert packed([100000, 60001, 60000, 33000])[0]["huge"] == 2
    f, giants = packed([33000, 60000, 500000, 60001], cost=[4.0, 3.0, 2.0, 1.0])
    assert f["huge"] == 1 and giants == [500000, 33000, 60000, 60001]
    assert packed([100000] * 9)[0]["huge"] == 9 and packed([100000] * 10)[0]["huge"] == 0  # 72 and 80 of 152 SMs
    assert packed([50000] * 4)[0]["huge"] == 4 and packed([50000] * 5)[0]["huge"] == 0  # half as many
    assert packed([32768])[0]["huge"] == 1 and packed([32767])[0]["huge"] == 0
    assert packed([40000] + [1000] * 3760)[0]["huge"] == 1 and packed([40000] + [1000] * 3780)[0]["huge"] == 0

"""The hemi-Dslash launcher refuses what the kernel it would choose leaves out
(reductions, fused CG updates) instead of running without it: an internal
client (tests/c_client/dslash_requests.cu) links libhmc.so and makes each such
request on a context without a GPU behind it.  Nothing is launched."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
EINVAL = 1


@pytest.fixture(scope="module")
def rows(tmp_path_factory):
    from paper_1805_03560_gb300 import build as B
    B.build()
    exe = str(tmp_path_factory.mktemp("requests") / "dslash_requests")
    subprocess.run([B.nvcc(), *B.ARCH, *B.FLAGS, "-I", B.CSRC,
                    os.path.join(ROOT, "tests", "c_client", "dslash_requests.cu"),
                    "-L", B.HERE, "-lhmc", "-Xlinker", "-rpath", "-Xlinker", B.HERE, "-o", exe],
                   check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
    return [line.split(" ", 2) for line in out.splitlines()]


def test_requests_no_kernel_carries_out_are_refused(rows):
    assert len(rows) == 16
    wrong = [r for r in rows if int(r[1]) != EINVAL]
    assert not wrong, wrong
    assert all(r[2].startswith("dslash: ") for r in rows)

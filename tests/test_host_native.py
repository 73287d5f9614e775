"""Host-side rules of the native library, checked without a GPU by the small
program host_checks.cu, which is compiled against the library's sources."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def checks(tmp_path_factory):
    from paper_2206_02255_gb300 import build
    exe = str(tmp_path_factory.mktemp("host") / "host_checks")
    nvcc = os.path.join(build.cuda_home(), "bin", "nvcc")
    subprocess.run([nvcc] + build.NVCC_COMMON + ["-I", build.CSRC, os.path.join(HERE, "host_checks.cu"),
                    "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("name", ["queue_leaf_entries", "level_ticket_counter", "leaf_item_counter",
                                  "pool_does_not_fit", "occupancy_by_device",
                                  "chained_launch_error"])
def test_host_rule(checks, name):
    r = subprocess.run([checks, name], stdout=subprocess.PIPE, text=True)
    assert r.returncode == 0, r.stdout

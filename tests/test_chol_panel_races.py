"""The Cholesky panel's diagonal block (csrc/chol_panel.cuh) compiled for the host: no two threads touch a shared word, one
of them storing, without a barrier between them; and L L^+ is the block."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2403_04252_gb300", "csrc")


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    out = str(tmp_path_factory.mktemp("chol") / "chol_panel")
    subprocess.run(["g++", "-std=c++20", "-O1", "-pthread", "-I", CSRC, os.path.join(HERE, "chol_panel_host.cpp"), "-o", out],
                   check=True)
    return out


@pytest.mark.parametrize("nb", [1, 2, 31, 32])
def test_every_shared_store_of_the_panel_is_ordered(program, nb):
    open_pairs, err, info = subprocess.run([program, str(nb)], check=True, capture_output=True, text=True).stdout.split()
    assert int(open_pairs) == 0 and int(info) == 0
    # nb multiply-adds per element of a block with entries below 2 + nb / 50
    assert float(err) <= 8 * nb * 2.0 ** -53 * (2 + nb / 50)

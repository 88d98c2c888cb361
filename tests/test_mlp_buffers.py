"""A network whose buffers could not be enlarged for a large batch goes on with smaller ones: every allocation
of the large pass is made to fail in turn, on a stand-in for the CUDA runtime (no GPU; on one, a copy or a
kernel would be handed the null pointer of a buffer that was lost)."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lines(mess, tmp_path_factory):
    from paper_2406_03121_gb300 import build
    out = str(tmp_path_factory.mktemp("host") / "mlp_buffers")
    host = os.path.join(HERE, "host")
    subprocess.run([build._nvcc()] + build.NVCC_FLAGS + ["-cudart", "none", os.path.join(host, "mlp_buffers.cu"),
                                                         os.path.join(host, "fake_cudart.cpp"), "-o", out], check=True)
    return subprocess.run([out], check=True, capture_output=True, text=True).stdout.split("\n")


def _passes(lines):
    """(failing allocation, status of the large pass, status of the small one after it, its buffers whole)"""
    rows = [tuple(map(int, ln.split())) for ln in lines if ln[:1].isdigit()]
    assert len(rows) >= 10 and rows[-1][1] == 0      # in the last one nothing was left to fail
    return rows[:-1]


def test_the_input_buffer_is_allocated_again(mess, lines):
    k, large, small, whole = _passes(lines)[0]
    assert (large, small, whole) == (mess.MESS_ENOMEM, mess.MESS_OK, 1)
    assert "null 0" in lines


def test_the_activation_buffers_are_allocated_again(mess, lines):
    for k, large, small, whole in _passes(lines)[1:]:
        assert (large, small, whole) == (mess.MESS_ENOMEM, mess.MESS_OK, 1), k


def test_a_destroyed_network_holds_nothing(lines):
    assert "held 0" in lines

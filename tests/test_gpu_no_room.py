"""Where device memory runs out.  The allocator that runs out is a fake on the host (fake_alloc/limit.c,
compiled here and loaded before the CUDA runtime's users in a child process)."""
import os
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def shim(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("shim") / "limit.so")
    subprocess.run(["gcc", "-O1", "-shared", "-fPIC", os.path.join(HERE, "fake_alloc", "limit.c"), "-o", out, "-ldl",
                    "-lpthread"], check=True)
    return out


def _child(shim, check, precision, p):
    r = subprocess.run([sys.executable, os.path.join(HERE, "no_room_child.py"), shim, check, precision, str(p)],
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and "CHILD OK" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]


@pytest.mark.parametrize("precision,p", [("fp64", 1), ("fp32", 2), ("mixed", 2)])
def test_refused_allocations_of_a_creation_leave_nothing(shim, precision, p):
    _child(shim, "creation", precision, p)


@pytest.mark.parametrize("p", [1, 2, 3])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_calls_run_in_the_memory_they_cannot_do_without(shim, precision, p):
    _child(shim, "room", precision, p)


def test_adjoint_leaves_steps_on_another_stream_alone(shim):
    _child(shim, "streams", "fp64", 3)

"""Rules of the host code that need no GPU."""
import os
import re
import subprocess

import pytest


def _symbols():
    from paper_1809_07088_gb300 import build
    return subprocess.run(["nm", "--defined-only", build.build()], capture_output=True, text=True).stdout


def test_atom_count_of_the_corner_maxima_is_64_bit():
    """ds::corner_xmax counts model x site x cell: 16 sites of 128^3 cells and 64 supercells are 2^31 atoms,
    which a 32-bit count would turn into none (x_max = 0, order 2).  The first parameter of its mangled
    name is long long."""
    names = set(re.findall(r"_ZN2ds11corner_xmaxE\w+", _symbols()))
    assert names
    assert all(re.match(r"_ZN2ds11corner_xmaxEx", n) for n in names)


def _host_program(folder, source, obj):
    """An object file of the library linked with stand-ins for the CUDA runtime (source)."""
    from paper_1809_07088_gb300 import build
    build.build()
    exe = str(folder / source[:-3])
    cmd = [build._nvcc(), *build.ARCH, *build.FLAGS, "-cudart", "none",
           os.path.join(os.path.dirname(os.path.abspath(__file__)), source), os.path.join(build.OUT, obj), "-o", exe, "-lpthread"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return exe


@pytest.fixture(scope="module")
def serving_host(tmp_path_factory):
    return _host_program(tmp_path_factory.mktemp("serving"), "serving_host.cu", "serving.o")


@pytest.mark.parametrize("case", ["planning_fails", "planning_fails_without_a_slot"])
def test_refused_request_frees_its_events_outside_the_lock(serving_host, case):
    """A displacive request whose planning fails is dropped without a driver call under the context's lock."""
    r = subprocess.run([serving_host, case], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stderr


def test_two_waiters_of_one_ticket(serving_host):
    """The result of a ticket goes to one of two threads that wait for it; the other is told that the ticket is
    unknown."""
    r = subprocess.run([serving_host, "two_waiters"], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stderr


def test_shared_amplitude_route_holds_nothing_when_its_scratch_cannot_be_had(tmp_path):
    exe = _host_program(tmp_path, "subbox_host.cu", "subbox_cells.o")
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stderr

"""Rules of the host code that need no GPU."""
import re
import subprocess


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

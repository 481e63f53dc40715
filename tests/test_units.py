"""How launches are cut into units, on the host: the largest batches, and scratch
that grows with the units."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2208_09136_gb300", "csrc")

MAIN = r"""
#include "units.cu"
#include <cstdio>
#include <cstdlib>
using namespace rqa;
// cells SERIES NE | lines SERIES NE OTHERS OTHER_NE UNIT_BANDS
int main(int argc, char **argv)
{
    const bool lines = argv[1][0] == 'l';
    const int64_t s = atoll(argv[2]), ne = atoll(argv[3]);
    const uint64_t p = (uint64_t)ne * (ne - 1) / 2;
    if (!lines) {
        const Split sp = split_cells(s * p, COUNT_NB, 152);
        printf("%d %d %lld\n", sp.nb, sp.rc, (long long)(s * units_of_series(ne, sp, false)));
        return 0;
    }
    const int64_t t = atoll(argv[4]), me = atoll(argv[5]);
    const int64_t bands = s * ((ne + 30) / 32) + t * ((me + 30) / 32);
    const Split sp = split_lines(s * p + t * ((uint64_t)me * (me - 1) / 2), bands, (int32_t)ne, atoi(argv[6]), 152);
    const int64_t units = s * units_of_series(ne, sp, false, LINE_BAND) + t * units_of_series(me, sp, false, LINE_BAND);
    printf("%d %d %lld %lld\n", sp.nb, sp.rc, (long long)units, (long long)(units * sp.nb * (int64_t)LINE_EDGE_BYTES));
    return 0;
}
"""


@pytest.fixture(scope="module")
def split(tmp_path_factory):
    d = tmp_path_factory.mktemp("units")
    (d / "main.cpp").write_text(MAIN)
    exe = str(d / "main")
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-I", "/usr/local/cuda/include", str(d / "main.cpp"), "-o", exe],
                   check=True)

    def run(*args):
        out = subprocess.run([exe] + [str(a) for a in args], check=True, capture_output=True, text=True).stdout
        return [int(v) for v in out.split()]
    return run


# the counting rounds take at most 2^31 - 1 units and count a unit in 32 bits
@pytest.mark.parametrize("series,ne", [(1, 3 << 25), (7, 3 << 25), (100, 3 << 25), (700, 3 << 25), (4, 10000), (1, 2)])
def test_units_of_the_counting_rounds(split, series, ne):
    nb, rc, units = split("cells", series, ne)
    assert 1 <= units < 2**31
    assert nb * 128 * rc < 2**32
    if series == 1 or ne < 1 << 20:
        assert rc <= 585 * 28  # as before for batches that fitted


# row chunks keep 2560 bytes for every band a unit may have: no more bands than
# the longest series has, whatever the tuned size
@pytest.mark.parametrize("unit_bands", [0, 1, 64])
def test_edge_scratch_of_the_line_pass(split, unit_bands):
    nb, rc, units, edges = split("lines", 1, 300, 19000, 33, unit_bands)
    assert rc < 300 and nb <= 10
    assert edges < 1 << 29
    nb, rc, units, edges = split("lines", 4, 10000, 0, 2, unit_bands)
    assert nb == max(unit_bands, 1) and edges < 1 << 26

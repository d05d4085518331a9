"""Host arithmetic of the persistent launch (no GPU): compiled from its header
with the C++ compiler and checked over the whole range of its arguments."""
import os
import re
import subprocess

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_0909_5215_gb300", "csrc")


def compiled(tmp_path, body):
    src = tmp_path / "t.cpp"
    src.write_text('#include <cstdio>\n#include <cstdlib>\n#include "hd_units.h"\nusing namespace hd;\n'
                   "int main() {\n%s\nreturn 0; }\n" % body)
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-O1", "-I", CSRC, str(src), "-o", exe], check=True)
    return subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split()


def test_arrivals_of_a_launch_stay_below_two_to_the_32(tmp_path):
    """Arrivals at a replica's barrier, all that one launch can make, fit the 32 bits that count them."""
    out = compiled(tmp_path, 'for (int nc = 0; nc <= 5000; ++nc) printf("%d\\n", persist_steps_max(nc));\n'
                             'printf("%d %d\\n", PERSIST_BARRIERS, PERSIST_BARRIERS_0);')
    steps, (per, first) = [int(v) for v in out[:-2]], [int(v) for v in out[-2:]]
    for nc, n in enumerate(steps):
        assert n >= 100000
        assert (n * per + first) * max(nc, 1) < 2 ** 32
        assert n == 2 ** 31 - 1 or ((n + 1) * per + first) * max(nc, 1) >= 2 ** 32
    # 3,600,000 steps of 608 CTAs do not, even at two barriers a step
    assert (3600000 * 2 + first) * 608 >= 2 ** 32 and steps[608] < 3600000
    # the count is that of the kernel: every barrier in its step loop, and one before it
    text = open(os.path.join(CSRC, "hd_kernels.cu")).read()
    body = text[text.index("k_persist(Dev D, int nsteps) {"):text.index("// ---------------------------------------------------------------- launchers")]
    assert len(re.findall(r"grp_barrier\(D, r, nc, B", body)) == per + first
    # and hd_step goes by it
    api = open(os.path.join(CSRC, "hd_api.cu")).read()
    assert "std::min(left, c->persist_steps)" in api and "persist_steps_max(" in api


def test_units_stay_inside_their_tile(tmp_path):
    """Every unit, also an empty one, starts at an atom of its tile, and a tile's units are its atoms, once each."""
    out = compiled(tmp_path, 'for (int w = 8; w <= 32; w *= 2) for (int n = 1; n <= 128; ++n) for (int k = 0; k < 128 / w; ++k) {'
                             ' const UnitSpan u = unit_span(1000, n, w, k); printf("%d %d %d %d %d\\n", w, n, k, u.first, u.n); }')
    v = [tuple(map(int, out[q:q + 5])) for q in range(0, len(out), 5)]
    atoms = {}
    for w, n, k, first, m in v:
        assert 1000 <= first < 1000 + n and 0 <= m <= w and first + m <= 1000 + n
        atoms.setdefault((w, n), []).extend(range(first, first + m))
    assert all(got == list(range(1000, 1000 + n)) for (w, n), got in atoms.items())

"""Threads per block and lanes per particle of the pair passes: what the caller
asked for where one thread has a particle, else the library's rules, on both
sides of each line (csrc/sph_internal.h, compiled for the host)."""
import subprocess

import pytest

MAIN = """
#include <cstdio>
#include <cstdlib>
#include "sph_internal.h"
int main(int argc, char** argv) {
  for (int k = 1; k + 2 < argc; k += 3) {
    sph::DevState S;
    S.fp64 = atoi(argv[k]);
    S.n = atoi(argv[k + 1]);
    S.pass_threads = atoi(argv[k + 2]);
    const sph::PassShape a = sph::pass_a_shape(S, true), s = sph::pass_a_shape(S, false), b = sph::pass_b_shape(S);
    printf("%d %d %d %d %d %d\\n", a.threads, a.lanes, s.threads, s.lanes, b.threads, b.lanes);
  }
}
"""

# (fp64, n, asked) -> pass A, pass A with feature surfaces, pass B
CASES = {
    (0, 16384, 0): ((256, 1), (256, 1), (256, 8)), (0, 16385, 0): ((256, 1), (256, 1), (256, 1)),
    (0, 16384, 128): ((128, 1), (128, 1), (256, 8)), (0, 16385, 128): ((128, 1), (128, 1), (128, 1)),
    (0, 524287, 0): ((256, 1), (256, 1), (256, 1)), (0, 524288, 0): ((256, 1), (256, 1), (128, 1)),
    (0, 524288, 256): ((256, 1), (256, 1), (256, 1)), (0, 524288, 128): ((128, 1), (128, 1), (128, 1)),
    (1, 8192, 0): ((128, 4), (32, 1), (128, 4)), (1, 8193, 0): ((32, 1), (32, 1), (32, 1)),
    (1, 8192, 256): ((128, 4), (256, 1), (128, 4)), (1, 8193, 256): ((256, 1), (256, 1), (256, 1)),
    (1, 131072, 0): ((32, 1), (32, 1), (32, 1)), (1, 131073, 0): ((64, 1), (64, 1), (64, 1)),
    (1, 131073, 128): ((128, 1), (128, 1), (128, 1)), (1, 131073, 256): ((256, 1), (256, 1), (256, 1)),
}


@pytest.fixture(scope="module")
def shapes(tmp_path_factory):
    # here, not above: the submodule takes the place of the package's build()
    from paper_1906_07925_gb300.build import flags, nvcc
    d = tmp_path_factory.mktemp("rules")
    src, exe = d / "rules.cu", d / "rules"
    src.write_text(MAIN)
    subprocess.run([nvcc(), *flags(), str(src), "-o", str(exe)], check=True, capture_output=True)
    args = [str(v) for key in CASES for v in key]
    out = subprocess.run([str(exe), *args], check=True, capture_output=True, text=True).stdout.split()
    v = [int(t) for t in out]
    rows = [tuple(zip(v[q:q + 6:2], v[q + 1:q + 6:2])) for q in range(0, len(v), 6)]
    return dict(zip(CASES, rows))


@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(map(str, c)))
def test_a_pair_pass_launches_as_asked(shapes, case):
    assert shapes[case] == CASES[case]

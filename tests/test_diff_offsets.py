"""Host-only: the parked odd sweep of the diffusion numbers its populations'
slots in 32 bits.  The form a launch variant runs in is taken from the source
(compiled here as a host program), and wherever that is the parked one the
sweep's 32-bit arithmetic has to name the slots that 64-bit arithmetic names
and to tell a node's own slots from its neighbours'."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PARKED, RECORDS, PLAIN = 9, 6, 5
M32 = 1 << 32


def limit(q):  # largest pitch (a multiple of 64 nodes) of q populations below 2^32
    return (M32 - 1) // q // 64 * 64


# below, at and above the limits; 1024 x 724 x 724 at a pore fraction of 0.421 and full
CASES = [(q, rec, p) for q in (7, 19) for rec in (0, 1)
         for p in (64, 5_760_000, limit(q) - 64, limit(q), limit(q) + 64, 226_050_944, 536_756_224 // 64 * 64)]


@pytest.fixture(scope="module")
def forms(tmp_path_factory):
    from paper_1410_1921_gb300 import build
    d = tmp_path_factory.mktemp("offsets")
    src = d / "forms.cu"
    src.write_text('#include <cstdio>\n#include "diff_core.cuh"\nint main() {\n' + "".join(
        f'  for (int v = 0; v < 10; ++v) std::printf("%d ", om::diff_odd_variant(v, {q}, {rec}, {p}ll));\n'
        '  std::puts("");\n' for q, rec, p in CASES) + "}\n")
    subprocess.run([build._nvcc(), "-std=c++17", "-I", build.CSRC, "-I", os.path.join(ROOT, "include"), str(src), "-o",
                    str(d / "forms")], check=True, capture_output=True)
    out = subprocess.run([str(d / "forms")], check=True, capture_output=True, text=True).stdout
    return dict(zip(CASES, ([int(x) for x in line.split()] for line in out.splitlines())))


@pytest.mark.parametrize("q,rec,pitch", CASES)
def test_parked_only_where_its_offsets_reach(forms, q, rec, pitch):
    form = forms[(q, rec, pitch)]
    assert form[:6] == [0, 1, 2, 3, 4, 5]
    if not rec:
        assert form[6:] == [PLAIN] * 4
        return
    assert form[6:9] == [6, 7, 8]
    assert form[9] == (PARKED if pitch <= limit(q) else RECORDS)
    if form[9] != PARKED:
        return
    for i in range(1, q):  # slot of population i at node n, and of its opposite: all distinct names below 2^32
        for n in (0, pitch - 1):
            off = (i * pitch + n) % M32
            assert off == i * pitch + n
            assert (off - i * pitch) % M32 < pitch                            # that population's own: a neighbour's slot
            for o in (i - 1, i + 1):                                          # opposites are neighbours in the numbering
                if 1 <= o < q:
                    assert (off - o * pitch) % M32 >= pitch

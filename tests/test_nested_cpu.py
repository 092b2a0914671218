"""The nested elimination's tables on the CPU: tests/nested_tree_check.cpp (compiled here) checks
every even lattice up to 64 x 64 in both forms of the leaves, and carries the elimination out in
complex double on 6 x 6 to 20 x 20 sites against a pivoted dense inverse."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def rows(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("nested") / "check")
    subprocess.run([shutil.which("g++") or "g++", "-O2", "-std=c++17", "-I",
                    os.path.join(ROOT, "paper_2311_04435_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "nested_tree_check.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe, "20"], check=True, capture_output=True, text=True)
    return [ln.split() for ln in r.stdout.splitlines()]


def test_every_lattice_in_both_forms(rows):
    assert {(int(r[0]), int(r[1])) for r in rows} == {(L, f) for L in range(6, 65, 2) for f in (0, 1)}


def test_fronts_fit_where_the_blocks_are_kept(rows):
    """A block's fronts (16 bytes per entry) take less room than the dense float32 block (8 bytes,
    rows padded to 32), except up to 8 x 8 sites, where F and W (N columns) lie behind it."""
    for L, form, entries in ((int(r[0]), int(r[1]), int(r[2])) for r in rows):
        N = L * L
        room = 8 * N * (-(-N // 32) * 32) + (2 * 8 * N * N if L <= 8 else 0)
        assert 16 * entries + 8 * 600 <= room, (L, form)


def test_elimination_matches_a_dense_inverse(rows):
    """Im z = 0.3, t = 1.3, random site energies: rounding grows by at most (4t / Im z)^2 = 300
    and by the sums' lengths; 1e-11 is 150 times that times 2^-52."""
    done = [r for r in rows if float(r[5]) >= 0.0]
    assert len(done) == 2 * len(range(6, 21, 2))
    for r in done:
        assert float(r[5]) <= 1e-11 * int(r[0]) ** 2 and float(r[6]) <= 1e-11, r

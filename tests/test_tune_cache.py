"""Host test of pd_autotune's cache lines (csrc/pd_tune.h): a line is read back as written, and only for the very form
of the step that it was made for; a line of the earlier format, which says nothing about the automatic mapping, is
passed over."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HDR = os.path.join(ROOT, "paper_2309_11273_gb300", "csrc")
FIELDS = ["n", "bonds", "entries", "dim", "precision", "bodies", "kinematics", "solver", "influence", "lattice", "shadow_lo",
          "bond_cache", "stage", "validate", "resident"]

SRC = r"""
#include "pd_tune.h"
static pd::TuneProblem problem(const long long* v, const char* dev) {
  pd::TuneProblem p;
  p.n = v[0]; p.bonds = v[1]; p.entries = v[2]; p.dim = v[3]; p.precision = v[4]; p.bodies = v[5]; p.kinematics = v[6];
  p.solver = v[7]; p.influence = v[8]; p.lattice = v[9]; p.shadow_lo = v[10]; p.bond_cache = v[11]; p.stage = v[12];
  p.validate = v[13]; p.resident = v[14]; p.device = dev;
  return p;
}
extern "C" void line_of(const long long* v, const char* dev, const int* t, char* out) {
  pd::TuneChoice c;
  c.block = t[0]; c.split = t[1]; c.pairs = t[2]; c.ring = t[3]; c.automatic = t[4] != 0;
  std::strcpy(out, pd::tune_line(pd::tune_key(problem(v, dev)), c).c_str());
}
extern "C" int parse(const char* line, const long long* v, const char* dev, int* t) {
  pd::TuneChoice c;
  if (!pd::tune_parse(line, pd::tune_key(problem(v, dev)), &c)) return 0;
  t[0] = c.block; t[1] = c.split; t[2] = c.pairs; t[3] = c.ring; t[4] = c.automatic ? 1 : 0;
  return 1;
}
"""


@pytest.fixture(scope="module")
def so(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("tune")
    (d / "t.cc").write_text(SRC)
    subprocess.run([cxx, "-std=c++17", "-O1", "-shared", "-fPIC", "-I" + HDR, str(d / "t.cc"), "-o", str(d / "t.so")], check=True)
    return ctypes.CDLL(str(d / "t.so"))


BASE = [1600, 41000, 45000, 2, 0, 1, 0, 0, 0, 0, 0, 1, 1, 0, 1]


def _line(so, v, t, dev=b"NVIDIA GB300"):
    out = ctypes.create_string_buffer(1024)
    so.line_of((ctypes.c_longlong * 15)(*v), dev, (ctypes.c_int * 5)(*t), out)
    return out.value


def _parse(so, line, v, dev=b"NVIDIA GB300"):
    t = (ctypes.c_int * 5)(*([-9] * 5))
    return list(t) if so.parse(line, (ctypes.c_longlong * 15)(*v), dev, t) else None


@pytest.mark.parametrize("choice", [[256, 1, 1, 0, 1], [64, 2, 0, 3, 0]])
def test_a_line_reads_back(so, choice):
    line = _line(so, BASE, choice)
    assert line.endswith(b"\n") and len(line) < 700
    assert _parse(so, line, BASE) == choice


@pytest.mark.parametrize("k", range(len(FIELDS)))
def test_a_line_of_another_form_is_passed_over(so, k):
    other = list(BASE)
    other[k] += 1
    assert _parse(so, _line(so, other, [64, 1, 1, 0, 0]), BASE) is None, FIELDS[k]


def test_other_devices_and_formats_are_passed_over(so):
    assert _parse(so, _line(so, BASE, [64, 1, 1, 0, 0], b"other"), BASE) is None
    full = _line(so, BASE, [64, 1, 1, 0, 0])
    assert _parse(so, full.rsplit(b" ", 1)[0] + b"\n", BASE) is None  # four numbers
    old = b"osbpd n=1600 bonds=41000 entries=45000 dim=2 prec=0 bodies=1 lattice=0 dev=NVIDIA GB300|64 1 1 0\n"
    assert _parse(so, old, BASE) is None
    for bad in (b"", b"no bar\n", b"|64 1 1 0 0\n", full.replace(b"|64", b"|x")):
        assert _parse(so, bad, BASE) is None


CAND = r"""
#include "pd_tune.h"
extern "C" int candidates(int fp64, int lattice, int try_pairs, int pairs, int ring, int* out) {
  int n = 0;
  for (const pd::TuneChoice& t : pd::tune_candidates(fp64, lattice, try_pairs, pairs, ring)) {
    int* o = out + 5 * n++;
    o[0] = t.block; o[1] = t.split; o[2] = t.pairs; o[3] = t.ring; o[4] = t.automatic;
  }
  return n;
}
"""


@pytest.mark.parametrize("fp64,lattice,try_pairs", [(1, 0, 1), (1, 0, 0), (0, 1, 0), (0, 0, 0)])
def test_what_an_untuned_context_runs_is_timed_too(tmp_path, fp64, lattice, try_pairs):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    (tmp_path / "c.cc").write_text(CAND)
    subprocess.run([cxx, "-std=c++17", "-O1", "-shared", "-fPIC", "-I" + HDR, str(tmp_path / "c.cc"), "-o",
                    str(tmp_path / "c.so")], check=True)
    out = (ctypes.c_int * 500)()
    n = ctypes.CDLL(str(tmp_path / "c.so")).candidates(fp64, lattice, try_pairs, 1, 0, out)
    got = [tuple(out[5 * k:5 * k + 5]) for k in range(n)]
    assert len(set(got)) == n
    pairs = [1, 0] if try_pairs else [1]
    assert [t for t in got if t[4]] == ([(256, 1, p, 0, 1) for p in pairs] if fp64 or lattice else [])
    splits = [1] if lattice else [1, 2, 4]
    rings = [0, 1, 2, 3] if lattice else [0]
    assert {t[:4] for t in got if not t[4]} == {(b, s, p, r) for b in (64, 128, 256, 512) for s in splits
                                                if (b // 32) % s == 0 for p in pairs for r in rings}

"""The launch rules of the row-split block orthonormalisation
(csrc/orth_rs_plan.h), compiled for the host: every call that takes the grid
form finds its shares inside the scratch planned for its mode, whichever of
the mode's blocks needs the most."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2308_01480_gb300", "csrc")

SOURCE = r"""
#include "orth_rs_plan.h"
#include <algorithm>
using namespace ttr;

// Alg. 3's blocks for an m x n unfolding (n large): b columns q + 1 times,
// capped at m in all.
static std::vector<int> krylov_blocks(int64_t m, int b, int q) {
  int64_t cols = std::min<int64_t>(b, m);
  std::vector<int> out{(int)cols};
  for (int j = 0; j < q && cols < m; ++j) {
    out.push_back((int)std::min<int64_t>(b, m - cols));
    cols += out.back();
  }
  return out;
}

extern "C" {

// The scratch of a mode; need[i]: what call i takes by itself in the grid
// form, -1 for a call that does not take it.  Returns the number of calls.
int mode_plan(int64_t m, int b, int q, int restarts, int ctas, int64_t smem, int64_t* scratch, int64_t* need) {
  const OrthGridLimits lim{ctas, (size_t)smem};
  std::vector<OrthCall> calls = orth_calls(b, krylov_blocks(m, b, restarts ? 0 : q), restarts != 0);
  *scratch = (int64_t)orth_grid_plan(m, lim, &calls);
  for (size_t i = 0; i < calls.size(); ++i) {
    OrthGridShape s;
    const bool fits = orth_grid_shape(m, calls[i].kq0 + calls[i].c, calls[i].zc, lim, &s);
    need[i] = fits && calls[i].grid ? (int64_t)s.scratch_floats() : -1;
  }
  return (int)calls.size();
}

// Over m in [1, m_max] (every step-th), b, q: the first mode whose scratch
// does not hold one of its calls, or whose shape breaks a limit; 0 if none.
int64_t sweep(int64_t m_max, int64_t step, int ctas, int64_t smem, int64_t* accepted) {
  const OrthGridLimits lim{ctas, (size_t)smem};
  *accepted = 0;
  for (int64_t m = 1; m <= m_max; m += step)
    for (int b = 1; b <= 64; ++b)
      for (int q = 0; (q + 1) * b <= 256; ++q) {
        std::vector<OrthCall> calls = orth_calls(b, krylov_blocks(m, b, q), false);
        const size_t scratch = orth_grid_plan(m, lim, &calls);
        for (const OrthCall& c : calls) {
          OrthGridShape s;
          if (!c.grid) continue;
          ++*accepted;
          if (!orth_grid_shape(m, c.kq0 + c.c, c.zc, lim, &s) || s.scratch_floats() > scratch || s.smem > lim.smem ||
              s.nr > ctas || (int64_t)s.nr * s.rows < m || (int64_t)(s.nr - 1) * s.rows >= m)
            return m * 100000 + b * 100 + q;
        }
      }
  return 0;
}
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("orth_plan")
    src, so = d / "plan.cpp", d / "plan.so"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(so)], check=True)
    lib = ctypes.CDLL(str(so))
    lib.sweep.restype = ctypes.c_int64
    return lib


def _mode(plan, m, b, q, restarts=0, ctas=152, smem=218 * 1024):
    scratch, need = ctypes.c_int64(), (ctypes.c_int64 * 64)()
    n = plan.mode_plan(ctypes.c_int64(m), b, q, restarts, ctas, ctypes.c_int64(smem), ctypes.byref(scratch), need)
    return scratch.value, list(need)[:n]


@pytest.mark.parametrize("ctas,smem", [(152, 218 * 1024), (152, 218720), (152, 200000), (148, 221000), (132, 218 * 1024)])
def test_every_grid_call_fits_the_planned_scratch(plan, ctas, smem):
    accepted = ctypes.c_int64()
    assert plan.sweep(ctypes.c_int64(45000), ctypes.c_int64(89), ctas, ctypes.c_int64(smem), ctypes.byref(accepted)) == 0
    assert accepted.value > 100000


@pytest.mark.parametrize("m,b,q,widest", [(11250, 55, 2, 1), (9000, 50, 3, 2), (9000, 64, 1, 0)])
def test_scratch_covers_earlier_blocks_when_the_last_is_refused(plan, m, b, q, widest):
    """Modes whose last block does not fit shared memory while earlier ones do:
    152 or fewer CTAs' shares of (pad4(kq0 + c) + pad4(b)) pad4(b) floats,
    twice, and their sums twice."""
    scratch, need = _mode(plan, m, b, q)
    assert need[-1] == -1 and need[widest] > 0 and need[widest + 1] == -1
    pad = lambda x: (x + 3) // 4 * 4
    rows = -(-m // 152)
    e = (pad(b * (widest + 1)) + pad(b)) * pad(b)
    assert need[widest] == 4 + 2 * -(-m // rows) * e + 2 * e
    assert scratch == max(need)


def test_restarted_calls_and_no_device(plan):
    scratch, need = _mode(plan, 12000, 60, 3, restarts=1)
    assert len(need) == 2 and scratch == max(need) > 0
    assert _mode(plan, 12000, 60, 3, ctas=0) == (0, [-1] * 4)


@pytest.mark.parametrize("m,b,q,full", [(44394, 18, 5, 232176), (40417, 21, 4, 230000), (45946, 26, 2, 228880)])
def test_blocks_that_fit_only_the_tight_layout_keep_the_grid_form(plan, m, b, q, full):
    """Layouts whose split partial products, sized for Q^T Z as well, take the
    last block past the 221,920 bytes of a CTA."""
    assert full > 221920
    scratch, need = _mode(plan, m, b, q, smem=221920)
    assert min(need) > 0 and scratch == max(need)

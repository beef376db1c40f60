"""The exact-slice products' plan arithmetic (csrc/exactplan.h), compiled for the host: every piece
of K fits its workspace, and every workspace that holds 64 terms' operands is enough."""
import os
import random
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2309_08572_gb300", "csrc")

DRIVER = r"""
#include <cstdio>
#include "exactplan.h"
using namespace mpdo;
// one line a product: m n k batch gram workspace (0: the entry points' own)
int main() {
  long m, n, k, ws; int batch, gram;
  while (std::scanf("%ld %ld %ld %d %d %ld", &m, &n, &k, &batch, &gram, &ws) == 6) {
    const size_t w = ws ? (size_t)ws : exact_ws_bytes(m, n, k, batch, gram);
    const long kc = exact_piece(m, n, k, batch, gram, w);
    const bool fits = exact_operand_bytes(m, n, std::min(k, 64L), batch, gram) <= w;
    bool ok = fits == (kc > 0) && (kc == k || kc % 64 == 0);
    long pieces = 0;
    for (long k0 = 0; kc > 0 && k0 < k; k0 += kc, ++pieces) {
      const long kn = std::min(kc, k - k0);
      const ExactPlan p = exact_piece_plan(m, n, kn, batch, gram, w);
      ok = ok && exact_operand_bytes(m, n, kn, batch, gram) + exact_part_bytes(p) <= w;
      ok = ok && p.ctas <= kExactSms && p.ctas * p.per >= p.total && (p.ctas - 1) * p.per < p.total;
      ok = ok && (p.parts || p.per % p.nst == 0 || p.total == 0);
    }
    std::printf("%d %ld\n", ok ? 1 : 0, pieces);
  }
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    cxx = shutil.which("g++") or pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("plan")
    (d / "t.cpp").write_text(DRIVER)
    subprocess.run([cxx, "-std=c++17", "-O2", "-I", CSRC, str(d / "t.cpp"), "-o", str(d / "t")],
                   check=True)

    def run(rows):
        out = subprocess.run([str(d / "t")], input="\n".join(" ".join(map(str, r)) for r in rows),
                             capture_output=True, text=True, check=True).stdout.split()
        return list(zip(map(int, out[::2]), map(int, out[1::2])))
    return run


MB = 1 << 20


def test_pieces_fit(plan):
    """Sizes of the update's products in the handles' workspaces and of the entry points in their
    own, beside ones that a shorter piece's larger plan overran or refused."""
    rng = random.Random(7)
    rows = [(105, 105, 10962, 1, 1, 64 * MB), (120, 64, 3264, 3, 0, 64 * MB),
            (839, 36, 45027, 2, 0, 64 * MB), (2, 2, 8740, 1, 1, 0), (9, 9, 18704, 1, 1, 0),
            (10, 2, 8123, 3, 0, 0)]
    for _ in range(20000):
        def log(lo, hi):
            return int(round(lo * (hi / lo) ** rng.random()))
        m, k, b = log(1, 3000), log(1, 60000), rng.choice([1, 1, 2, 3, 9])
        gram = rng.randrange(2)
        n = m if gram else log(1, 3000)
        rows.append((m, n, k, b, gram, rng.choice([0, 64 * MB, 256 * MB, log(MB // 4, 64 * MB)])))
    bad = [r for r, (ok, _) in zip(rows, plan(rows)) if not ok]
    assert not bad, (len(bad), bad[:10])


def test_own_workspace_takes_one_piece(plan):
    """With the workspace that the entry points ask for, pieces of up to 4096 terms."""
    rng = random.Random(8)
    rows = []
    for _ in range(20000):
        n, k = rng.randint(1, 900), int(round(10 ** rng.uniform(0, 4.5)))
        gram = rng.randrange(2)
        rows.append((n if gram else rng.randint(1, 900), n, k, rng.choice([1, 1, 3]), gram, 0))
    bad = [r for r, (ok, p) in zip(rows, plan(rows)) if not ok or p > (r[2] + 4095) // 4096]
    assert not bad, (len(bad), bad[:10])


def test_empty_products(plan):
    """No rows, no columns or no batch: nothing to plan, and no division by a plan of nothing."""
    rows = [(0, 5, 7, 1, 0, 0), (5, 0, 7, 1, 0, 0), (0, 0, 300, 2, 1, 0), (4, 4, 9, 0, 1, 0)]
    for r in rows:
        ((ok, _),) = plan([r])
        assert ok, r


ROUTES = r"""
#include <cstdio>
#include "exactplan.h"
using namespace mpdo;
int main() {
  // threshold given (0, below and above the default) or not; a small product, one that the FP64 cores
  // do faster, a large one, one with a short side
  const long size[4][4] = {{20, 20, 20, 0}, {41, 41, 1968, 1}, {400, 400, 5043, 1}, {15, 900, 900, 0}};
  for (const ExactRoute& r : {ExactRoute{0, true}, ExactRoute{1 << 20, true}, ExactRoute{1 << 24, true},
                              ExactRoute{1 << 21, false}})
    for (const auto& s : size) std::printf("%d ", r.takes(s[0], s[1], s[2], 1, s[3] != 0) ? 1 : 0);
}
"""


def test_given_threshold_forces_the_route(tmp_path):
    """A threshold from the environment decides alone, in every caller (updates and eigensolver share
    the rule); otherwise the estimate has a say."""
    cxx = shutil.which("g++") or pytest.skip("no host compiler")
    (tmp_path / "r.cpp").write_text(ROUTES)
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(tmp_path / "r.cpp"), "-o",
                    str(tmp_path / "r")], check=True)
    out = subprocess.run([str(tmp_path / "r")], capture_output=True, text=True, check=True).stdout
    assert list(map(int, out.split())) == [1, 1, 1, 0, 0, 1, 1, 0, 0, 0, 1, 0, 0, 0, 1, 0]

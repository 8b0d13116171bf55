"""The short path's records, on the host: a reaction that may take the short
path has a code of its jump table that says the shapes of its sides, and
factors that are its coefficients.  Every pair of sides of up to four species
with coefficients 1 to 4 (and 8), reversible and not."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

PROGRAM = r"""
#include <cstdio>
#include <cstring>
#include <functional>
#include <map>
#include <vector>

#include "rxn_pack.h"

using namespace pj;

int main() {
  std::vector<std::vector<int>> sides;  // coefficients, descending
  std::vector<int> cur;
  std::function<void(int)> grow = [&](int most) {
    if (!cur.empty()) sides.push_back(cur);
    if (cur.size() == PJ_MAX_SP) return;
    for (int v = most; v >= 1; v--) {
      cur.push_back(v);
      grow(v);
      cur.pop_back();
    }
  };
  grow(4);
  sides.push_back({8});
  const int factors[5] = {1, 2, 2, 3, 3};  // of the shapes in the jump table
  int bad = 0, lean = 0;
  for (const auto& f : sides)
    for (const auto& b : sides)
      for (int rev = 0; rev < 2; rev++) {
        Rxn r;
        std::memset(&r, 0, sizeof r);
        r.rev = rev;
        for (int a = 0; a < 2 * PJ_MAX_SP; a++) r.sp[a] = -1;
        std::map<int, int> want[2];
        for (int side = 0; side < 2; side++) {
          const auto& c = side ? b : f;
          for (size_t a = 0; a < c.size(); a++) {
            r.sp[side * PJ_MAX_SP + a] = (int)(3 + 5 * side + a);
            r.nu[side * PJ_MAX_SP + a] = c[a];
            want[side][32 * r.sp[side * PJ_MAX_SP + a]] = c[a];
          }
          (side ? r.nprod : r.nreac) = (int)c.size();
          r.shape[side] = side_shape(&r.nu[side * PJ_MAX_SP], (int)c.size());
        }
        pack_head(r, true);
        if (!r.head.lean) continue;
        lean++;
        const int sf = r.head.code / 6, sb = r.head.code % 6 - 1;
        bool ok = r.head.code < 30 && sf == r.shape[0] && sb == (rev ? r.shape[1] : -1);
        ok = ok && factors[sf] == r.head.nf && (sb < 0 || factors[sb] == r.head.nb);
        for (int side = 0; side < 2; side++) {
          std::map<int, int> got;
          for (int u = 0; u < (side ? r.head.nb : r.head.nf); u++) got[side ? r.head.b[u] : r.head.f[u]]++;
          ok = ok && got == want[side];
        }
        if (!ok) {
          bad++;
          std::printf("code %d shapes %d %d rev %d\n", r.head.code, r.shape[0], r.shape[1], rev);
        }
      }
  // 5 forward shapes times 5 reversible ones, and times 6 irreversible products (3A too)
  std::printf("lean %d bad %d\n", lean, bad);
  return bad != 0 || lean != 5 * 5 + 5 * 6;
}
"""


def test_short_path_records(tmp_path):
    src, exe = tmp_path / "pack.cpp", tmp_path / "pack"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_1809_01029_gb300", "csrc"), "-I",
                    os.path.join(ROOT, "include"), "-I", os.path.join(CUDA, "include"), str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout[-2000:]

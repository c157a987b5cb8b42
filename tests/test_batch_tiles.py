"""Host check of the batch's launch shapes (no GPU): a small program packs batch segments as gp_batch_create
does.  A batch runs the default shape of its outputs and of the faces of all its segments, and every default shape
is within the limits of the kernels."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2503_00246_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "gp_launch.h"
using namespace gp;
int bad = 0;
template <int D, int K, class A>
void check(const char* name) {
  const int64_t sizes[] = {0, 1, 999, 1001, 2500, 2501, 5000, 8000, 11000, 14000, 18000, 20000, 23000, 30000, 45000, 60000, 1000000};
  for (int f = 0; f < 34; ++f) {
    const LaunchForm form{f >= 17, sizes[f % 17]};
    Tiles want, got;
    std::vector<unsigned char> fs, ls;
    std::vector<SegSpec> in(3);
    int fb = 0, lb = 0, nf = 0, nl = 0;
    const Tiles def = default_tiles_t<D, K, typename A::V>(form);
    if (!resolve_tiles<D, K, typename A::V>(want, form) || want.fb != def.fb || want.lcb != def.lcb || want.lnt != def.lnt ||
        face_smem<D, K, typename A::V>(def.fb) > MAX_DYN_SMEM) {
      std::printf("FAIL %s d=%d k=%d limits\n", name, D, K);
      ++bad;
      return;
    }
    const int cb = lift_cells<D, K, typename A::V>(want, form.compact);
    for (int i = 0; i < 3; ++i) {
      const int faces = 7 + 100 * i, owners = 50 + 333 * i;
      for (int a = 0; a < 4; ++a) in[i].fa.fstart[a] = a == 0 ? 0 : faces;   // faces of normal x only
      in[i].la.nlift = owners;
      in[i].fa.nzruns = 0;
      nf += (faces + want.fb - 1) / want.fb;
      nl += (owners + cb - 1) / cb;
    }
    if (!pack_batch<D, K, A>(in, form, got, fs, ls, fb, lb) || fb != nf || lb != nl || got.fb != want.fb ||
        got.lcb != want.lcb || got.lnt != want.lnt) {
      std::printf("FAIL %s d=%d k=%d %s, %d faces: %d of %d face CTAs, %d of %d lift CTAs\n", name, D, K, form.compact ? "compact" : "W_F",
                  (int)form.faces, fb, nf, lb, nl);
      ++bad;
    }
  }
}
template <int D, class A, int... Ks>
void all(const char* name, std::integer_sequence<int, Ks...>) { (check<D, Ks + 1, A>(name), ...); }
// the instances of the compact form cover what store_compact asks for, at every size
template <int D, int K>
void check_form() {
  for (int mb = 0; mb <= 1 << 16; mb = mb ? 2 * mb : 1) {
    const bool c = store_compact(D, K, (int64_t)mb << 20);
    if ((c && !StoreCompact<D, K, float>::value) || (!c && StoreCompact<D, K, float>::always)) {
      std::printf("FAIL compact d=%d k=%d %d MB\n", D, K, mb);
      ++bad;
    }
  }
}
template <int D, int... Ks>
void all_forms(std::integer_sequence<int, Ks...>) { (check_form<D, Ks + 1>(), ...); }
int main() {
  const auto ks = std::make_integer_sequence<int, 8>{};
  all_forms<2>(ks); all_forms<3>(ks);
  all<2, ArF32>("f32", ks); all<3, ArF32>("f32", ks);
  all<2, ArF64>("f64", ks); all<3, ArF64>("f64", ks);
  all<2, ArFF>("ff", ks); all<3, ArFF>("ff", ks);
  return bad ? 1 : 0;
}
"""


def _nvcc():
    for c in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", shutil.which("nvcc")):
        if c and os.path.exists(c):
            return c
    return None


def test_batches_run_the_default_shape_of_their_form(tmp_path):
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not available")
    src = tmp_path / "tiles.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "tiles"
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-I", CSRC, "-I", os.path.join(ROOT, "include"), str(src), "-o", str(exe)],
                   check=True, capture_output=True, timeout=300)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0, out.stdout + out.stderr

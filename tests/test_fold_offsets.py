"""Row offsets of the strided two-step passes, on the host: the byte offset that the kernels' own function gives a thread
equals the 64-bit one at every supported row stride, for every plan, without a GPU."""
import subprocess

from paper_2209_11922_gb300 import build

SRC = r"""
#include <cstdio>
#include "fold_dst.cuh"
using namespace etd;
template <class T, class F> int check(const char* name, int n) {
  static const long long len[] = {4, 6, 8, 12, 16, 24, 32, 48, 64, 96, 128, 192, 256, 384, 512, 768, 1024, 1536, 2048};
  int bad = 0, rows = 0;
  auto one = [&](long long row, long long stride) {
    for (int col = 0; col < FOLD_MAX_COLUMN; col += 2) {
      ++rows;
      if ((long long)fold_offset<F, T>((int)row, (size_t)stride, col) != (row * stride + col) * (long long)sizeof(T)) ++bad;
    }
  };
  for (long long x : len)
    for (long long y : len)
      for (long long stride : {x, x * y}) {   // y axis, z axis
        for (int s = 0; s < F::SLOTS; ++s) {
          one(F::row1(s), stride);
          one(F::row2(s), stride);
        }
        for (int l = 0; l < F::UA; ++l) {
          one(l, stride);
          one(F::partner_row(l), stride);
        }
      }
  // every row of the axis is reached once by step A and once by step B
  int a[2048] = {}, b[2048] = {};
  for (int l = 0; l < F::UA; ++l)
    for (int r = 0; r < F::H; ++r) {
      ++a[l + r * F::L];
      ++a[F::partner_row(l) + (F::PARTNER_STEPS + r) * F::L];
    }
  for (int s = 0; s < F::SLOTS; ++s)
    for (int i = 0; i < F::HV; ++i) {
      ++b[F::row1(s) + i * F::STEP];
      ++b[F::row2(s) + i * F::STEP];
    }
  int miss = 0;
  for (int j = 0; j < n; ++j) miss += (a[j] != 1) + (b[j] != 1);
  printf("%s %d %d %d %d %d\n", name, n, (int)sizeof(T), rows, bad, miss);
  return bad + miss;
}
int main() {
  int bad = 0;
@CALLS@
  return bad ? 1 : 0;
}
"""


def test_every_row_offset_is_exact(tmp_path):
    calls = []
    for tk, tn in build.TYPES.items():
        for kind, lengths, f in (("fold", build.FOLD, "Fold<{t}, {n}>"), ("foldm", build.FOLDM[tk], "Fold<{t}, {n}, true>"),
                                 ("foldh", build.FOLDH[tk], "FoldH<{t}, {n}>")):
            calls += [f'  bad += check<{tn}, {f.format(t=tn, n=n)}>("{kind}", {n});' for n in lengths]
    src = tmp_path / "offsets.cu"
    src.write_text(SRC.replace("@CALLS@", "\n".join(calls)))
    exe = tmp_path / "offsets"
    subprocess.run([build.nvcc(), "-O1", "-std=c++17", *build.ARCH, "--expt-relaxed-constexpr", f"-I{build.CSRC}",
                    f"-I{build.INCLUDE}", "-o", str(exe), str(src)], check=True, capture_output=True, text=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    rows = [ln.split() for ln in r.stdout.splitlines()]
    assert len(rows) == len(calls)
    wrong = [ln for ln in rows if ln[4] != "0" or ln[5] != "0"]
    assert not wrong and r.returncode == 0, wrong
    assert all(int(ln[3]) > 10000 for ln in rows)

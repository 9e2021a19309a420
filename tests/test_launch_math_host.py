"""Index arithmetic of the kernels and their launches (csrc/launch_math.h), compiled with
the host compiler and compared with Python's integers at the sizes where 32 bits end."""
import os
import re
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2601_20550_gb300", "csrc")


def run(tmp_path, body):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text('#include <cstdio>\n#include "launch_math.h"\nint main() {\n' + body + "\n}\n")
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-fsanitize=undefined",
                    "-fno-sanitize-recover=undefined", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    return subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()


# hierarchies that fit one GPU and are accepted: 12 exponentials at depth 10 (42 GB a state),
# d = 36 with 2042975 ADOs, and small bases with as many matrices
@pytest.mark.parametrize("d,n_ado", [(64, 646646), (36, 2042975), (216, 24310), (6, 1 << 26), (1, 1 << 30)])
def test_ado_offsets_pass_32_bits(tmp_path, d, n_ado):
    ns = [0, 1, (1 << 31) // (d * d) - 1, (1 << 31) // (d * d), n_ado - 1]
    out = run(tmp_path, "".join(f'  printf("%lld\\n", (long long)heom::ado_offset({n}, {d}));\n' for n in ns))
    assert [int(v) for v in out] == [n * d * d for n in ns]


def test_fp64_kernels_take_ado_offsets_from_there():
    """No 32-bit index of an item (an ADO of a branch) in the FP64 kernels, and no 32-bit
    product of an ADO index with d^2: an int dd appears only beside 64-bit indexes or within
    one block's items."""
    src = open(os.path.join(CSRC, "f64_stage.cu")).read()
    for body in re.split(r"__global__", src)[1:]:
        body = body.split("\n}\n", 1)[0]
        assert not re.search(r"const int (first|i0|item)\b", body), body[:200]
        if re.search(r"const int [^;]*\bdd = ", body):
            assert not re.search(r"(?<![\w.])n \* dd\b", body), body[:200]


def test_a_shape_kept_by_another_kernel_is_not_used(tmp_path):
    """All steps in one launch (512 threads) and a launch per stage (at most 384) record their
    shapes under one key; a stage takes a kept shape only if it is one of its own."""
    out = run(tmp_path, """
  heom::ShapeMap kept{{{0, 9072}, {512, 28}}, {{0, 100}, {128, 7}}, {{0, 200}, {256, 9}}};
  const std::vector<heom::Shape> mine{{256, 7}, {128, 7}, {64, 7}};
  printf("%d ", heom::kept_shape(kept, 0, 9072, mine[0], mine) != nullptr);
  printf("%d ", heom::kept_shape(kept, 0, 100, mine[0], mine)->first);
  printf("%d ", heom::kept_shape(kept, 0, 200, {256, 9}, mine)->second);
  printf("%d ", heom::kept_shape(kept, 1, 100, mine[0], mine) != nullptr);
  printf("%d", heom::kept_shape(kept, 0, 101, mine[0], mine) != nullptr);""")
    assert out == ["0", "128", "9", "0", "0"]


def test_blocks_of_a_launch(tmp_path):
    """A grid beyond 2^31 - 1 blocks is refused, not truncated; work that can be split is taken
    in launches that hold whole items and end."""
    out = run(tmp_path, """
  printf("%u ", heom::grid_blocks(0x7fffffffLL));
  for (int64_t b : {0x80000000LL, 0x100000000LL, -1LL}) {
    bool refused = false;
    try { heom::grid_blocks(b); } catch (const std::invalid_argument &) { refused = true; }
    printf("%d ", refused);
  }
  for (int per : {1, 3, 14})
    for (int64_t items : {0LL, 5LL, 0x7fffffffLL, 2800000000LL, 9000000000LL}) {
      int64_t rest = items, done = 0, n = 0;
      int launches = 0;
      for (; rest > 0; rest -= n, done += n, ++launches) {
        n = heom::launch_share(rest, per);
        heom::grid_blocks(n * per);
      }
      printf("%d ", done == items && launches == (items + 0x7fffffffLL / per - 1) / (0x7fffffffLL / per));
    }""")
    assert out == ["2147483647", "1", "1", "1"] + ["1"] * 15


def test_tiled_launches_check_their_grids():
    for name in ("kernels.cu", "f64_stage.cu"):
        src = open(os.path.join(CSRC, name)).read()
        assert not re.search(r"<<<\(unsigned\)\(items", src), name
        assert not re.search(r"blocks = \(unsigned\)", src), name

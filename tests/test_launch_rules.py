"""The launch rules (csrc/launch_rules.h, plain C++) over the sizes that hierarchies have, compiled for the host.

- coarse stencil: every tile it picks has a kernel, fits the reduction's partials, and leaves few lanes idle;
- fine stencil: the FP64 kernel needs 144 registers, and a larger budget only makes more waves;
- early starts: launches that would crowd their predecessor wait for its end.
"""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0811_4331_gb300", "csrc")


def _run(tmp_path, body):
    if not shutil.which("g++"):
        pytest.skip("g++ not available")
    src = tmp_path / "rules.cpp"
    src.write_text("#include <cstdio>\n#include \"launch_rules.h\"\nusing namespace wmg;\nint main() {\n%s\n}\n" % body)
    exe = tmp_path / "rules"
    subprocess.run(["g++", "-O1", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout
    return [tuple(int(x) for x in line.split()) for line in out.splitlines()]


def test_coarse_tiles(tmp_path):
    rows = _run(tmp_path, """
  const int elems[] = {16, 8, 4};
  for (int elem : elems)
    for (long n = 2; n <= 128; n += n < 20 ? 2 : 6)
      for (long V = 1; V <= 20000; V += V < 130 ? 1 : V / 7)
        for (int r = 1; r <= 64; r += r < 6 ? 1 : 5) {
          const CoarseShape s = coarse_shape(elem, n, V, r, 152);
          const int bv = coarse_bv(elem, V);
          printf("%d %d %ld %ld %d %d %d %d %ld %ld %ld %d\\n", elem, bv, n, V, r, s.ir, s.rb, s.lb, s.pitch,
                 coarse_ctas(n, s.ir, s.lb, s.pitch), coarse_blocks(n, V, r),
                 coarse_has(elem, bv, s.ir, s.rb, s.lb));
        }""")
    assert len(rows) > 10000
    for elem, bv, n, V, r, ir, rb, lb, pitch, ctas, blocks, has in rows:
        case = (elem, n, V, r)
        assert has, (case, ir, rb, lb)
        assert ctas <= blocks, case
        groups = V // bv
        assert ctas * lb >= -(-n // ir) * pitch and pitch >= groups, case
        # lanes: FP64 (bound by arithmetic) idles in the last CTA alone, the others less than a third of a row
        assert pitch == groups if elem == 16 else 2 * pitch < 3 * groups, case
        assert pitch == groups or pitch % lb == 0, case


def test_fp64_stencil_budget(tmp_path):
    (threads,), = _run(tmp_path, 'printf("%d\\n", stencil_threads(16, 1, false));')
    assert 65536 // threads // 8 * 8 < 144 + 32


def test_crowded_launches_wait(tmp_path):
    # CTAs, places of an SM, whether an early start pays (FP64 transfers, even-odd split, FP64 stencils, measured)
    cases = [(384, 6, 1), (512, 6, 0), (625, 6, 0), (768, 6, 1), (324, 5, 1), (432, 5, 0), (648, 5, 1), (256, 3, 0),
             (336, 3, 0), (1024, 3, 1)]
    rows = _run(tmp_path, "\n".join('printf("%%d\\n", (int)chain_fits(%d, %d, 152));' % c[:2] for c in cases))
    assert [r[0] for r in rows] == [c[2] for c in cases]


def test_dot_tiles_fill_their_waves(tmp_path):
    """FP32: waves times tiles per CTA, with a CTA's own 0.3 tile times, within 3 % of the best of the range; and two
    right-hand sides per thread count their own rows and places."""
    rows = _run(tmp_path, """
  for (long tiles = 9; tiles < 20000; tiles += tiles / 5 + 1)
    for (long lanes = 1; lanes <= 64; lanes += lanes < 8 ? 1 : 8)
      for (int per_sm = 3; per_sm <= 4; ++per_sm)
        printf("%ld %ld %d %d\\n", tiles, lanes, per_sm, dot_tiles(tiles, lanes, per_sm, 152, 8));""")
    for tiles, lanes, per_sm, k in rows:
        def time(q):
            waves = -(-(-(-tiles // q) * lanes) // (per_sm * 152))
            return float("inf") if q > 24 and waves > 1 else waves * (q + 0.3)

        assert 1 <= k <= 32 and time(k) <= 1.031 * min(time(q) for q in range(1, 33)), (tiles, lanes, per_sm)
    src = open(os.path.join(CSRC, "wilson.cu")).read()
    assert "dot_tiles(grid.x, nrhs / NR, wilson_threads<S, NR, true>() / NT" in src


def test_coarsest_product_and_dots(tmp_path):
    """Row form: two rows per FP64 CTA where four leave an SM with a fifth more; FP32 above 3,584 rows goes to the tiled
    product with 13.  Overlaps: more blocks only on long vectors and few lanes, at most the partial buffer's."""
    rows = _run(tmp_path, "\n".join("printf(\"%%d\\n\", %s);" % e for e in (
        "matvec_rows_per_cta(2048, 1, 152)", "matvec_rows_per_cta(1216, 1, 152)", "matvec_most(1, 3072)",
        "matvec_most(1, 4096)", "matvec_most(0, 8192)", "multidot_grid(384, 1, 8, 152, 1216)",
        "multidot_grid(98304, 1, 8, 152, 1216)", "multidot_grid(98304, 1, 16, 152, 1216)",
        "multidot_grid(98304, 5, 8, 152, 1216)", "multidot_grid(98304, 12, 8, 152, 1216)", "multidot_grid(1, 1, 8, 152, 1216)")))
    assert [r[0] for r in rows] == [2, 4, 16, 12, 16, 96, 608, 304, 121, 152, 1]

"""What kernels ask the L2 for ahead of the kernel before them: rules that need no device, compiled with the host compiler, and what the
sources must say.  (A request moves no data, so no result shows whether it is the right one.)"""
import os
import re
import subprocess

import pytest

from paper_2605_19561_b200 import torq
from test_pair_handshake import CSRC, _conditions


def _run(tmp_path, body):
    src = tmp_path / "check.cpp"
    src.write_text('#include <cstdio>\n#include "l2_requests.cuh"\nint main() {\n' + body + "\n  return 0;\n}\n")
    exe = str(tmp_path / "check")
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I" + CSRC, str(src), "-o", exe], check=True)
    res = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert res.returncode == 0, res.stdout


def test_the_lanes_of_a_warp_ask_for_all_of_a_matrix_once(tmp_path):
    """Every byte of a B x B bf16 matrix (B a multiple of 8, up to 128) in exactly one lane's share, shares whole 16-byte pieces."""
    _run(tmp_path, r"""
  for (int b = 8; b <= 128; b += 8) {
    const int bytes = 2 * b * b;
    int next = 0;
    for (int lane = 0; lane < 32; ++lane) {
      const int n = torq::lane_share_bytes(lane, bytes);
      if (n < 0 || n % 16 || (n && torq::lane_share_first(lane, bytes) != next)) { std::printf("B %d lane %d\n", b, lane); return 1; }
      next += n;
    }
    if (next != bytes) { std::printf("B %d: %d bytes of %d\n", b, next, bytes); return 1; }
  }
""")


def test_the_structured_rotation_asks_for_r_b_wherever_it_is_one_strip():
    """By the geometry that the comment gives as the reason, not by one width."""
    body = re.sub(r"//.*", "", open(os.path.join(CSRC, "rotate_structured.cuh")).read())
    asks = [m.start() for m in re.finditer(r"prefetch_l2\w*\((?:&tmRB|[^;]*R_B)", body)]
    assert len(asks) == 1
    sizes = {t for t in _conditions(body, asks[0]) if re.search(r"nblocks|b_tiles|k_tiles|\bd\b", t)}
    assert sizes == {"b_tiles == 1", "lane_share_bytes lane, 2 * nblocks * nblocks > 0"}, sizes


@pytest.mark.parametrize("name,tensor,extent", [("rotate_quantize_pair.cuh", "tmX", "M"), ("mxfp4_gemm_wide.cuh", "tmB", "N"),
                                                ("rotate_structured.cuh", "tmX3", "M")])
def test_no_box_that_lies_wholly_outside_its_tensor_is_asked_for(name, tensor, extent):
    """Tiles go on beyond the last token, feature or row of W: a CTA whose part of a tile begins there asks for nothing.  (The one-wave rotation
    does ask, and the L2 then has nothing to fetch: the guard costs its short calls more than the request.)"""
    body = re.sub(r"//.*", "", open(os.path.join(CSRC, name)).read())
    asks = [m.start() for m in re.finditer(r"tma_prefetch_l2_\wd\(&%s," % tensor, body)]
    assert asks
    for at in asks:
        assert any(t.endswith(" < " + extent) for t in _conditions(body, at)), _conditions(body, at)


@pytest.mark.parametrize("M,d", [(1500, 2048), (2048, 4096), (2300, 2048), (3600, 2048), (4096, 2304), (4500, 1792), (8192, 1024), (16384, 512), (2048, 14336)])
def test_pairs_of_one_row_tile_ask_for_its_first_k_steps(M, d, tmp_path):
    """The first wave's tiles: in every row tile each pair asks for another step, and those of wide tiles for the first ones without a gap."""
    tiles = torq.torq_pair_tile_list(M, d, 74)[:74]
    body = re.sub(r"//.*", "", open(os.path.join(CSRC, "rotate_quantize_pair.cuh")).read())
    assert re.search(r"kt = x_step_of_tile\(tcol0, narrow0\);\s+[^}]*tma_prefetch_l2_2d\(&tmX, kt \* ", body)
    rows = "".join("{%d, %d, %d}," % t for t in tiles)
    _run(tmp_path, r"""
  const struct { int mp, col, width; } t[] = {""" + rows + r"""};
  for (const auto& a : t) {
    const int step = torq::x_step_of_tile(a.col, a.width == 192);
    int same = 0, before = 0, wide = 0;
    for (const auto& b : t)
      if (b.mp == a.mp) {
        same += torq::x_step_of_tile(b.col, b.width == 192) == step;
        before += torq::x_step_of_tile(b.col, b.width == 192) < step;
        wide += b.width == 192;
      }
    if (same != 1 || (wide == 0 && before != step)) { std::printf("row tile %d column %d: step %d\n", a.mp, a.col, step); return 1; }
  }
""")

"""What kernels ask the L2 for ahead of the kernel before them: rules that need no device, compiled with the host compiler, and what the
sources must say.  (A request moves no data, so no result shows whether it is the right one.)"""
import os
import re
import subprocess

import pytest

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

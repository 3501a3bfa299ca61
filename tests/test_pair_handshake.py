"""Host-side rules of the CTA-pair kernels, compiled with the host compiler."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_19561_b200", "csrc")


def _run(tmp_path, body):
    src = tmp_path / "check.cpp"
    src.write_text('#include <cstdio>\n#include "pair_handshake.cuh"\nint main() {\n' + body + "\n  return 0;\n}\n")
    exe = str(tmp_path / "check")
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I" + CSRC, str(src), "-o", exe], check=True)
    res = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert res.returncode == 0, res.stdout


def test_every_accumulator_arrival_is_waited_for(tmp_path):
    """A pair's epilogue sends one arrival per tile it announces; its issuer, before the tile that reuses an accumulator, waits
    for the arrival of that accumulator's tile before.  At the end no arrival is left over (it could reach a CTA that has
    exited) and no wait has gone without one (it would run out)."""
    _run(tmp_path, r"""
  for (int accs = 1; accs <= 2; ++accs)
    for (int npairs = 1; npairs <= 9; ++npairs)
      for (int total = 1; total <= 60; ++total)
        for (int pair = 0; pair < npairs && pair < total; ++pair) {
          int sent[2] = {0, 0}, waited[2] = {0, 0}, t = 0;
          for (int tile = pair; tile < total; tile += npairs, ++t) {
            const int a = t % accs;
            if (t >= accs) ++waited[a];
            if (torq::accumulator_is_waited_for(tile, npairs, accs, total)) ++sent[a];
          }
          for (int a = 0; a < accs; ++a)
            if (sent[a] != waited[a]) {
              std::printf("accs %d pairs %d tiles %d pair %d: %d sent, %d waited for\n", accs, npairs, total, pair, sent[a], waited[a]);
              return 1;
            }
        }
""")


def test_paced_wait_ends_whatever_the_clock_does(tmp_path):
    _run(tmp_path, r"""
  long long now = 0;
  int slept = 0;
  auto frozen = [&] { return now; };
  torq::paced_wait(1000, 7, frozen, [&] { ++slept; });
  if (slept != 7) { std::printf("frozen clock: %d\n", slept); return 1; }
  slept = 0;
  torq::paced_wait(1000, 7, frozen, [&] { ++slept; now += 400; });
  if (slept != 3) { std::printf("running clock: %d\n", slept); return 1; }
  slept = 0;
  torq::paced_wait(1000, 7, frozen, [&] { ++slept; });
  if (slept != 0) { std::printf("time already past: %d\n", slept); return 1; }
""")

"""Rules of the kernels that need no device: host-side ones, compiled with the host compiler, and what their sources must say."""
import os
import re
import subprocess

import pytest

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
  // start of the wait, cycles, what a turn adds to the counter: 40 each, 40 over the wrap, a jump back, a jump ahead, no wait
  struct { unsigned since, cycles; int step[4]; int turns; } cases[] = {
      {1000u, 100u, {40, 40, 40, 40}, 3}, {0xFFFFFFF0u, 100u, {40, 40, 40, 40}, 3}, {1000u, 100u, {40, -500, 40, 40}, 2},
      {1000u, 100u, {40, 1000000, 40, 40}, 2}, {1000u, 0u, {40, 40, 40, 40}, 0}};
  for (auto& c : cases) {
    unsigned now = c.since;
    int turns = 0;
    torq::paced_wait(c.since, c.cycles, [&] { return now; }, [&] { now += (unsigned)c.step[turns & 3]; ++turns; });
    if (turns != c.turns) { std::printf("since %u cycles %u: %d turns\\n", c.since, c.cycles, turns); return 1; }
  }
""")


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith(".cuh")
                                        and re.search(r"^  griddep_launch_dependents\(\);", open(os.path.join(CSRC, f)).read(), re.M)))
def test_no_limit_of_a_wait_counts_the_kernel_before(name):
    """A kernel starts while the one before it in the stream still runs, for as long as that takes.  So a role either passes
    griddepcontrol.wait, which has no limit, before its first wait that has one, or the clock of all its waits for what other roles
    bring after that starts behind it."""
    body = re.sub(r"//.*", "", open(os.path.join(CSRC, name)).read())
    body = body[re.search(r"^  griddep_launch_dependents\(\);", body, re.M).start():]
    roles = re.split(r"^  (?:if \(warp == \d+\) \{|\} else if \(warp == \d+\) \{|\} else \{)$", body, flags=re.M)
    before, roles = roles[0], roles[1:]
    assert len(roles) >= 3 and sum("mbar_wait" in r for r in roles) >= 3
    if "griddep_wait();" in before:
        return
    for role in roles:
        first = re.search(r"mbar_wait", role)
        if first is None or "griddep_wait();" in role[:first.start()]:
            continue
        waits = re.findall(r"mbar_wait\w*(<true>)?\((\w+)", role)
        # a wait for a free accumulator passes at once in the first tiles and comes behind their instructions in later ones
        assert waits and all(dep == "<true>" or bar == "acce_bar" for dep, bar in waits), waits
    ptx = open(os.path.join(CSRC, "sm100_ptx.cuh")).read()
    assert re.search(r"if \(BEHIND_DEP && t0 == 0\) griddep_wait\(\);\s+unsigned long long now = globaltimer_ns\(\);\s+if \(t0 == 0\) t0 = now;", ptx)


def test_a_wait_reports_what_it_waits_for():
    """The site that a wait names when it gives up is that of its barrier: one site per kind of barrier, none shared."""
    kinds = {"full_bar": "SITE_MMA_FULL", "empty_bar": "SITE_PRODUCER_EMPTY", "acce_bar": "SITE_MMA_ACC_EMPTY", "accf_bar": "SITE_EPI_ACC_FULL",
             "alloc_bar": "SITE_PEER_TMEM"}
    sites = re.search(r"enum WaitSite : int \{(.*?)\};", open(os.path.join(CSRC, "sm100_ptx.cuh")).read(), re.S).group(1)
    ids = re.findall(r"(SITE_\w+) = (\d+)", sites)
    assert len({i for _, i in ids}) == len(ids) and set(kinds.values()) <= {n for n, _ in ids}
    seen = set()
    for f in os.listdir(CSRC):
        for bar, site in re.findall(r"mbar_wait\w*(?:<true>)?\((\w+_bar)\b[^;{]*?(SITE_\w+)\)", open(os.path.join(CSRC, f)).read()):
            if bar in kinds:
                assert site == kinds[bar], (f, bar, site)
                seen.add(bar)
    assert seen == set(kinds)


def _conditions(body, at):
    """What has to hold for the statement at `at` to run: the conditions of the blocks around it and of its own if / for, their
    && taken apart, flags that are declared once replaced by what they stand for."""
    named = dict(re.findall(r"bool (?:\w+ = [^;]*?, )?(\w+) = ([^;?]*?);", body))
    opens, depth = [], 0
    for m in re.finditer(r"[{}]", body[:at]):
        if m.group() == "{":
            head = body[max(body.rfind(c, 0, m.start()) for c in "{}") + 1:m.start()]
            opens.append(head[head.rfind(";\n") + 1:])
        elif opens:
            opens.pop()
    own = body[max(body.rfind("{\n", 0, at), body.rfind("}\n", 0, at), body.rfind(";\n", 0, at)):at]
    terms = set()
    for text in opens + [own]:
        for cond in re.findall(r"(?:if(?: constexpr)?|for) \((.*)\)", text + ")"):
            for t in re.split(r"&&|;", cond.replace("(", " ").replace(")", " ")):
                t = " ".join(t.split())
                terms |= {" ".join(x.split()) for x in named.get(t, t).split("&&")}
    return terms


@pytest.mark.parametrize("name", ["rotate_quantize_wide.cuh", "rotate_quantize_pair.cuh"])
def test_an_instance_that_does_not_wait_for_r_intra_sends_no_arrival(name):
    """The arrival that tells the leader of the other CTA's R_intra stands behind every condition on the instance and on the arguments
    that the leader's wait for it stands behind: one that nobody waits for could reach a CTA that has exited."""
    body = re.sub(r"//.*", "", open(os.path.join(CSRC, name)).read())
    wait = _conditions(body, re.search(r"mbar_wait\w*(?:<true>)?\(ri_bar", body).start())
    arrive = _conditions(body, re.search(r"mbar_arrive\w*\(map_to_cta\(ri_bar", body).start())
    wanted = {t for t in wait if re.search(r"FMT|RANGE|R_intra|total_tiles", t) and " = " not in t}
    assert any("R_intra" in t for t in wanted) and any(re.search(r"FMT|RANGE", t) for t in wanted), wait
    assert wanted <= arrive, (wanted, arrive)

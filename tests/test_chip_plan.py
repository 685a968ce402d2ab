"""How a batch is dealt to the SMs by the on-chip solve (csrc/emd_chip_plan.cuh, host code): every cell
in one CTA, what a CTA and a gather's planes can hold, and which solves go on chip at all."""

import json
import os
import random
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1808_07284_gb300", "csrc")
CAP = 152

PROBE = r"""
#include <chrono>
#include <cstdio>
#include "emd_chip_plan.cuh"
int main() {  // a request a line: isotropic, SMs, number of gathers, then their (nr, nt)
  int iso, cap, B;
  while (scanf("%d %d %d", &iso, &cap, &B) == 3) {
    std::vector<int> nt(B), nr(B), on;
    for (int b = 0; b < B; ++b) if (scanf("%d %d", &nr[b], &nt[b]) != 2) return 1;
    bool march = false;
    const auto t0 = std::chrono::steady_clock::now();
    const emd::ChipPlan p = emd::choose_on_chip(B, nt.data(), nr.data(), cap, iso != 0, false, on, &march);
    const double ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
    printf("{\"ms\": %f, \"march\": %d, \"on\": [", ms, march);
    for (size_t i = 0; i < on.size(); ++i) printf("%s%d", i ? ", " : "", on[i]);
    printf("], \"waves\": [");
    for (size_t w = 0; w < p.waves.size(); ++w) {
      printf("%s{\"form\": %d, \"jobs\": [", w ? ", " : "", p.form[w]);
      for (size_t i = 0; i < p.waves[w].size(); ++i) {
        const emd::ChipJob &J = p.waves[w][i];
        printf("%s[%d, %d, %d, %d, %d, %d, %d, %d, %d]", i ? ", " : "", J.gather, J.seg, J.strip, J.segs, J.strips, J.i0,
               J.h, J.group, J.rows);
      }
      printf("]}");
    }
    printf("]}\n");
    fflush(stdout);
  }
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "probe.cpp").write_text(PROBE)
    exe = d / "probe"
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", CSRC, str(d / "probe.cpp"), "-o", str(exe)], check=True)

    def run(requests):
        text = "\n".join(" ".join(map(str, [int(iso), CAP, len(sizes)] + [v for s in sizes for v in s]))
                         for iso, sizes in requests)
        out = subprocess.run([str(exe)], input=text, capture_output=True, text=True, check=True).stdout
        return [json.loads(line) for line in out.splitlines()]

    return run


def align256(n):
    return (n + 255) & ~255


def check(sizes, p):
    forms = {0: 128, 1: 128, 2: 385}
    seen = {}
    for wave in p["waves"]:
        assert 0 < len(wave["jobs"]) <= CAP
        assert wave["form"] == 0 if not p["march"] else wave["form"] in (1, 2)
        for gather, seg, strip, segs, strips, i0, h, group, rows in wave["jobs"]:
            nr, nt = sizes[p["on"][gather]]
            assert h + 3 <= rows <= forms[wave["form"]] and group == segs * strips
            assert strips == -(-nt // 120)
            assert h >= (1 if seg == segs - 1 else 2) and i0 + h <= nr
            assert (seg, strip) not in seen.setdefault(gather, {})
            seen[gather][seg, strip] = (i0, h, id(wave), segs, strips, rows, wave["form"])
    assert sorted(seen) == list(range(len(p["on"]))) and p["on"] == sorted(set(p["on"]))
    for gather, jobs in seen.items():
        nr, nt = sizes[p["on"][gather]]
        i0, h, wave, segs, strips, rows, form = jobs[0, 0]
        assert len(jobs) == segs * strips and len({j[2] for j in jobs.values()}) == 1
        for strip in range(strips):
            at = 0
            for seg in range(segs):
                assert jobs[seg, strip][0] == at
                at += jobs[seg, strip][1]
            assert at == nr
        ntp = (nt + 31) // 32 * 32
        need = 16 * ((4 * segs * ntp if segs > 1 else 0) + 4 * strips * nr)
        if form == 2:
            need += 4 * segs * strips * rows * 640
        assert need <= 9 * align256(4 * nr * ntp)


def log_int(rng, lo, hi):
    return round(lo * (hi / lo) ** rng.random())


def test_every_cell_has_one_cta(plan):
    rng = random.Random(5)
    requests = [(rng.random() < 0.5, [(log_int(rng, 1, 3000), log_int(rng, 2, 40000))]) for _ in range(1500)]
    requests += [(False, [(nr, nt)]) for nr in (1, 2, 3, 12, 13, 125, 126, 382, 383) for nt in (2, 120, 121, 18240, 18241)]
    requests += [(rng.random() < 0.5, [(log_int(rng, 1, 1300), log_int(rng, 64, 9000)) for _ in range(rng.randint(2, 40))])
                 for _ in range(200)]
    answers = plan(requests)
    assert len(answers) == len(requests) and sum(1 for a in answers if a["waves"]) > len(requests) // 2
    for (_, sizes), p in zip(requests, answers):
        check(sizes, p)


def test_no_gather_larger_than_the_chip(plan):
    for p in plan([(iso, [s]) for iso in (0, 1) for s in ((9, 156001), (1200, 17000), (5000, 5000))]):
        assert not p["on"] and not p["waves"]


def test_the_isotropic_cost_streams_where_tall_ctas_are_slower(plan):
    """Four gathers of 648 x 8000 with the isotropic cost take 180 us a pass in tall CTAs, one after the
    other, and 172 streamed together; a single one 45 against 54.  The other cost is the faster one on chip
    throughout, and so is this one in lower CTAs."""
    stream = [[(648, 8000)] * 4, [(648, 8000)] * 16]
    chip = [[(648, 8000)], [(1146, 5639)], [(643, 6915)], [(480, 4000)] * 16, [(128, 1000)], [(400, 3000)] * 8]
    for p in plan([(1, s) for s in stream]):
        assert not p["on"]
    for s, p in zip(stream + chip, plan([(0, s) for s in stream + chip])):
        assert len(p["on"]) == len(s)
    for s, p in zip(chip, plan([(1, s) for s in chip])):
        assert len(p["on"]) == len(s)


def first_fit(sizes, p):
    """The gathers of each wave by first fit, the ones of most CTAs first, at the heights of the plan."""
    jobs = {J[0]: J for wave in p["waves"] for J in wave["jobs"]}
    waves = []
    for g in sorted(jobs, key=lambda g: (-jobs[g][7], g)):
        group, rows = jobs[g][7:]
        for w in waves:
            if w["used"] + group <= CAP and w["tall"] == (rows > 128):
                break
        else:
            w = dict(used=0, tall=rows > 128, members=[])
            waves.append(w)
        w["used"] += group
        w["members"].append(g)
    return [w["members"] for w in waves]


def uneven(n, seed):
    rng = random.Random(seed)
    return [(rng.randint(16, 76), rng.randint(600, 2100)) for _ in range(n)]


def test_waves_are_filled_by_first_fit(plan):
    rng = random.Random(9)
    batches = [[(log_int(rng, 9, 1200), log_int(rng, 64, 9000)) for _ in range(rng.randint(2, 60))] for _ in range(150)]
    batches += [uneven(400, 1), [(100, 1500), (643, 6915), (30, 700)] * 50, [(64, 8000)] * 30]
    answers = plan([(0, s) for s in batches])
    assert sum(1 for p in answers if len(p["waves"]) > 3) > 50
    for sizes, p in zip(batches, answers):
        got = []
        for wave in p["waves"]:
            seen = dict.fromkeys(J[0] for J in wave["jobs"])
            got.append(list(seen))
        assert got == first_fit(sizes, p)


def test_a_plan_takes_time_in_proportion_to_the_batch(plan):
    """First fit over every wave for every gather took the square of it: 4 ms for 2000, 240 for 20,000."""
    small, large = uneven(2000, 2), uneven(20000, 3)
    ms = [min(p["ms"] for p in plan([(0, s)] * 3)) for s in (small, large)]
    assert ms[1] < 25.0 * ms[0], ms

"""The distribution of a launch's work units over CTA pairs (gq_pipeline.cuh), compiled for the host: every k-step of every
unit is worked on exactly once, and no unit is accumulated in longer runs than the cut across units gives it, short runs apart.

The second is about accuracy: the tensor core's fp32 accumulation truncates, so that a longer run loses more.
"""
import os
import random
import subprocess

import pytest

from paper_2505_07004_b200 import build as gq_build
from test_gpu_hessian_cut import ACROSS, EVENLY

HERE = os.path.dirname(os.path.abspath(__file__))
PAIRS = 74                       # of a GPU with 148 SMs
SHORT_RUN = 16                   # k-steps (of 64 tokens) up to which a run's truncation does not show


@pytest.fixture(scope="module")
def items(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("schedule") / "items")
    subprocess.check_call([gq_build._nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-o", exe,
                           os.path.join(HERE, "schedule_items.cu")])

    def run(launches):
        text = "".join("%d %d %d %d\n" % launch for launch in launches)
        out = subprocess.run([exe], input=text, stdout=subprocess.PIPE, universal_newlines=True, check=True).stdout
        plans = []
        for line in out.splitlines():
            if line.startswith("plan"):
                plans.append((tuple(int(v) for v in line.split()[1:]), []))
            elif line != "end":
                plans[-1][1].append(tuple(int(v) for v in line.split()))
        assert len(plans) == len(launches)
        return plans
    return run


def launches():
    rng = random.Random(4)
    some = [(rng.randint(1, 300), int(2 ** rng.uniform(0, 9)), PAIRS, rng.randint(0, 3) > 0) for _ in range(600)]
    return [(u, k, p, int(b)) for u, k, p, b in some] + [(u, k, PAIRS, 1) for u in (1, 2, 26, 37, 38, 72, 73, 75) for k in (1, 2, 15, 16, 17, 33, 256)]


def test_every_kstep_once(items):
    for (units, ksteps, pairs, balanced), ((_, tail_units, tail_pairs), work) in zip(launches(), items(launches())):
        done = {}
        for pair, unit, ks0, ks1 in work:
            assert 0 <= pair < pairs and 0 <= unit < units and 0 <= ks0 < ks1 <= ksteps
            done.setdefault(unit, []).append((ks0, ks1))
        assert len(done) == units
        for pieces in done.values():
            pieces.sort()
            assert pieces[0][0] == 0 and pieces[-1][1] == ksteps
            assert all(a[1] == b[0] for a, b in zip(pieces, pieces[1:]))
        assert tail_pairs <= pairs and (balanced or all(len(p) == 1 for p in done.values()))


def test_runs_are_not_longer_than_across_units(items):
    cut = [launch for launch in launches() if launch[3] and launch[0] % PAIRS]
    kinds = set()
    for (units, ksteps, pairs, _), ((full, tail_units, tail_pairs), work) in zip(cut, items(cut)):
        runs = {}
        for _, unit, ks0, ks1 in work:
            if unit >= full * pairs:
                runs.setdefault(unit, []).append(ks1 - ks0)
        longest = max(max(r) for r in runs.values())
        total = tail_units * ksteps
        across = min(max(total // 8, tail_units), pairs)               # pairs that the cut across units takes
        evenly = tail_pairs % tail_units == 0 and tail_pairs != across
        kinds.add(evenly)
        if evenly:
            assert longest <= SHORT_RUN
        else:
            assert longest <= min(ksteps, -(-total // across))
    assert kinds == {True, False}


def hessian_launch(d_in, n, g):
    """(units, k-steps) of a Hessian launch: 256 x 256 tiles on the upper triangle for every two groups, and for an odd last
    group the pairs of neighbouring column tiles by row tile."""
    nj = -(-d_in // 256)
    slots = nj // 2 * (nj // 2 + 1) + (nj if nj % 2 else 0)
    return nj * (nj + 1) // 2 * (g // 2) + (slots if g % 2 else 0), -(-n // 64)


def test_ways_of_the_launches_that_run_on_the_gpu(items):
    """What tests/test_gpu_hessian_cut.py says about its launches."""
    plans = items([hessian_launch(*shape) + (PAIRS, 1) for shape in EVENLY + ACROSS])
    for shape, ((full, tail_units, tail_pairs), work) in zip(EVENLY + ACROSS, plans):
        units, ksteps = hessian_launch(*shape)
        tail = [w for w in work if w[1] >= full * PAIRS]
        of_pair = [len([w for w in tail if w[0] == p]) for p in range(tail_pairs)]
        lengths = {w[3] - w[2] for w in tail}
        if shape in EVENLY:
            assert tail_pairs % tail_units == 0 and set(of_pair) == {1}
        else:
            assert tail_pairs == PAIRS and max(of_pair) == 2 and len(lengths) > 2 and tail_units * ksteps % PAIRS != 0
            assert shape[1] % 64 != 0
    assert {p[0][0] for p in plans} == {0, 1}                         # with and without a whole round before

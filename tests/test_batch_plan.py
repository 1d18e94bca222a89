"""The split of a batched launch of width 0 over CTAs, on the host.

`batch_plan_check.cpp` (beside this file) is compiled against the planner and given batches on
grids of 30 to 9241 buses (their levels and flops) for every compiled CTA shape.  A plan uses
the slots it has: directions that fit half the slots get a CTA each, so no small grid's
block waits in one CTA beside idle SMs; more of them take half of the slots or more, and
no second wave where the caps allow it.
"""
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
N_SM = 152
#        levels, flops, n_x, tail rows
GRIDS = {30: (48, 2432, 53, 16), 118: (84, 10700, 181, 16), 300: (80, 32144, 539, 32), 500: (128, 52068, 899, 32),
         1354: (168, 154120, 2447, 48), 2869: (264, 378760, 5227, 80), 9241: (544, 1456252, 17036, 128)}
PER_SM = {384: 2, 256: 3, 192: 4, 128: 6}


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("g++ not available")
    exe = str(tmp_path_factory.mktemp("plan") / "batch_plan_check")
    subprocess.run([cxx, "-std=c++17", "-O2", "-Wall", "-o", exe, os.path.join(HERE, "batch_plan_check.cpp")], check=True)

    def run(threads, mix):
        rows = [f"{N_SM} {PER_SM[threads]} {int(threads == 384)} {len(mix)}"]
        for grid, n in mix:
            lev, flops, n_x, tail = GRIDS[grid]
            rows.append(f"{lev} {flops} {n} {min(max(n, 1), 256, 4096 // tail)} {n_x} {int(n_x > 1024)}")
        out = subprocess.run([exe], input="\n".join(rows), capture_output=True, text=True, check=True).stdout.split()
        return [(int(g), a == "1") for g, a in zip(out[::2], out[1::2])]
    return run


MIXES = [[(500, 17), (30, 10), (118, 2), (30, 130), (300, 7)], [(30, 150)], [(118, 3), (9241, 1), (30, 60)],
         [(9241, 64)], [(118, 64)] * 8, [(30, 0), (118, 5)], [(1354, 64)] * 8, [(30, 256)] * 16,
         [(118, 40)] * 6 + [(1354, 100)] * 3 + [(2869, 60), (9241, 30)], [(9241, 256)] * 32, [(118, 1)] * 32]
rng = np.random.default_rng(2)
MIXES += [[(int(rng.choice(list(GRIDS))), int(np.exp(rng.uniform(0, np.log(300))))) for _ in range(rng.integers(1, 33))]
          for _ in range(40)]


@pytest.mark.parametrize("threads", list(PER_SM))
def test_plans_use_the_slots(plan, threads):
    slots, half = N_SM * PER_SM[threads], N_SM * (PER_SM[threads] // 2)
    for mix in MIXES:
        p = plan(threads, mix)
        rest = [(grid, n, g) for (grid, n), (g, alone) in zip(mix, p) if not alone]
        cap = {grid: min(256, 4096 // GRIDS[grid][3]) for grid in GRIDS}
        for grid, n, g in rest:
            assert (g == 0) if n == 0 else (1 <= g <= n and -(-n // g) <= cap[grid]), (mix, p)
        n_rest, used = sum(n for _, n, _ in rest), sum(g for _, _, g in rest)
        if sum(-(-n // cap[grid]) for grid, n, _ in rest) <= slots:
            assert used <= slots, (mix, p)
        if n_rest == sum(n for _, n in mix):
            # nothing beside: one each, or half the slots in use (less what whole CTAs leave over)
            assert used == n_rest if n_rest <= half else used > 0.45 * half, (mix, p)
        least = min((GRIDS[grid][2] for (grid, n), (_, a) in zip(mix, p) if a), default=None)
        for (grid, n), (g, alone) in zip(mix, p):
            assert not alone or (threads == 384 and GRIDS[grid][2] > 1024)
            if least is not None and n > 0:
                assert alone == (GRIDS[grid][2] >= least), (mix, p)      # every item of the grids chosen

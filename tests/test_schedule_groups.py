"""The parts of the schedule (host code, csrc/hfx_schedule.h) that the dense pass's ragged rows and the shared
launches of the forward and x passes rely on, through a small probe program:

* with ragged rows, every off-diagonal block pair is the dense pass's, and in the layout with the last block's
  orbitals as rows every pair of such a block pair has a place of its own, row r in couples r b/2 ... r b/2 + b/2 - 1;
* groups are runs of whole batches that cover them in order, hold at most the couples asked for unless a single
  batch takes more, cannot take in the next batch, and the largest is what a transform buffer is sized by."""
import json
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INCLUDE = "/usr/local/cuda/include"


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None or not os.path.isdir(CUDA_INCLUDE):
        pytest.skip("g++ or the CUDA headers are missing")
    exe = str(tmp_path_factory.mktemp("groups") / "probe")
    subprocess.run([gxx, "-std=c++17", "-O1", "-I", CUDA_INCLUDE, os.path.join(ROOT, "tests", "schedule_groups_probe.cpp"),
                    "-o", exe], check=True)
    return lambda *a: json.loads(subprocess.run([exe] + [str(int(x)) for x in a], check=True, capture_output=True).stdout)


@pytest.mark.parametrize("b", [4, 8])
@pytest.mark.parametrize("n_orb", [1, 7, 8, 9, 12, 15, 16, 17, 27, 64, 117])
def test_ragged_rows(probe, b, n_orb):
    nb, last = (n_orb + b - 1) // b, (n_orb - 1) % b + 1
    for ragged in (False, True):
        S = probe(n_orb, b, 10 ** 9, ragged, 0)
        slots = list(zip(S["slot_blocks"][0::2], S["slot_blocks"][1::2]))
        assert sorted(S["dense_slots"] + S["diag_slots"] + S["generic_slots"]) == list(range(len(slots)))
        for k, (I, J) in enumerate(slots):
            full = last == b or J < nb - 1
            assert (k in S["dense_slots"]) == (I != J and (full or ragged))
            assert (k in S["diag_slots"]) == (I == J and full)
            if I != J and not full and ragged:
                places = [j * b + i for j in range(last) for i in range(b)]
                couples = S["slot_couple_base"][k + 1] - S["slot_couple_base"][k]
                assert sorted(places) == list(range(2 * couples))
                for j in range(last):
                    assert {t >> 1 for t in places[j * b:(j + 1) * b]} == set(range(j * b // 2, (j + 1) * b // 2))


@pytest.mark.parametrize("n_orb", [3, 16, 27, 64, 117, 128])
@pytest.mark.parametrize("budget", [40, 200, 10 ** 9])
@pytest.mark.parametrize("limit", [0, 1, 64, 300, 1000, 10 ** 9])
def test_groups(probe, n_orb, budget, limit):
    S = probe(n_orb, 8, budget, True, limit)
    base, first, group = S["slot_couple_base"], S["batch_slot_begin"], S["group_begin"]
    batch = [base[first[b + 1]] - base[first[b]] for b in range(len(first) - 1)]
    assert group[0] == 0 and group[-1] == len(batch) and len(group) == S["ngroups"] + 1
    assert all(a < c for a, c in zip(group, group[1:]))
    size = [sum(batch[a:c]) for a, c in zip(group, group[1:])]
    assert all(s <= limit or c - a == 1 for s, a, c in zip(size, group, group[1:]))
    assert all(s + batch[c] > limit for s, c in zip(size, group[1:-1]))
    assert S["max_group_couples"] == max(size)

"""The host runtime with every launcher of the library (tests/launch_mock.cpp): the sessions of
test_api_host.py on the launch of lone queries and the merged launch of query pairs, and plans
whose boundary slots and unit ranges are where they can go wrong."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import test_api_host as api


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    inc = api._cuda_include()
    if shutil.which("g++") is None or inc is None:
        pytest.skip("no host C++ compiler or CUDA headers")
    path = str(tmp_path_factory.mktemp("launch") / "launch_mock")
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-I", api.CSRC, "-I", inc, "-I",
                    api.HERE, "-x", "c++", os.path.join(api.CSRC, "api.cu"), "-x", "c++",
                    os.path.join(api.CSRC, "cluster_merge.cu"), "-x", "c++",
                    os.path.join(api.HERE, "launch_mock.cpp"), "-o", path], check=True)
    return path


@pytest.mark.parametrize("session", [api.test_score_batch_cells_and_rerun, api.test_allpairs_parts,
                                     api.test_cluster_merge_plain_ranked_and_batched])
def test_sessions_on_every_launcher(exe, session):
    session(exe)


def test_ranked_lists_with_a_run_of_long_subjects(exe):
    """A learned ClusterMerge whose lists, cut by count, put a run of long subjects, many times
    the mean, into one task of a lone query of several passes: its streams are longer than a
    boundary slot and the task runs in pieces."""
    rng = np.random.default_rng(3)
    short, long = (lambda n: rng.integers(40, 60, size=n)), (lambda n: rng.integers(1900, 2000, size=n))
    L = np.concatenate([long(10), short(246), short(206), long(50)])
    H = api.Harness(exe)
    H.add("seqs %d %s" % (len(L), " ".join(map(str, L))), None)
    H.add("sym 1", None)
    H.add("sparse 1", None)
    H.add("tuning 16 256", None)
    H.add("cm 300 338 15 1 0", api._expect_cm(api._oracle_cm(L, 300, 338, 15, 1, 0, True)))
    H.run()


def test_pipelined_tasks_stay_in_one_range(exe):
    """Lists of a few queries of many passes: an equal share of the cost ends inside a task, whose
    passes have to stay with one ticket all the same."""
    rng = np.random.default_rng(8)
    H = api.Harness(exe)
    for k, q in ((1, 9000), (3, 6000), (7, 2000), (40, 700)):
        L = np.concatenate([rng.integers(q, q + 500, size=k), rng.integers(100, 400, size=5)])
        pairs = [(a, int(rng.integers(0, k + 5))) for a in range(k) for _ in range(6)]
        flat = " ".join("%d %d" % p for p in pairs)
        H.add("seqs %d %s" % (len(L), " ".join(map(str, L))), None)
        H.add("sym 0", None)
        H.add("score 0 %d %s" % (len(pairs), flat),
              api._expect_values("score", [api._score(a, b, L, False) for a, b in pairs]))
    H.run()


@pytest.mark.parametrize("lengths", [[300] * 12 + [700] * 9,              # no query pair at 16 warps
                                     list(range(520, 920, 5))])            # a merged launch
def test_autotune_times_the_work_it_counts(exe, lengths):
    """The autotuner runs a plan to warm up and again for the time: both runs launch the same tasks
    and units in the same order, and all of the cells that it divides by the time."""
    out = subprocess.run([exe, "autotune"] + [str(n) for n in lengths], capture_output=True, text=True)
    assert "contract violated" not in out.stderr, out.stderr
    words = out.stdout.split()
    assert words[:6] == ["error", "0", "runs", "24", "differ", "0"], out.stdout
    assert words[7] == words[9], out.stdout


@pytest.mark.parametrize("lengths,huge", [([2200000, 3000, 2300000, 200, 2500], True),
                                          ([2100000, 2100000, 3000], False)])
def test_cells_of_huge_scores_have_their_slots(exe, lengths, huge):
    """Pairs that may score 2^28 take the long pairs of their round to the kernel for such scores,
    whose slots lie behind the boundary columns of the other pairs' strips."""
    out = subprocess.run([exe, "cells"] + [str(n) for n in lengths], capture_output=True, text=True)
    assert "contract violated" not in out.stderr, out.stderr
    words = out.stdout.split()
    assert words[:4] == ["error", "0", "differ", "0"] and (int(words[5]) > 0) == huge, out.stdout

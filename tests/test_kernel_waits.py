"""The rules that keep the give-up path of the kernels with bounded waits from hanging, checked on their source (a kernel
that breaks one of them hangs now and then, which no GPU test should be the first to find)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2411_00850_b200", "csrc")
KERNELS = ("linear_prefill.cu", "linear_skinny.cu")


def _source(name):
    return re.sub(r"//.*", "", open(os.path.join(CSRC, name)).read())


def _kernels(name):
    """The bodies of the file's kernels that look at the status word."""
    return [part for part in re.split(r"__global__", _source(name))[1:] if "no_one_gave_up(p.status)" in part]


@pytest.mark.parametrize("name", KERNELS)
def test_threads_that_meet_go_by_one_read_of_the_status_word(name):
    # other CTAs write the word while this one starts: warps that read it one by one may start with different verdicts,
    # and the one that skips its loop never comes to the others' named barrier
    assert not re.search(r"volatile[^;]*\(\s*p\.status\s*\)", _source(name)), "a read of the status word outside no_one_gave_up()"
    assert len(_kernels(name)) == (2 if name == "linear_prefill.cu" else 1)
    for text in _kernels(name):
        (read,) = re.finditer(r"no_one_gave_up\(p\.status\)", text)
        line = text[text.rindex("\n", 0, read.start()):read.start()]
        if re.search(r"__shfl_sync\(0xFFFFFFFFu, lane == 0 \? \(int\)$", line):   # one verdict per warp
            assert not re.search(r"bar\.(sync|red)", text), "a barrier between warps whose verdicts may differ"
            continue
        assert re.search(r"\btid == \d+ && |if \(tid == \d+ && rank == 0\) go_s = $", line), "read by more than one thread"
        after = text[read.start():]
        store, use = re.search(r"\bgo_s = go;|$", after).start(), re.search(r"bool ok = [^;]*go_s", after).start()
        barrier = after[store if store < use else 0:use]
        assert re.search(r"__syncthreads\(\)|cluster_sync_all\(\)", barrier), "no barrier between the read and its use"


@pytest.mark.parametrize("name", KERNELS)
def test_named_barriers_follow_a_verdict_of_all_their_warps(name):
    text = _source(name)
    for m in re.finditer(r"bar\.sync \d+, 128", text):
        assert "bar.red.and.pred" in text[:m.start()], "a named barrier without a common verdict before it"


@pytest.mark.parametrize("name", KERNELS)
def test_every_wait_for_another_role_has_a_limit(name):
    text = _source(name)
    assert not re.search(r"mbarrier\.(try|test)_wait", text), "waits go through mbar_wait / mbar_wait_warp"


@pytest.mark.parametrize("name", KERNELS)
def test_mmas_and_their_commits_come_from_one_lane(name):
    # a tcgen05.commit tracks the MMAs of the thread that makes it: from another lane it arrives at once, and what waits for it
    # gives tensor memory and shared memory back under MMAs in flight
    for text in _kernels(name):
        lanes = set()
        for call in re.finditer(r"\bumma_(?:f16|ts|commit)\w*\(", text):
            conditions = re.findall(r"if \((?:[^\n]*\W)?(elected|elect_one\(\)|lane == 0)\W", text[:call.start()])
            lanes.add("lane 0" if conditions[-1] == "lane == 0" else "elected")
        assert len(lanes) == 1, "issued by one lane and committed by another"

"""The rules that keep the give-up path of the kernels with bounded waits from hanging, checked on their source (a kernel
that breaks one of them hangs now and then, which no GPU test should be the first to find)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2411_00850_b200", "csrc")
KERNELS = ("linear_prefill.cu", "linear_skinny.cu")


def _source(name):
    return re.sub(r"//.*", "", open(os.path.join(CSRC, name)).read())


@pytest.mark.parametrize("name", KERNELS)
def test_a_cta_goes_by_one_read_of_the_status_word(name):
    # other CTAs write the word while this one starts: warps that read it one by one may start with different verdicts,
    # and the one that skips its loop never comes to the others' named barrier
    text = _source(name)
    assert not re.search(r"volatile[^;]*\(\s*p\.status\s*\)", text), "a read of the status word outside no_one_gave_up()"
    reads = list(re.finditer(r"no_one_gave_up\(p\.status\)", text))
    assert reads
    for m in reads:
        line = text[text.rindex("\n", 0, m.start()):m.start()]
        assert re.search(r"\btid == \d+ && |if \(tid == \d+ && rank == 0\) go_s = $", line), "read by more than one thread"
        after = text[m.start():]
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

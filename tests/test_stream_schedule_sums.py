"""The persistent streamed kernel's order of work with its two buffers of coupled sums
(csrc/dk_stream.cu: fine step m works on buffer (m / 4) % 2, coarse step cn reads
buffer cn % 2): the dependencies of tests/test_stream_schedule.py give every read
what the sequential order writes; a coarse step that reads the other buffer, and
fine steps that do not wait for coarse steps at all, are caught."""
import importlib.util
import os

import pytest

_spec = importlib.util.spec_from_file_location(
    "stream_schedule", os.path.join(os.path.dirname(__file__), "test_stream_schedule.py"))
ref = importlib.util.module_from_spec(_spec)
_spec.loader.exec_module(ref)
_one_buffer = ref.reads_writes


def _two_buffers(it, n, coupled, swap=0):
    kind, m = it[0], it[4]
    buf = (m >> 2) & 1 if kind == 0 else (m + swap) & 1
    R, W = _one_buffer(it, n, coupled)

    def key(x):
        return ("z", buf) + x[1:] if x[0] == "z" else x

    return {key(x) for x in R}, {key(x) for x in W}


@pytest.mark.parametrize("n,count,M,ctas", [(64, 2, 16, 3), (128, 1, 12, 5)])
def test_two_buffers_of_sums(monkeypatch, n, count, M, ctas):
    monkeypatch.setattr(ref, "reads_writes", _two_buffers)
    for seed in range(2):
        assert ref.run_schedule(n, count, M, True, ctas, seed) > 0


def test_reading_the_other_buffer_is_caught():
    """In the sequential order itself: no coarse step finds the sums of its own four
    fine steps in the other buffer."""
    its, *_ = ref.items(128, 1, 16, True)
    for swap, right in ((0, True), (1, False)):
        version = {}
        for it in its:
            R, W = _two_buffers(it, 128, True, swap)
            if it[0] == 1:
                steps = {version.get(x, -1) for x in R if x[0] == "z"}
                assert (steps == {4 * it[4] + 3}) == right
            version.update({x: it[4] for x in W if it[0] == 0})


def _unordered(drop):
    """Pairs (coarse step, later fine step) of which the fine one overwrites sums that
    the coarse one reads and does not depend on it, directly or through other items."""
    its, tr, tc, ct = ref.items(128, 1, 16, True)
    index = {it: k for k, it in enumerate(its)}
    before = []
    for it in its:
        anc = set()
        for kind, s, i, j, target in ref.deps(it, True, tr, tc, ct, drop):
            if target > 0:
                k = index[(0 if kind == "f" else 1, s, i, j, target - 1)]
                anc |= before[k] | {k}
        before.append(anc)
    rws = [_two_buffers(it, 128, True) for it in its]
    bad = 0
    for k, it in enumerate(its):
        if it[0] == 0 and it[4] >= 4 and it[4] % 4 == 0:
            sums = {x for x in rws[k][1] if x[0] == "z"}
            bad += sum(its[c][0] == 1 and c not in before[k] and bool(sums & rws[c][0]) for c in range(k))
    return bad


def test_fine_steps_must_wait_for_coarse_steps():
    assert _unordered(None) == 0
    assert _unordered("coarse_of_fine") > 0

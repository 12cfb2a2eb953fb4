"""The hand-over protocols of the kernels, run by CPU threads (tests/handover_mock.cpp) over the kernels' own word arithmetic
(csrc/handover.h).

Words carry the number of the call that wrote them, taken from a counter to which every call adds 1 << 16 in all, so small batches,
CTA pairs with adapters and CTA pairs without take turns on one workspace and nothing is cleared.  A bounded wait that runs out
(one writer is withheld) sets the time-out bit, every CTA still leaves, and the call costs one time-out, not one for every
word; after the reset the interface asks for the next call is clean.  Nothing here touches a GPU."""
import os
import re
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2410_09615_b200", "csrc")
TIMEOUT_BIT = 1 << 7
LINE = re.compile(r"call (\d+) kind (\d) status (\d+) number (\d+) departures (\d+) wrong (\d+) expired (\d+)")


@pytest.fixture(scope="module")
def mock(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("mock") / "handover_mock")
    subprocess.run(["g++", "-O2", "-std=c++17", "-Wall", "-Werror", "-pthread", os.path.join(HERE, "handover_mock.cpp"), "-o", exe], check=True)
    return exe


def run(exe, *args):
    out = subprocess.run([exe, *[str(a) for a in args]], check=True, capture_output=True, text=True, timeout=120).stdout.splitlines()
    return [tuple(int(x) for x in LINE.match(l).groups()) for l in out if l.startswith("call")], out


def test_shares_cover_the_list_and_their_words_never_meet(mock):
    _, out = run(mock, "shares")
    assert out[0].startswith("shares ")


@pytest.mark.parametrize("ctas,makers,words,pairs,t_pairs,tiles,stages", [
    (2, 1, 5, 1, 1, 1, 1),
    (8, 3, 40, 6, 5, 4, 7),           # parts of tiles and whole tiles in one list
    (12, 4, 16, 8, 8, 2, 27),         # every tile in four parts
    (5, 2, 90, 4, 2, 6, 3),           # whole tiles only
    (9, 1, 33, 7, 7, 3, 5),           # parts that end and start inside tiles
])
def test_kernels_take_turns_on_one_workspace(mock, ctas, makers, words, pairs, t_pairs, tiles, stages):
    rows, _ = run(mock, ctas, makers, words, pairs, t_pairs, tiles, stages, 24, 0, 1 << 26)
    assert len(rows) == 24
    for k, (call, kind, status, number, departures, wrong, expired) in enumerate(rows, 1):
        assert call == k and number == k and status == 0
        assert departures == k << 16              # whatever the kind and the number of CTAs
        assert wrong == 0 and expired == 0        # every word and sum fetched was this call's


@pytest.mark.parametrize("withhold", [1, 2, 4, 5])
def test_a_wait_that_runs_out_costs_one_time_out_and_nobody_stays_behind(mock, withhold):
    ctas, makers, words, pairs = 6, 2, 64, 4
    rows, out = run(mock, ctas, makers, words, pairs, 4, 3, 5, 9, withhold, 20000)
    assert len(rows) == 9
    since = 0
    for call, kind, status, number, departures, wrong, expired in rows:
        since += 1
        assert departures == since << 16 and number == since                # every CTA left, also from the broken call
        if call == withhold:
            assert status & TIMEOUT_BIT and wrong > 0
            # small batches: CTAs that wait at the same time may run out together, but none twice (32 words are missing);
            # pairs: once a CTA
            assert 1 <= expired <= (ctas - makers if kind == 0 else 2 * pairs)
            at = next(i for i, l in enumerate(out) if l.startswith(f"call {call} "))
            assert out[at + 1] == "reset"
            since = 0                                                       # counted from the reset
        else:
            assert status == 0 and wrong == 0 and expired == 0


def test_every_wait_of_the_small_batch_kernel_can_be_ended_by_another():
    """The loops of its waits ask, now and then, whether the call has been given up (its CTAs would else each wait their full time
    for every step of a T that never comes)."""
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "fwd_small.cu")).read())
    for wait in ("mbar_wait", "wait_words"):
        body = text[text.index(f"bool {wait}("):]
        assert "give_up(" in body[:body.index("\n}\n")], wait
    give_up = text[text.index("bool give_up("):]
    give_up = give_up[:give_up.index("\n}\n")]
    assert "is_of(ld_gpu64(sync + 1), call)" in give_up and "st_gpu64(sync + 1" in give_up

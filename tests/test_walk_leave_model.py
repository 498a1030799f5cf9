"""How a multi-step launch leaves its barrier and unit words (walk_common.cuh,
walk_leave), checked on a model: CTAs arrive at K - 1 bounded barriers, one
whose wait runs out arrives at no further one, every CTA counts itself out and
the last to leave zeroes the words.  Whatever the interleaving and whoever's
wait runs out, the words are zero when the launch ends, no CTA passes a
barrier that another has not reached, and no CTA arrives after the zeroing, so
a launch queued behind a failed one starts clean."""
import random

import pytest


def _launch(rnd, words, ctas, barriers, patience, count_failed=True):
    """One launch over words = [arrivals, left]; returns the number of waits that ran out."""
    step = [0] * ctas    # barriers passed
    polls = [None] * ctas  # polls left of the current wait
    state = ["run"] * ctas
    failed = 0
    zeroed = False
    while any(s != "gone" for s in state):
        c = rnd.choice([i for i in range(ctas) if state[i] != "gone"])
        if state[c] == "run":
            if step[c] == barriers:
                state[c] = "leave"
            else:
                assert not zeroed, "arrival after the words were zeroed"
                words[0] += 1
                polls[c] = patience
                state[c] = "wait"
        elif state[c] == "wait":
            if words[0] >= (step[c] + 1) * ctas:
                assert all(step[i] + (state[i] != "run") > step[c] or step[i] > step[c] for i in range(ctas)), \
                    "passed a barrier early"
                step[c] += 1
                state[c] = "run"
            elif polls[c] == 0:
                failed += 1
                state[c] = "leave" if count_failed else "gone"
            else:
                polls[c] -= 1
        else:
            words[1] += 1
            if words[1] == ctas:
                words[0] = words[1] = 0
                zeroed = True
            state[c] = "gone"
    return failed


@pytest.mark.parametrize("patience", [0, 1, 3, 10 ** 9])
@pytest.mark.parametrize("ctas", [1, 2, 5])
def test_words_are_zero_after_every_launch(ctas, patience):
    ran_out = 0
    for seed in range(300):
        rnd = random.Random(seed)
        words = [0, 0]
        for _ in range(3):  # launches one behind the other
            ran_out += _launch(rnd, words, ctas, barriers=rnd.randrange(5), patience=patience) > 0
            assert words == [0, 0]
    assert (ran_out > 0) == (ctas > 1 and patience < 10 ** 9)


def test_a_failed_cta_that_is_not_counted_leaves_them_set():
    with pytest.raises(AssertionError):
        for seed in range(300):
            rnd = random.Random(seed)
            words = [0, 0]
            for _ in range(3):
                _launch(rnd, words, 5, barriers=3, patience=3, count_failed=False)
                assert words == [0, 0]

"""Which form a search takes, one warp per query or a team of warps: the choice
needs no GPU."""
import random

import pytest

from tests import forms

U8, I8, F32 = 0, 1, 2
PQ_F32, PQ_BF16, EXACT, PQ_Q8 = 0, 1, 2, 3
LIMIT = 227 * 1024


def test_every_choice_fits_in_shared_memory():
    # over what a search accepts; where the one-warp form itself is refused,
    # nothing is chosen in its place
    rng = random.Random(1)
    seen = set()
    for _ in range(60_000):
        mode, dtype = rng.randrange(4), rng.randrange(3)
        d = rng.randint(1, 512)
        M = rng.randint(1, min(128, d))
        k = rng.choice([1, 10, 32, 33, 100, 256])
        L = rng.randint(k, 1024)
        form, size = forms.choice(dtype, rng.choice([100, 50_000, 2**30]), d, M, rng.randint(1, 128), mode,
                                  rng.randint(10, 20), L, k, rng.choice([1, 150, 400, 900, 1300, 10_000, 10**6]),
                                  rng.randrange(2), rng.randrange(2), rng.randrange(2), rng.choice([132, 148, 152]))
        assert form in (1, 3, 4)
        assert size <= LIMIT or form == 1
        seen.add((mode, form))
    assert len(seen) == 12


@pytest.mark.parametrize("case,want", [
    # (element type, n, d, M, R, mode, filter, L, k, queries, over the link): the fastest one measured
    ((U8, 10**6, 128, 32, 64, PQ_F32, 16, 224, 10, 10_000, 0), 4),
    ((U8, 10**6, 128, 32, 64, PQ_F32, 16, 64, 10, 1, 0), 4),
    ((U8, 10**6, 128, 32, 64, EXACT, 16, 48, 10, 10_000, 0), 1),
    ((U8, 10**6, 128, 32, 64, PQ_Q8, 15, 160, 10, 10_000, 1), 1),
    ((F32, 300_000, 96, 48, 68, PQ_F32, 16, 128, 10, 3_000, 0), 4),
    ((U8, 100_000, 130, 32, 64, EXACT, 16, 150, 10, 1_200, 0), 1),       # registers hold five, shared memory 20
    ((U8, 100_000, 128, 32, 64, PQ_Q8, 17, 150, 10, 1_200, 0), 1),       # one warp holds all of them at once
    ((I8, 19_000, 100, 50, 68, PQ_Q8, 16, 142, 40, 1_343, 0), 1),
    ((F32, 100_000, 128, 32, 68, EXACT, 15, 66, 40, 1_148, 1), 1),       # rows over the host link
    ((F32, 100_000, 200, 50, 64, EXACT, 16, 64, 10, 600, 1), 1),
    ((U8, 100_000, 128, 32, 64, EXACT, 16, 32, 10, 600, 1), 1),
    ((U8, 17_000, 128, 32, 64, EXACT, 16, 366, 40, 1_233, 1), 3),
])
def test_measured_choices(case, want):
    *shape, link = case
    assert forms.choice(*shape, link)[0] == want


def test_server_choices():
    # the form of every launch alike: fitted to a full GPU, not to the launch
    shape = (U8, 10**6, 128, 32, 64)
    assert forms.choice(*shape, PQ_BF16, 16, 256, 10, 1, 0, 1, 1)[0] == 4
    assert forms.choice(*shape, PQ_Q8, 15, 160, 10, 1, 0, 1, 1)[0] == 1
    assert forms.choice(F32, 5_000, 96, 96, 32, PQ_F32, 20, 80, 10, 20, 0, 1, 1)[0] == 1

"""GPU parity at the sizes where a dispatch changes its path: every count is
compared bit by bit with the CPU oracle."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fb():
    from paper_0905_2203_gb300 import build as b
    b.build()
    from paper_0905_2203_gb300 import binding
    return binding


@pytest.fixture(scope="module")
def ctx(fb):
    c = fb.Context(0)
    yield c
    c.close()


@pytest.fixture(scope="module")
def mid():
    return synth.c2_mid()


def oracle_counts(ty, tm, offs, ct, lo, hi):
    c, _ = oracle.count_many(ty, tm, offs, ct, lo, hi)
    return c.astype(np.int64)


@pytest.mark.parametrize("device", [False, True])
@pytest.mark.parametrize("wide", [1, 15, 100])
def test_few_episodes_over_a_long_recording(fb, ctx, mid, wide, device):
    """At most 256 episodes over more than 2^20 events: segments while spans
    are narrow (wide 1), segments with the overflowing episodes recounted
    grid-wide (15: about 12 events of a type in the longest span), grid-wide
    at once (100)."""
    import torch
    s, cfg = mid
    st = ctx.load_stream(s.types, s.times, s.n_types)
    bins = [(a * wide, b * wide) for a, b in cfg["bins"]]
    offs, ct, lo, hi = synth.random_candidates(0xFE0200 + wide, 40, s.n_types, 1, 6, bins, s.chains, 0.5)
    want = oracle_counts(s.types, s.times, offs, ct, lo, hi)
    args = (offs, ct, lo, hi)
    if device:
        args = tuple(torch.from_numpy(a.view(np.int16) if a.dtype == np.uint16 else a).cuda() for a in args)
        torch.cuda.synchronize()
    got = ctx.count_episodes(st, fb.Cands(*args)).astype(np.int64)
    assert np.array_equal(got, want), np.nonzero(got != want)[0][:5]
    assert want.max() > 0
    st.free()

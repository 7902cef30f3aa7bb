"""Bounded device waits that give up: a team of a tensor-core conversion ends
together, whether all of its threads give up or one does, and after about a second at
the path's own limit.
"""
import numpy as np
import pytest

from test_gpu_parity import g  # noqa: F401


@pytest.fixture()
def ctx(g):
    c = g.Context(g.Params(12, 4, 4, 4, 54, 55, 64), device=True)
    yield c
    c.close()


@pytest.mark.gpu
@pytest.mark.parametrize("partial", [False, True])
@pytest.mark.parametrize("tries", [1, 1000, 1 << 16])
def test_team_ends_together(g, ctx, tries, partial):
    passes, _ = g.he_probe_wait(ctx, tries, partial)
    # the third tile is lost; nobody begins the fourth, and nobody stays behind
    if tries > 1:
        assert np.array_equal(passes, np.full(256, 3)), passes
    else:  # a wait of one try may be lost earlier
        assert passes.min() == passes.max() <= 3, passes


@pytest.mark.gpu
def test_limit_is_short(g, ctx):
    passes, ms = g.he_probe_wait(ctx, 1 << 18, False)
    assert np.array_equal(passes, np.full(256, 3))
    assert 500 < ms < 4_000, ms


@pytest.mark.gpu
def test_bad_arguments(g, ctx):
    for tries in (0, -1, (1 << 18) + 1):
        with pytest.raises(g.HeError):
            g.he_probe_wait(ctx, tries, False)

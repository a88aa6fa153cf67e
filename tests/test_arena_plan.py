"""Rigs' arenas from fvv_query_arena alone (no GPU needed): the coarse hull reads the
table of the first camera's pixels whatever its images' size (Sec. II-B-1), so every
rig that is accepted has one; and silhouettes are refused by the size of their rows
of words, not by that of their blocked copy."""
import dataclasses

import numpy as np
import pytest

from synth import make_rig


@pytest.fixture(scope="module")
def fvv():
    from paper_1903_11785_gb300.build import build
    build()
    from paper_1903_11785_gb300 import fvv as mod
    return mod


def _sized(n, sides):
    """A rig of n cameras with images of these sides (the rest of "tiny")."""
    rig = make_rig("tiny")
    side = np.asarray([sides[k % len(sides)] for k in range(n)], np.int32)
    return dataclasses.replace(rig, P=rig.P[:n], centre=rig.centre[:n], width=side, height=side)


def _shared(fvv, rig):
    """Bytes of the arena that are not a slot's."""
    p = fvv.make_params(rig)
    one, two = (fvv.fvv_query_arena(fvv.make_desc(rig, max_slots=k, host_staging=0), p) for k in (1, 2))
    return 2 * one - two


@pytest.mark.parametrize("n,sides", [(1, (65535,)), (1, (65505,)), (1, (65504,)), (3, (65535, 64)), (3, (64, 65535))])
def test_every_rig_has_its_coarse_table(fvv, n, sides):
    rig = _sized(n, sides)
    assert _shared(fvv, rig) == _shared(fvv, _sized(n, (64,)))
    dims = np.ceil((np.asarray(rig.vol_max) - np.asarray(rig.vol_min)) / rig.coarse_m - 1e-6)
    assert _shared(fvv, rig) >= 4 * n * int(dims.prod())


def test_silhouettes_up_to_their_rows_words(fvv):
    ask = lambda n: fvv.fvv_query_arena(fvv.make_desc(_many(n), 1, 0), fvv.make_params(_many(n)))  # noqa: E731
    rig = make_rig("tiny")

    def _many(n):
        k = [i % rig.n_cams for i in range(n)]
        return dataclasses.replace(rig, P=rig.P[k], centre=rig.centre[k], width=np.full(n, 65535, np.int32),
                                   height=np.full(n, 65535, np.int32))

    # 32 cameras: 32 x 65535 x 2048 words, less than 2^32, and as many tiles of 32 x 32 pixels as make 2^32 words
    assert ask(32) > 4 * (32 * 65535 * 2048 + (1 << 32))
    with pytest.raises(Exception, match="silhouettes too large"):
        ask(33)

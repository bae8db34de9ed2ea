"""Extents in every form the binding takes, and extents that change between calls (no GPU needed)."""
import numpy as np
import torch

import paper_1901_07294_gb300 as wd

WANT = wd.field_bytes((8, 8, 8, 8), wd.SITES_FULL, wd.F32)


def test_extents_are_read_at_each_call():
    """An extent held in a tensor or array may be changed in place between two calls."""
    for make in (torch.tensor, np.array):
        for form in (list, tuple):
            d = form(make(8) for _ in range(4))
            assert wd.field_bytes(d, wd.SITES_FULL, wd.F32) == WANT
            d[3][...] = 16
            assert wd.field_bytes(d, wd.SITES_FULL, wd.F32) == 2 * WANT


def test_extents_of_any_integer_like_type():
    for d in ((8, 8, 8, 8), [8] * 4, "8888", np.full(4, 8), torch.full((4,), 8), [np.array(8)] * 4, [np.array([8])[0]] * 4,
              [8.0, 8, True * 8, np.int16(8)], iter([8, 8, 8, 8])):
        assert wd.field_bytes(d, wd.SITES_FULL, wd.F32) == WANT

"""GPU parity at the sizes where a kernel's tiles, remainders and dispatch lines lie, against the
float64 oracle on the same bytes (tolerances: tests/harness.py)."""
from dataclasses import replace

import numpy as np
import pytest
import torch

from oracle import elitekv_oracle as O
from paper_2503_01586_b200 import inputs as gen

from . import harness as H

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ek():
    from paper_2503_01586_b200 import binding
    binding.lib()
    return binding


@pytest.mark.parametrize("n_items", [1, 4, 5, 16, 17, 33])
def test_combine_items_per_sequence(ek, n_items):
    """The combine holds 16 items' statistics in half a warp and 4 partial results in flight: one
    sequence of n_items one-tile items (the two-pass kernel's tile is 128 tokens), and a second row
    in the same warp with fewer."""
    w = gen.shrink(gen.LLAMA7B_75, B=2, ctx=128 * n_items)
    st = H.setup(w, lens=[128 * n_items, 65], decode_kernel=2)
    _, tile, n_workers, max_items, overhead = ek.elitekv_decode_plan_info(st.layer, st.cache, 2)
    _, first, _ = ek.elitekv_plan_workers(st.lens_dev, tile, n_workers, max_items, overhead)
    assert first.tolist() == [0, n_items, n_items + 1]
    H.check_parity(st, H.run_decode(st), H.sample_units(st, 24, seed=n_items))

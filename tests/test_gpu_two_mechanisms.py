"""Handles side by side: a mechanism loaded (and used) after a larger one leaves the larger
one's kernels the shared memory they need, and both give the results they give alone."""
import copy

import numpy as np
import pytest
import torch

from gpu_util import library, to_dev
from paper_2508_16105_gb300 import autograd, rde_chem, synth

pytestmark = pytest.mark.gpu


def step(m, cells):
    lnA, E = rde_chem.rde_mech_get_arrhenius(m.handle, m.R)
    p = to_dev(cells.p)
    args = [to_dev(x).requires_grad_(True) for x in (cells.T, cells.Y, lnA, E)]
    T, Y, status = autograd.chem_step(m, 1e-9, p, *args)
    g = torch.autograd.grad((T, Y), args, (torch.full_like(T, 1e-3), torch.ones_like(Y)))
    assert (status == 0).all()
    return [x.detach().cpu().numpy() for x in (T, Y) + tuple(g)]


def smaller(mech, n):
    m = copy.deepcopy(mech)
    m.reactions = m.reactions[:n]
    return m


@pytest.mark.parametrize("kind", ["block", "generic"])
def test_a_smaller_mechanism_loaded_later(kind):
    library()
    if kind == "block":
        big, flags = synth.large_mechanism(16105), 0
        small = smaller(big, 100)
    else:
        big, flags = synth.h2_air_mechanism(16105), rde_chem.RDE_LOAD_GENERIC
        small = smaller(big, 12)
    cells = synth.field_cells(big, 24, seed=46)
    a = rde_chem.Mechanism(big.to_text(), rtol=1e-5, flags=flags)
    alone = step(a, cells)
    b = rde_chem.Mechanism(small.to_text(), rtol=1e-5, flags=flags)
    first = step(b, cells)
    again = step(a, cells)
    after = step(b, cells)
    a.close()
    b.close()
    for x, y in zip(alone + first, again + after):
        assert np.array_equal(x, y)

"""Adjoint of cells whose species take no part in a third body ([M] exactly zero)."""
import copy

import numpy as np
import pytest
import torch

from gpu_util import library, to_dev
from paper_2508_16105_gb300 import autograd, rde_chem, synth

pytestmark = pytest.mark.gpu


def test_gradients_are_finite_without_a_third_body(h2mech):
    library()
    mech = copy.deepcopy(h2mech)
    rx = next(r for r in mech.reactions if r.kind == "THREEBODY")
    rx.eff = dict(rx.eff, N2=0.0, O2=0.0)
    cells = synth.uniform_cells(mech, 64, seed=43)
    n2, o2 = mech.index("N2"), mech.index("O2")
    cells.Y[:, :8] = 0.0
    cells.Y[n2, :8] = np.linspace(1.0, 0.65, 8)     # the first cell is pure N2
    cells.Y[o2, :8] = 1.0 - cells.Y[n2, :8]
    cells.T[:8] = np.linspace(600.0, 1300.0, 8)
    out = []
    for flags in (rde_chem.RDE_LOAD_REQUIRE_SPECIALIZED, rde_chem.RDE_LOAD_GENERIC):
        m = rde_chem.Mechanism(mech.to_text(), rtol=1e-7, flags=flags)
        lnA, E = rde_chem.rde_mech_get_arrhenius(m.handle, m.R)
        p = to_dev(cells.p)
        args = [to_dev(x).requires_grad_(True) for x in (cells.T, cells.Y, lnA, E)]
        T, Y, status = autograd.chem_step(m, 1e-9, p, *args)
        g = torch.autograd.grad((T, Y), args, (torch.full_like(T, 1e-3), torch.ones_like(Y)))
        assert (status == 0).all()
        out.append([x.cpu().numpy() for x in g])
        m.close()
    for s, q in zip(*out):
        assert np.isfinite(s).all() and np.isfinite(q).all()
    # nothing of note reacts in the first cells, whose few steps differ by rounding only:
    # 10^3 rounded terms a step, 10^3 2^-53 < 2e-13, leaving a factor of 500 for the steps
    for k in (0, 1):
        a, b = out[0][k][..., :8], out[1][k][..., :8]
        assert np.abs(a - b).max() <= 1e-10 * np.abs(b).max()

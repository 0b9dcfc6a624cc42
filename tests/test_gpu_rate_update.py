"""rde_mech_set_arrhenius after loading parameters outside the fixed-point format: the step
and its adjoint equal those of a handle loaded with the final parameters, bit for bit."""
import copy

import numpy as np
import pytest
import torch

from gpu_util import assert_parity, library, run_oracle, to_dev
from paper_2508_16105_gb300 import autograd, rde_chem, synth

pytestmark = pytest.mark.gpu


def test_parameters_come_back_into_the_format(h2mech):
    library()
    wild = copy.deepcopy(h2mech)
    wild.reactions[4].A, wild.reactions[4].E = 1e17, 900.0
    cells = synth.uniform_cells(h2mech, 96, seed=41)
    out = []
    for text in (h2mech.to_text(), wild.to_text()):
        m = rde_chem.Mechanism(text, rtol=1e-7, flags=rde_chem.RDE_LOAD_REQUIRE_SPECIALIZED)
        if not out:
            lnA, E = rde_chem.rde_mech_get_arrhenius(m.handle, m.R)
            lnA, E = torch.as_tensor(lnA.copy()), torch.as_tensor(E.copy())
        p, T, Y = to_dev(cells.p), to_dev(cells.T), to_dev(cells.Y)
        args = [x.clone().requires_grad_(True) for x in (T, Y, lnA.cuda(), E.cuda())]
        Tn, Yn, status = autograd.chem_step(m, 1e-9, p, *args)
        g = torch.autograd.grad((Tn, Yn), args, (torch.ones_like(Tn), torch.ones_like(Yn)))
        out.append([x.detach().cpu().numpy() for x in (Tn, Yn, status) + tuple(g)])
        m.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
    o = run_oracle(h2mech, cells, 1e-9, rtol=1e-7)
    assert_parity(dict(T=out[1][0], Y=out[1][1], status=out[1][2]), o)

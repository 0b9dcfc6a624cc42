"""The CTA-per-cell kernel on a mechanism with more distinct gather coefficients than a term
of its plan counts in one page."""
import numpy as np
import pytest

from gpu_util import assert_parity, run_gpu, run_oracle
from paper_2508_16105_gb300 import rde_chem, synth
from test_host_kernels import many_efficiencies

pytestmark = pytest.mark.gpu


def test_more_coefficients_than_a_page():
    mech = many_efficiencies(1300)
    for x in mech.reactions:
        x.A *= 1e5
    cells = synth.field_cells(mech, 8, seed=45, fractions=(0.2, 0.4, 0.4))
    cells.Y[:] += 0.01
    cells.Y /= cells.Y.sum(axis=0, keepdims=True)
    g = run_gpu(mech, cells, 1e-8, schedule=rde_chem.RDE_SCHED_BLOCK)
    o = run_oracle(mech, cells, 1e-8)
    assert (o["status"] == 0).all() and np.abs(o["Y"] - cells.Y).max() > 1e-4
    assert_parity(g, o)
    assert abs(int(g["n_acc"].sum()) - int(o["n_acc"].sum())) <= 8

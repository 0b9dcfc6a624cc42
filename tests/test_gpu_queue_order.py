"""The library's own queue order, on block tables and in graphs: a cell's result is the same
bits in any order, on either queue kernel, and a graph keeps the order buffer it was made with."""
import numpy as np
import pytest
import torch

from gpu_util import library, to_dev
from paper_2508_16105_gb300 import rde_chem, synth

pytestmark = pytest.mark.gpu

DT, RTOL = 5e-10, 1e-5


def mechanism():
    library()
    mech = synth.h2_air_mechanism(16105)
    return mech, rde_chem.Mechanism(mech.to_text(), rtol=RTOL, flags=rde_chem.RDE_LOAD_REQUIRE_SPECIALIZED)


def blocks_of(cells, sizes, pad):
    """Blocks of the given sizes with padded leading dimensions; every third hint is set."""
    keep, table, at = [], [], 0
    for s in sizes:
        c = slice(at, at + s)
        Y = torch.zeros(cells.Y.shape[0], s + pad, dtype=torch.float64, device="cuda")
        Y[:, :s] = to_dev(cells.Y[:, c])
        hint = np.zeros(s)
        hint[::3] = DT / (1 + np.arange(len(hint[::3])) % 50)
        b = dict(p=to_dev(cells.p[c]), T=to_dev(cells.T[c]), Y=Y, h_hint=to_dev(hint),
                 status=torch.full((s,), -1, dtype=torch.int32, device="cuda"),
                 n_acc=torch.zeros(s, dtype=torch.int32, device="cuda"))
        keep.append(b)
        table.append(rde_chem.make_block(n=s, ldY=s + pad, **b))
        at += s
    return keep, torch.frombuffer(bytearray(rde_chem.block_table_bytes(table)), dtype=torch.uint8).cuda(), at


def gather(keep, sizes):
    get = lambda k: torch.cat([b[k][..., :s] for b, s in zip(keep, sizes)], -1).cpu().numpy()
    return {k: get(k) for k in ("T", "Y", "h_hint", "status", "n_acc")}


@pytest.mark.parametrize("threads", [0, 128, 256])
@pytest.mark.parametrize("sizes", [[40, 0, 1, 333, 7], [3000, 0, 1, 11000, 7, 6500]])
def test_block_table_in_any_order(threads, sizes):
    """Above 152 x 128 cells the library orders the queue itself (dt / h_hint or T^2 p)."""
    mech, m = mechanism()
    n = sum(sizes)
    cells = synth.field_cells(mech, n, seed=47, fractions=(0.4, 0.3, 0.3))
    out = []
    for order in (None, to_dev(np.arange(n), dtype=torch.int64)):
        keep, table, total = blocks_of(cells, sizes, 5)
        rde_chem.rde_chem_advance_ex(m.handle, DT, blocks=table, n_blocks=len(sizes), n_total=total, order=order,
                                     threads_per_cta=threads)
        torch.cuda.synchronize()
        assert all((b["Y"][:, s:] == 0).all() for b, s in zip(keep, sizes))
        out.append(gather(keep, sizes))
    # the same cells as one block on the 128-thread kernel
    keep, table, total = blocks_of(cells, [n], 0)
    b = keep[0]
    hint = np.concatenate([h["h_hint"].cpu().numpy() for h in blocks_of(cells, sizes, 5)[0]])
    b["h_hint"].copy_(to_dev(hint))
    rde_chem.rde_chem_advance_ex(m.handle, DT, cells=rde_chem.make_block(**b), order=to_dev(np.arange(n), dtype=torch.int64),
                                 threads_per_cta=128)
    torch.cuda.synchronize()
    out.append(gather(keep, [n]))
    m.close()
    assert (out[0]["status"] == 0).all()
    for k in out[0]:
        assert np.array_equal(out[0][k], out[1][k]) and np.array_equal(out[0][k], out[2][k]), k


def test_graph_after_the_order_has_grown():
    mech, m = mechanism()
    cells = synth.field_cells(mech, 20000, seed=48)
    more = synth.field_cells(mech, 50000, seed=49)
    p, T0, Y0 = to_dev(cells.p), to_dev(cells.T), to_dev(cells.Y)
    T, Y = T0.clone(), Y0.clone()
    g = rde_chem.rde_chem_graph_create(m.handle, 2, DT, cells=rde_chem.make_block(p, T, Y))
    out = []
    for _ in range(2):
        T.copy_(T0)
        Y.copy_(Y0)
        rde_chem.rde_chem_graph_launch(g)
        torch.cuda.synchronize()
        out.append((T.clone(), Y.clone()))
        rde_chem.rde_chem_advance_ex(m.handle, DT, cells=rde_chem.make_block(to_dev(more.p), to_dev(more.T),
                                                                             to_dev(more.Y)))
        torch.cuda.synchronize()
    rde_chem.rde_chem_graph_destroy(g)
    m.close()
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    assert not torch.equal(out[0][0], T0)


def test_a_refused_graph_takes_no_memory():
    """The arguments are checked before room for the order is made (2 GB here)."""
    mech, m = mechanism()
    table = torch.zeros(256, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    with pytest.raises(rde_chem.RdeError):
        rde_chem.rde_chem_graph_create(m.handle, 1, DT, blocks=table, n_blocks=2000, n_total=1 << 28)
    assert torch.cuda.mem_get_info()[0] > free - (1 << 30)
    m.close()

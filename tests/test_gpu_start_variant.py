"""The staging mode that double-float operators, their solver and smoother kernels, batches and multi-block
launches start with, by degree, kind and size; and that the mode changes no bit of a result."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cw():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2607_03413_gb300 as cw
    from paper_2607_03413_gb300 import build
    build.build()
    cw.load()
    return cw


@pytest.mark.parametrize("p,kind,dims,stage", [
    (5, 2, (20, 20, 20), 1), (7, 2, (30, 30, 20), 1),  # the mass operator has one metric component
    (5, 1, (19, 12, 8), 1), (5, 1, (19, 12, 9), 2), (5, 3, (19, 12, 9), 2),  # 456 and more tiles of 4 cells
    (7, 1, (19, 12, 4), 1), (7, 1, (19, 8, 10), 2), (7, 3, (19, 8, 10), 2),  # 456 and 760 tiles of 2 cells
    (7, 1, (19, 8, 11), 1), (7, 1, (32, 32, 15), 1), (7, 1, (32, 32, 16), 2), (7, 3, (32, 32, 16), 1),
    (2, 1, (30, 30, 30), 1), (4, 3, (20, 20, 20), 1), (6, 1, (16, 16, 16), 1)])
def test_staging_mode_of_a_new_operator(cw, p, kind, dims, stage):
    op = cw.Operator(cw.Mesh.box(*dims, perturb=0.1), p, kind, cw.CW_GEOM_METRIC, cw.CW_PREC_F64)
    assert op.variant()[1] == stage


@pytest.mark.parametrize("p", [5, 7])
def test_solver_and_smoother_in_both_modes(cw, p):
    import torch
    m0 = synth.box_mesh(2, 2, 1, perturb=0.1)
    ops = [cw.Operator(cw.Mesh.from_synth(m), p, cw.CW_LAPLACE, cw.CW_GEOM_METRIC, cw.CW_PREC_F64, cw.CW_BC_DIRICHLET0)
           for m in (m0, synth.refine(m0))]
    mg = cw.Multigrid(ops)
    b = ops[1].load_vector(0)
    got = []
    for stage in (1, 2):
        ops[1].set_variant(0, stage)
        u = mg.smooth(1, b, torch.zeros_like(b), 2)
        x, st, rc = ops[1].cg_solve(b, rtol=1e-8)
        assert rc == cw.CW_OK
        got.append((u.clone(), x.clone(), st.iterations))
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1]) and got[0][2] == got[1][2]


@pytest.mark.parametrize("p,n", [(5, 2), (5, 7), (7, 2), (7, 13)])
def test_multi_block_in_both_modes(cw, p, n):
    """Eight blocks of n^3 cells in one launch: modes 1 and 2 by the cells of all blocks together."""
    import torch
    blocks = synth.cube_blocks(2, n, perturb=0.1, seed=5).blocks
    ops = [cw.Operator(cw.Mesh.from_synth(m), p, cw.CW_LAPLACE, cw.CW_GEOM_METRIC, cw.CW_PREC_F64) for m in blocks]
    mb = cw.MultiBlock(ops)
    g = torch.Generator(device="cuda").manual_seed(p)
    x = torch.rand(sum(o.L for o in ops), dtype=torch.float64, device="cuda", generator=g) * 2 - 1
    y = mb.apply(x)
    ref = torch.cat([o.apply(part.clone()) for o, part in zip(ops, x.split([o.L for o in ops]))])
    assert torch.equal(y, ref)

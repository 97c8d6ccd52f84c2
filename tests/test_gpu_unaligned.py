"""Vectors that start one value past an aligned address take the value-by-value paths (no bulk copy, no wide
line accesses): the results are bit-identical to those on aligned vectors, for every degree and precision, on
meshes with a ragged last tile."""
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


def shifted(t):
    import torch
    buf = torch.empty(t.numel() + 1, dtype=t.dtype, device="cuda")
    buf[1:] = t
    return buf[1:]


@pytest.mark.parametrize("geom", [0, 1, 2], ids=["affine", "metric", "recompute"])
@pytest.mark.parametrize("prec", [0, 1, 2, 3, 4])
@pytest.mark.parametrize("p", [1, 2, 3, 4, 5, 6, 7])
def test_apply_and_dss(cw, p, prec, geom):
    import torch
    m = synth.box_mesh(5, 3, 3, perturb=0.1 if geom else 0.0)
    op = cw.Operator(cw.Mesh.from_synth(m), p, cw.CW_LAPLACE_MASS, geom, prec)
    x = op.gather(torch.from_numpy(synth.global_vector(m, p, seed=8)).cuda())
    for assemble in (False, True):
        ref = op.apply(x, assemble=assemble)
        got = op.apply(shifted(x), shifted(torch.zeros_like(x)), assemble=assemble)
        assert torch.equal(got, ref)
    v = torch.from_numpy(synth.cellwise_random(m, p, seed=9)).cuda().to(op.vec_dtype)
    for average in (False, True):
        assert torch.equal(op.dss(shifted(v), average=average), op.dss(v.clone(), average=average))


@pytest.mark.parametrize("prec", [0, 2], ids=["df64", "f32"])
@pytest.mark.parametrize("p", [1, 2, 3, 4, 5, 6, 7])
def test_cycle_parts(cw, p, prec):
    import torch
    m0 = synth.box_mesh(2, 3, 2, perturb=0.1)
    meshes = [m0, synth.refine(m0)]
    ops = [cw.Operator(cw.Mesh.from_synth(m), p, cw.CW_LAPLACE, cw.CW_GEOM_METRIC, prec, cw.CW_BC_DIRICHLET0)
           for m in meshes]
    mg = cw.Multigrid(ops)
    dt = ops[0].vec_dtype
    uc = ops[0].gather(torch.from_numpy(synth.global_vector(meshes[0], p, seed=1)).cuda())
    uf = ops[1].gather(torch.from_numpy(synth.global_vector(meshes[1], p, seed=2)).cuda())
    b = torch.from_numpy(synth.cellwise_random(meshes[1], p, seed=3)).cuda().to(dt)
    assert torch.equal(mg.prolong(1, shifted(uc), shifted(uf)), mg.prolong(1, uc))
    assert torch.equal(mg.restrict(1, shifted(uf), shifted(uc)), mg.restrict(1, uf))
    assert torch.equal(mg.smooth(1, shifted(b), shifted(uf), 2), mg.smooth(1, b, uf.clone(), 2))
    assert torch.equal(mg.vcycle(shifted(b), shifted(uf)), mg.vcycle(b, uf.clone()))

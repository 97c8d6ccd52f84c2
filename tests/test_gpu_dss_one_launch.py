"""The DSS of small meshes in one launch (one thread per grid node) against the axis passes written out
in torch: bit-identical for sums and averages in every vector type, on ragged meshes and at both ends of
the size range, alone, behind an operator that summed x-interfaces inside its tiles, and over several
blocks."""
import numpy as np
import pytest

import synth
from gpu_util import to_np

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


def passes(v, dims, p, average):
    """Algorithm struct_dss axis by axis on v [cells, n, n, n], in v's own type."""
    w = v.reshape(tuple(reversed(dims)) + (p + 1,) * 3).clone()
    for ax in (2, 1, 0):  # x, y, z
        if w.shape[ax] < 2:
            continue
        l = w.narrow(ax, 0, w.shape[ax] - 1).select(3 + ax, p)
        r = w.narrow(ax, 1, w.shape[ax] - 1).select(3 + ax, 0)
        s = l + r
        if average:
            s = s * 0.5
        l.copy_(s)
        r.copy_(s)
    return w.reshape(v.shape)


@pytest.mark.parametrize("average", [False, True], ids=["sum", "average"])
@pytest.mark.parametrize("prec", [0, 2, 4], ids=["f64", "f32", "bf16"])
@pytest.mark.parametrize("p,dims", [(1, (1, 1, 1)), (1, (2, 1, 1)), (1, (257, 3, 2)), (2, (3, 1, 5)), (3, (5, 4, 3)),
                                    (3, (20, 20, 20)), (3, (21, 20, 20)), (4, (1, 7, 1)), (7, (2, 3, 2)), (7, (10, 10, 11))])
def test_one_launch_equals_the_axis_passes(cw, p, dims, prec, average):
    import torch
    m = synth.box_mesh(*dims)
    op = cw.Operator(cw.Mesh.from_synth(m), p, cw.CW_MASS, cw.CW_GEOM_AFFINE, prec)
    v = torch.from_numpy(synth.cellwise_random(m, p, seed=4)).cuda().to(op.vec_dtype)
    v[::7] = 0.0
    v[3::11] *= 2.0 ** -120  # (bf16 and f32: still normal after three halvings)
    ref = passes(v, dims, p, average)
    assert torch.equal(op.dss(v, average=average), ref)


@pytest.mark.parametrize("prec", [0, 2, 3, 4])
@pytest.mark.parametrize("p,dims", [(1, (70, 3, 2)), (2, (17, 3, 5)), (3, (9, 5, 3)), (4, (11, 3, 2)), (6, (9, 2, 3))])
def test_assembled_apply_on_a_small_mesh(cw, p, dims, prec):
    """x-interfaces between and inside the operator's tiles, rows that are no multiple of the tile."""
    import torch
    m = synth.box_mesh(*dims, perturb=0.1)
    op = cw.Operator(cw.Mesh.from_synth(m), p, cw.CW_LAPLACE_MASS, cw.CW_GEOM_METRIC, prec)
    x = op.gather(torch.from_numpy(synth.global_vector(m, p, seed=5)).cuda())
    assert torch.equal(op.apply(x, assemble=True), passes(op.apply(x), dims, p, False))


@pytest.mark.parametrize("prec", [0, 2])
@pytest.mark.parametrize("p,nblocks", [(1, 2), (3, 2), (2, 3)])
def test_multi_block_in_one_launch_equals_block_by_block(cw, p, nblocks, prec):
    """8 and 27 blocks (more than one launch's table): the operators and the DSS of all blocks together
    against block by block, then the shared DoFs."""
    import torch
    blocks = synth.cube_blocks(nblocks, 2, perturb=0.1, seed=3).blocks
    ops = [cw.Operator(cw.Mesh.from_synth(b), p, cw.CW_LAPLACE, cw.CW_GEOM_METRIC, prec) for b in blocks]
    mb = cw.MultiBlock(ops)
    idx = mb.global_index()
    g = np.random.default_rng(6).uniform(-1, 1, mb.NG)
    x = torch.from_numpy(g[idx]).cuda().to(mb.vec_dtype)
    y = mb.apply(x)
    at = 0
    for o in ops:
        part = x[at:at + o.L].clone()
        assert torch.equal(y[at:at + o.L], o.apply(part))
        at += o.L
    ref = np.zeros(mb.NG)
    np.add.at(ref, idx, to_np(y))
    got = to_np(mb.apply(x, assemble=True))
    # at most 12 copies (8 inside a block's order, then across blocks): each sum errs by at most
    # 11 units in the last place of the sum of magnitudes
    mag = np.zeros(mb.NG)
    np.add.at(mag, idx, np.abs(to_np(y)))
    eps = 2.0 ** -53 if prec == 0 else 2.0 ** -24
    assert np.all(np.abs(got - ref[idx]) <= 2 * 64 * eps * mag[idx])

"""The DSS above the size up to which one launch per node does it: the axis passes and the y/z line launch, by
degree, vector type and size class, against the passes written out in torch, bit for bit; on aligned vectors and on
ones that start one value past an aligned address, alone and behind an operator that summed the x-interfaces
inside its tiles (rows that are no multiple of the tile)."""
import pytest

from test_gpu_dss_one_launch import passes
from test_gpu_unaligned import shifted

pytestmark = pytest.mark.gpu

# just above 2^19 entries; no dimension a multiple of a tile of 4 cells and more
DIMS = {2: (29, 27, 27), 3: (21, 19, 22), 4: (17, 18, 15), 5: (14, 14, 13), 6: (13, 11, 12), 7: (11, 10, 10)}


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


def vector(op, seed):
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    v = (torch.rand(op.L, dtype=torch.float64, device="cuda", generator=g) * 2 - 1).to(op.vec_dtype)
    v[::7] = 0.0
    v[3::11] *= 2.0 ** -120  # (bf16 and f32: still normal after three halvings)
    return v


def check(cw, p, dims, prec, average):
    import torch
    op = cw.Operator(cw.Mesh.box(*dims), p, cw.CW_MASS, cw.CW_GEOM_AFFINE, prec)
    v = vector(op, 10 * p + prec)
    ref = passes(v, dims, p, average)
    assert torch.equal(op.dss(shifted(v), average=average), ref)
    assert torch.equal(op.dss(v, average=average), ref)


@pytest.mark.parametrize("average", [False, True], ids=["sum", "average"])
@pytest.mark.parametrize("prec", [0, 2, 4], ids=["f64", "f32", "bf16"])
@pytest.mark.parametrize("p", sorted(DIMS))
def test_above_one_launch(cw, p, prec, average):
    assert DIMS[p][0] * DIMS[p][1] * DIMS[p][2] * (p + 1) ** 3 > 2 ** 19
    check(cw, p, DIMS[p], prec, average)


@pytest.mark.parametrize("average", [False, True], ids=["sum", "average"])
@pytest.mark.parametrize("p,dims,prec", [
    (3, (1, 91, 92), 2), (3, (91, 1, 92), 4), (3, (92, 91, 1), 2), (3, (8200, 1, 1), 2), (5, (1, 1, 2500), 4),
    (3, (33, 32, 32), 2),  # FP32 Q3 between 2^21 and 2^25 entries, and above
    (3, (81, 81, 81), 2),
    (3, (65, 64, 64), 0), (5, (43, 43, 43), 0), (7, (33, 32, 32), 0)],  # FP64 sums above 2^24 entries
    ids=str)
def test_shapes_and_sizes(cw, p, dims, prec, average):
    check(cw, p, dims, prec, average)


@pytest.mark.parametrize("geom", [1, 2], ids=["metric", "recompute"])
@pytest.mark.parametrize("prec", [0, 1, 2, 3, 4])
@pytest.mark.parametrize("p", sorted(DIMS))
def test_assembled_apply(cw, p, prec, geom):
    import torch
    op = cw.Operator(cw.Mesh.box(*DIMS[p], perturb=0.1), p, cw.CW_LAPLACE, geom, prec)
    x = op.gather(torch.rand(op.NG, dtype=torch.float64, device="cuda",
                             generator=torch.Generator(device="cuda").manual_seed(p)) * 2 - 1)
    ref = passes(op.apply(x), DIMS[p], p, False)
    assert torch.equal(op.apply(x, assemble=True), ref)
    assert torch.equal(op.apply(shifted(x), shifted(torch.zeros_like(x)), assemble=True), ref)


@pytest.mark.parametrize("p,dims", [(3, (65, 64, 64)), (5, (43, 43, 43))])
def test_assembled_apply_in_fp64_above_2e24_entries(cw, p, dims):
    import torch
    op = cw.Operator(cw.Mesh.box(*dims, perturb=0.1), p, cw.CW_LAPLACE, cw.CW_GEOM_METRIC, cw.CW_PREC_F64)
    x = vector(op, p)
    assert torch.equal(op.apply(x, assemble=True), passes(op.apply(x), dims, p, False))

"""Batches large enough that a persistent CTA works on several items and an item holds several tiles: the
staged metric and input tiles, their barriers' phases and the line buffers are used again and again. Every
variant against the per-operator apply, with one and several right-hand sides and ragged last tiles."""
import math

import pytest

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


def big_batch(cw, prec, p, kind):
    """One mesh of more than 3 x 24 tiles per SM (three tiles per item at least, and more items than resident
    CTAs), its last tile ragged, with three right-hand sides, and a small one with a single vector."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    probe = cw.Operator(cw.Mesh.box(2), p, kind, cw.CW_GEOM_METRIC, prec)
    tile = probe.variant()[2][0]
    probe.close()
    side = int(math.ceil((3.1 * 24 * sms * tile) ** (1 / 3))) | 1  # odd: no multiple of the tile
    ops = [cw.Operator(cw.Mesh.box(*d, perturb=0.1), p, kind, cw.CW_GEOM_METRIC, prec)
           for d in ((side, side, side), (7, 5, 3))]
    nrhs = [3, 1]
    g = torch.Generator(device="cuda").manual_seed(31 * p + kind)
    xs = [(torch.rand(r * o.L, dtype=torch.float64, device="cuda", generator=g) * 2 - 1).to(o.vec_dtype)
          for o, r in zip(ops, nrhs)]
    return ops, nrhs, xs, [torch.empty_like(x) for x in xs]


@pytest.mark.parametrize("kind", [1, 2, 3])
@pytest.mark.parametrize("prec", [0, 2], ids=["df64", "f32"])
@pytest.mark.parametrize("p", [1, 2, 3, 4, 5, 6, 7])
def test_many_tiles_per_cta(cw, p, prec, kind):
    import torch
    ops, nrhs, xs, ys = big_batch(cw, prec, p, kind)
    refs = [torch.cat([o.apply(x[r * o.L:(r + 1) * o.L].clone()) for r in range(n)])
            for o, x, n in zip(ops, xs, nrhs)]
    B = cw.Batch(ops, nrhs, xs, ys)
    for variant in (None, 0, 1, 2, 3, 4, 5):  # None: the one a batch starts with
        if variant is not None:
            B.set_variant(p, variant)
        for y in ys:
            y.fill_(float("nan"))
        B.launch()
        torch.cuda.synchronize()
        for y, ref in zip(ys, refs):
            if prec == 0:  # the same double-float operations per cell: bit-identical
                assert torch.equal(y, ref), variant
            else:  # FP32: the bound of the small batches' test
                assert ((y - ref).abs().max() <= 1e-6 * ref.abs().max()).item(), variant
    assert all(cw.cw_op_check(o.handle) == cw.CW_OK for o in ops)
    B.close()


@pytest.mark.parametrize("prec", [0, 2], ids=["df64", "f32"])
@pytest.mark.parametrize("p", [2, 3, 5])
def test_expired_wait_ends_the_staging_of_its_cta(cw, p, prec):
    """The batch's barriers armed with more bytes than the copies deliver: the waits run out. A metric tile is
    read from global memory instead, for that and every later tile and right-hand side, so the results stay
    right; an input tile gives zeros once per CTA, the later ones are read directly; both are reported, and a
    batch without the injection on the same operators runs as always."""
    import torch
    ops, nrhs, xs, ys = big_batch(cw, prec, p, 1)
    tol = 0.0 if prec == 0 else 1e-6  # as above
    refs = [torch.cat([o.apply(x[r * o.L:(r + 1) * o.L].clone()) for r in range(n)])
            for o, x, n in zip(ops, xs, nrhs)]
    for variant in (2, 4):
        for o in ops:
            cw.cw_op_inject_stall(o.handle, True)
        B = cw.Batch(ops, nrhs, xs, ys)
        B.set_variant(p, variant)
        for y in ys:
            y.fill_(float("nan"))
        B.launch()
        assert cw.cw_op_check(ops[0].handle) == cw.CW_ERR_TIMEOUT
        cw.cw_op_check(ops[1].handle)
        y, ref = ys[0], refs[0]
        assert torch.isfinite(y).all()
        if variant == 2:
            assert ((y - ref).abs().max() <= tol * ref.abs().max()).item()
        else:  # at most one tile of zeros per resident CTA (16 a SM at the most)
            cells = (y.view(nrhs[0], -1, (p + 1) ** 3) == 0).all(dim=2)
            tile = B.variant(p)[1]
            sms = torch.cuda.get_device_properties(0).multi_processor_count
            assert 0 < int(cells.sum()) <= 16 * sms * tile
            good = ~cells.unsqueeze(2).expand(-1, -1, (p + 1) ** 3).reshape(-1)
            assert ((y - ref)[good].abs().max() <= tol * ref.abs().max()).item()
        B.close()
        for o in ops:
            cw.cw_op_inject_stall(o.handle, False)
        B = cw.Batch(ops, nrhs, xs, ys)
        B.set_variant(p, variant)
        B.launch()
        assert cw.cw_op_check(ops[0].handle) == cw.CW_OK and cw.cw_op_check(ops[1].handle) == cw.CW_OK
        assert ((ys[0] - refs[0]).abs().max() <= tol * refs[0].abs().max()).item()
        B.close()

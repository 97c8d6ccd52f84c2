"""Batches of different degrees that exist at the same time: each gives its own operators' results, whichever was
created last, in both modes, launched in turn and side by side on two streams."""
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


@pytest.mark.parametrize("mode", [0, 1], ids=["grouped", "single"])
@pytest.mark.parametrize("prec", [0, 2], ids=["df64", "f32"])
def test_batches_of_different_degrees(cw, prec, mode):
    import torch
    made = []
    for p in (2, 5, 3, 7):
        op = cw.Operator(cw.Mesh.box(6, perturb=0.1), p, cw.CW_LAPLACE, cw.CW_GEOM_METRIC, prec)
        g = torch.Generator(device="cuda").manual_seed(p)
        x = (torch.rand(op.L, dtype=torch.float64, device="cuda", generator=g) * 2 - 1).to(op.vec_dtype)
        y = torch.empty_like(x)
        B = cw.Batch([op], [1], [x], [y])
        B.set_mode(mode)
        made.append((op, x, y, B, op.apply(x)))

    def check():
        torch.cuda.synchronize()
        for op, _, y, _, ref in made:
            if prec == 0:  # the same double-float operations: bit-identical
                assert torch.equal(y, ref)
            else:  # the bound of the batch tests
                assert ((y - ref).abs().max() <= 1e-6 * ref.abs().max()).item()
            y.fill_(float("nan"))

    for _, _, _, B, _ in made:
        B.launch()
    check()
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in made]
    for s, (_, _, _, B, _) in zip(streams, made):
        with torch.cuda.stream(s):
            B.launch(graph=True)
    check()
    for _, _, _, B, _ in made:
        B.close()

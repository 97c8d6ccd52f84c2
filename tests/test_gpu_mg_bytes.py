"""cw_mg_device_bytes is the sum of what a hierarchy allocates: a work vector and D_hat per level, right-hand
side and iterate below the finest, and on level 0 the dense inverse, its two vectors and two index maps."""
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,es", [(0, 8), (2, 4)], ids=["f64", "f32"])
@pytest.mark.parametrize("p,levels", [(1, 3), (3, 2)])
def test_device_bytes(p, levels, prec, es):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2607_03413_gb300 as cw
    ms = [synth.box_mesh(2, 3, 2, perturb=0.1)]
    while len(ms) < levels:
        ms.append(synth.refine(ms[-1]))
    ops = [cw.Operator(cw.Mesh.from_synth(m), p, cw.CW_LAPLACE, cw.CW_GEOM_METRIC, prec, cw.CW_BC_DIRICHLET0) for m in ms]
    mg = cw.Multigrid(ops)
    ni = (2 * p - 1) * (3 * p - 1) * (2 * p - 1)  # interior DoFs of the coarsest level
    want = sum(o.L * es * (2 if o is ops[-1] else 4) for o in ops)
    want += 8 * (ni * ni + 2 * ni) + 4 * ni + 4 * ops[0].L
    assert cw.cw_mg_device_bytes(mg.handle) == want

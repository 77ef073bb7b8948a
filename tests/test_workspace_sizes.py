"""What a handle's workspace is made of (host logic: runs without a GPU)."""
import pytest


def al(v):
    return (v + 255) // 256 * 256


@pytest.mark.parametrize("integ,stages", [("RK4", 4), ("HEUN", 2)])
@pytest.mark.parametrize("shape", [(16, 16, 16), (33, 17, 9)])
def test_small_fp32_lattices(integ, stages, shape):
    """The stage inputs of the small-lattice stage kernels (6N or 3N floats) where
    they are used, and not with path = 1, whose stage arrays are its own."""
    import paper_1610_04914_gb300 as sp
    n = shape[0] * shape[1] * shape[2]
    fused, generic = (sp.spin_workspace_size(sp.Params(*shape, integrator=getattr(sp, integ), path=p)) for p in (0, 1))
    inputs = al(4 * (6 if stages == 4 else 3) * n)
    assert generic - fused == al(4 * (stages + 1) * 3 * n) - inputs


def test_fp64_stage_inputs():
    """FP64: the second state and the stage inputs, 6N (RK4) or 3N doubles."""
    import paper_1610_04914_gb300 as sp
    n = 24 ** 3
    ws = [sp.spin_workspace_size(sp.Params(24, 24, 24, precision=64, integrator=i, path=p))
          for i, p in ((sp.RK4, 0), (sp.HEUN, 0), (sp.RK4, 1))]
    assert ws[0] - ws[1] == al(8 * 6 * n) - al(8 * 3 * n)
    assert ws[2] - ws[0] == al(8 * 15 * n) - al(8 * 6 * n)

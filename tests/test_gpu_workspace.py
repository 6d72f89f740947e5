"""Device memory that solves keep: no more than their own vectors."""
import pytest

from paper_2409_03030_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["mixed_f16", "mixed_f32", "multishift"])
def test_blocks_of_iterations_take_no_memory(kind):
    """The vectors of a block of iterations (directions of the mixed CG,
    residuals of the multi-shift CG) lie in the solver's own: what a solve adds
    to a field's device memory are the vectors that it names, so that whatever
    could be allocated beside a solved field still can.  Bound: their bytes, in
    whole pages of 2 MiB each; a second field is measured, with every kernel
    loaded by the first."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_03030_gb300 import jqcd
    dims, vh, nshift = (16, 16, 16, 32), 16 ** 3 * 16, 2
    b = synth.gaussian_spinor(dims, seed=61)
    mode = {"mixed_f16": jqcd.CG_MIXED_F16, "mixed_f32": jqcd.CG_MIXED_F32}.get(kind)

    def solve(g):
        if mode is None:
            g.cg_multishift(b, 0.12, [0.0, 0.3][:nshift], tol=1e-6)
        else:
            g.cg_solve(b, 0.12, tol=1e-6, mode=mode)

    hop = {"mixed_f16": 52, "mixed_f32": 96}.get(kind)
    # x_s, r_s; p, w, t -- or x_i and p_i of each shift -- and two scalar blocks
    sizes = [192 * vh] * (2 * nshift) + [1, 1] if mode is None else [96 * vh] * 2 + [hop * vh] * 3
    bound = sum(-(-s // 2 ** 21) * 2 ** 21 for s in sizes)
    with jqcd.Context(0) as ctx:
        fields = [ctx.gauge_upload(dims, synth.gauge(dims, "expi", eps=0.3, seed=62)) for _ in range(2)]
        for g in fields:  # the double-word solver's workspace, and the code of its kernels
            g.cg_solve(b, 0.12, tol=1e-6, mode=jqcd.CG_DW)
        solve(fields[0])
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        solve(fields[1])
        torch.cuda.synchronize()
        assert before - torch.cuda.mem_get_info()[0] <= bound

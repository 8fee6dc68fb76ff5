"""Double-float line solves (lbm_cfd_df): chunks are in registers, and in launches of more than
4560 blocks the double-float ones are loops in shared memory.  Both give the same bits: many
lines at once against the same lines a few at a time, with groups solved in FP32 and groups
across an interface side by side."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [4, 6])
@pytest.mark.parametrize("axis", [0, 1])
@pytest.mark.parametrize("n,lines", [(40, 80000), (37, 75997), (8, 160000), (5000, 3704), (1001, 2397)])
def test_many_lines_equal_few(cuda, n, lines, axis, order):
    from paper_1906_09530_gb300 import lbm_cfd_df
    torch = cuda
    gen = torch.Generator(device="cuda").manual_seed(n)
    u = torch.rand((lines, n), generator=gen, device="cuda", dtype=torch.float64) + 1.0
    steep = torch.arange(lines, device="cuda") // 24 % 3 == 1
    u[steep, : n // 2] *= 1e-5
    hi = u.float()
    lo = (u - hi.double()).float()

    def solve(a, b, second):
        h, lw = hi[a:b], lo[a:b]
        if axis == 1:
            h, lw = h.t(), lw.t()
        out = lbm_cfd_df(h.contiguous(), lw.contiguous(), axis, order, second)
        out = out if second else (out,)
        return [o.t() if axis == 1 else o for o in out]

    for second in (True, False):
        whole = solve(0, lines, second)
        few = [solve(a, min(a + 1920, lines), second) for a in range(0, lines, 1920)]
        for i, w in enumerate(whole):
            assert torch.isfinite(w).all()
            assert torch.equal(w, torch.cat([f[i] for f in few]))

"""lbm_cfd_df on pointers that are aligned for floats alone: contiguous views at an odd offset
give the bits of aligned copies, whichever of the inputs and outputs they are, for rows that
are whole 16-byte pieces and rows that are not."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("axis", [0, 1])
@pytest.mark.parametrize("nx,ny", [(64, 40), (8, 700), (700, 9), (37, 29)])
def test_any_float_alignment(cuda, nx, ny, axis):
    from paper_1906_09530_gb300 import lib
    torch = cuda
    gen = torch.Generator(device="cuda").manual_seed(nx)
    n = nx * ny
    hi = torch.rand(n, generator=gen, device="cuda") + 0.5
    hi[: n // 3] *= 1e-5  # (windows both above and below the factor that wants double-float)
    lo = hi * 2.0**-26 * torch.rand(n, generator=gen, device="cuda")

    def solve(offsets, second):
        bufs = [torch.full((n + 4,), -7.0, device="cuda") for _ in range(4)]
        v = [b[o:o + n] for b, o in zip(bufs, offsets)]
        v[0].copy_(hi)
        v[1].copy_(lo)
        assert [x.data_ptr() % 16 for x in v] == [4 * o for o in offsets]
        s = torch.cuda.current_stream().cuda_stream
        assert lib().lbm_cfd_df(v[0].data_ptr(), v[1].data_ptr(), v[2].data_ptr(),
                                v[3].data_ptr() if second else None, nx, ny, axis, 6, s) == 0
        torch.cuda.synchronize()
        for b, o in zip(bufs[2:], offsets[2:]):  # nothing written beside the outputs
            assert torch.all(b[:o] == -7.0) and torch.all(b[o + n:] == -7.0)
        return v[2].clone(), v[3].clone()

    for second in (True, False):
        want = solve((0, 0, 0, 0), second)
        for offsets in ((1, 0, 0, 0), (0, 2, 0, 0), (0, 0, 3, 0), (0, 0, 0, 1), (1, 1, 1, 1),
                        (1, 3, 2, 1)):
            assert all(torch.equal(a, b) for a, b in zip(solve(offsets, second), want))

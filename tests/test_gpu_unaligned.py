"""Gridding into buffers on 8-byte boundaries: the C ABI asks for doubles and 64-bit words, not for more."""
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_0906_3978_gb300 as wf  # noqa: E402

DEV = "cuda:0"


@pytest.mark.parametrize("n", [16, 48, 108, 256])
def test_grid_assign_on_8_byte_boundaries(n):
    wf.build()
    box = 2.0 * n
    pos = torch.from_numpy(synth.uniform_catalogue(5000, box, 3)).to(DEV)
    with wf.Context(0) as ctx:
        fine = torch.empty((2 * n) ** 3, dtype=torch.int64, device=DEV)
        ref = ctx.grid_assign(pos, n, box, wf.TSC, 2, fine_out=fine)
        off_fine = torch.empty((2 * n) ** 3 + 1, dtype=torch.int64, device=DEV)[1:]
        off_obs = torch.empty(n ** 3 + 1, dtype=torch.float64, device=DEV)[1:]
        assert off_fine.data_ptr() % 16 == 8 and off_obs.data_ptr() % 16 == 8
        ctx.grid_assign(pos, n, box, wf.TSC, 2, fine_out=off_fine, n_obs=off_obs)
        torch.cuda.synchronize()
        assert torch.equal(off_fine, fine)
        assert torch.equal(off_obs, ref.ravel())

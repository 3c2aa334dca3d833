"""Maps of the persistent batch kernel equal single requests bit for bit, also
where short rings fold many orders onto few spectrum entries (lmax well above a
ring's length) and at every block size the schedule can have."""
import pytest

from paper_1110_4874_gb300 import synthetic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1110_4874_gb300 as sh  # noqa: E402


# plans whose ring kernels run 128 threads a block, and one (rings of 4 x 800
# pixels) that runs 256
@pytest.mark.parametrize("nside,lmax", [(64, 256), (64, 1024), (128, 512), (100, 600), (800, 330)])
def test_persistent_batch_equals_single_requests(nside, lmax):
    plan = sh.Plan(nside, lmax, 1e-10)
    a = torch.from_numpy(synthetic.gaussian_alm(lmax, 3, seed=1)).cuda()
    want = plan.synthesize(a)
    for warps in (1, 2, 4, 8):
        maps = torch.zeros_like(want)
        b = sh.shtb_batch_create([(plan, a, maps)], autotune=False, warps_per_block=warps)
        sh.shtb_batch_run(b)
        sh.shtb_batch_status(b)
        assert torch.equal(maps, want), warps
        sh.shtb_batch_destroy(b)

"""Tails ahead of a front on the GPU: parts swept as a filter, whole, in halves and in quarters,
and the cells left over, give the same bits wherever a part begins."""
import numpy as np
import pytest

from paper_1407_2052_gb300 import workloads as W
from test_gpu_parity import A, dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()


@pytest.mark.parametrize("recon", ["MP5", "LIMO3"])
def test_tails_of_a_blast_do_not_depend_on_the_tile(recon):
    w, ref = W.blast3d(96, 16), None
    for tile in (None, (64, 8, 320), (64, 4, 160), (16, 32, 288), (40, 6, 192)):
        s = A().Solver(w.physics, w.ndim, w.integrator, w.gamma, w.cfl, w.domains, glm_cr=w.glm_cr,
                       recon=getattr(A(), recon))
        if tile:
            s.set_tile(*tile)
        U = dev(w.U)
        for _ in range(7):
            s.step_cfl(U)
        out = U.cpu().numpy().reshape(9, -1)
        if ref is None:
            ref = out
            bz = np.abs(out[7])
            assert bz.max() > 1e-3 and bz[bz > 0].min() < 1e-40
        assert np.array_equal(out, ref), tile
        s.close()

"""The default tile of a handle, on the GPU: threads that have work, segments that fit it."""
import pytest

from paper_1407_2052_gb300 import workloads as W
from test_gpu_parity import A

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()


def _tile(physics, n, nb, tune=False):
    nd = sum(m > 1 for m in n)
    s = A().Solver(physics, nd, A().SSPRK3, 1.4, 0.4, [W.Domain(n, (1.0 / n[0],) * 3, nb=nb)], glm_cr=0.18)
    if tune:
        U = torch.ones(s.nv * n[0], dtype=torch.float64, device="cuda")
        U[-n[0]:] = 10.0  # Euler's energy
        s.autotune(U, torch.full((1,), 1e-6, dtype=torch.float64, device="cuda"))
    t = s.get_tile()
    s.close()
    return t


@pytest.mark.parametrize("physics", [0, 1])
@pytest.mark.parametrize("n", [48, 512, 19000, 19500, 70000, 80000, 1000000, 4000000])
def test_a_tube_takes_no_more_threads_than_a_line_has_work(physics, n):
    """A tile of one line has few sweeps: beyond them threads wait. Many lines (a large tube)
    fill the GPU with one warp each."""
    nb = 1 if n < 32000 else n // 10000
    seg, lines, threads = _tile(physics, (n, 1, 1), (nb, 1, 1))
    assert lines == 1 and 32 <= threads <= 160
    if n >= 1000000:
        assert seg == 64 and threads == 32
    if n <= 512:
        assert seg == 16


def test_small_tubes_of_a_large_batch_keep_a_thread_per_sweep():
    """The plain path launches one domain at a time: nothing else fills the GPU then."""
    doms = [W.Domain((5000, 1, 1), (2e-4, 1.0, 1.0), offset=i * 9 * 5000) for i in range(40)]
    s = A().Solver(A().MHD_GLM, 1, A().SSPRK3, 1.4, 0.4, doms, glm_cr=0.18)
    assert s.get_tile()[2] >= 72  # nine variables in parts of 8 cells of a segment of 64
    s.close()


def test_tuning_a_tube_times_its_default_tile():
    n = 1000000
    assert _tile(0, (n, 1, 1), (100, 1, 1), tune=True)[2] <= 64


@pytest.mark.parametrize("physics, n, nb, seg", [
    (0, (48, 48, 48), (3, 3, 3), 16), (0, (57, 38, 76), (3, 2, 4), 32), (0, (512, 512, 1), (1, 1, 1), 32),
    (1, (36, 36, 36), (3, 3, 3), 16), (1, (20, 90, 40), (1, 6, 2), 32), (1, (400, 380, 1), (8, 4, 1), 32)])
def test_middling_work_takes_long_segments_from_twenty_waves_of_faces_on(physics, n, nb, seg):
    assert _tile(physics, n, nb)[0] == seg

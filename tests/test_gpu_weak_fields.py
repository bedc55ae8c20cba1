"""Components far weaker than the flow that carries them, and of any range, on the GPU."""
import numpy as np
import pytest

import oracle as O
from paper_1407_2052_gb300 import workloads as W
from test_gpu_parity import A, dev, ocfg, odom, rel_linf

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()


def _flow(n, B):
    """Smooth periodic 3D flow, 9 conserved variables; B: three fields of shape (nz, ny, nx)."""
    nx, ny, nz = n
    x, y, z = (2 * np.pi * (np.arange(m) + 0.5) / m for m in n)
    X, Y, Z = x.reshape(1, 1, nx), y.reshape(1, ny, 1), z.reshape(nz, 1, 1)
    rho = 1 + 0.2 * np.sin(X + Y) + 0 * Z
    vel = [0.3 * np.sin(Y + Z) + 0 * X, 0.2 * np.cos(X - Z) + 0 * Y, 0.1 * np.sin(X + Y) + 0 * Z]
    p = 1 + 0.1 * np.cos(Y) + 0 * rho
    e = p / (5.0 / 3.0 - 1) + 0.5 * rho * sum(v * v for v in vel) + 0.5 * sum(b * b for b in B)
    return np.stack([rho] + [rho * v for v in vel] + [e] + list(B) + [0 * rho])


def _domain(n):
    return W.Domain(n, tuple(2 * np.pi / m for m in n))


@pytest.mark.parametrize("recon", ["MP5", "LIMO3"])
def test_seed_field_evolves_linearly_at_any_strength(recon):
    """A field too weak to act back obeys linear equations, and MP5 accepts every one of its
    faces; LIMO3 switches at r dx, beyond the field. Powers of two then scale it bit for bit."""
    n = (22, 16, 12)
    rng = np.random.default_rng(3)
    B = [rng.uniform(-1, 1, n[::-1]) for _ in range(3)]
    got = []
    for k in (80, 150, 400):
        Bk = [np.ldexp(b, -k) for b in B]
        s = A().Solver(A().MHD_GLM, 3, A().SSPRK3, 5.0 / 3.0, 0.4, [_domain(n)], glm_cr=0.18, recon=getattr(A(), recon))
        U = dev(_flow(n, Bk))
        for _ in range(3):
            s.step_cfl(U)
        out = U.cpu().numpy().reshape(9, -1)
        out[5:] = np.ldexp(out[5:], k)
        got.append(out)
        s.close()
    assert np.abs(got[0][5:]).max() > 0.1
    for g in got[1:]:
        assert np.array_equal(got[0], g)


@pytest.mark.parametrize("recon", ["MP5", "LIMO3"])
@pytest.mark.parametrize("spread", [20, 45, 150])
def test_fields_of_any_range_do_not_depend_on_the_tile(spread, recon):
    """Field components whose neighbouring cells differ by up to 2^spread: every width of the
    sweeps' sums, and the cells taken by themselves, agree bit for bit whatever the parts."""
    n = (40, 24, 20)
    rng = np.random.default_rng(spread)
    B = [0.1 * rng.uniform(-1, 1, n[::-1]) * 2.0 ** rng.uniform(-spread, 0, n[::-1]) for _ in range(3)]
    U0, ref = _flow(n, B), None
    w = W.Workload("fields", A().MHD_GLM, 3, A().SSPRK3, 5.0 / 3.0, 0.4, [_domain(n)], U0, recon=getattr(A(), recon))
    for tile in (None, (16, 4, 96), (64, 4, 160), (32, 8, 320)):
        s = A().Solver(A().MHD_GLM, 3, A().SSPRK3, 5.0 / 3.0, 0.4, [_domain(n)], glm_cr=0.18, recon=w.recon)
        if tile:
            s.set_tile(*tile)
        U = dev(U0)
        dt = s.dt(U)
        s.step(U, dt)
        out = U.cpu().numpy()
        if ref is None:
            ref, step = out, float(dt[0].item())
        assert np.array_equal(out, ref), tile
        s.close()
    want, fl, _, _ = O.step(ocfg(w), odom(w.domains[0]), w.U, step)
    assert fl == 0 and rel_linf(ref.reshape(9, -1), want.reshape(9, -1), 2.0) < 1e-12

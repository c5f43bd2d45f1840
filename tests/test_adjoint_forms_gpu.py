"""Which kernels a reverse step runs (cmrt_params.adjoint_fused), and the row
wavefronts on lattices of the sizes that run them by themselves.

adjoint_fused = 1 asks for the row wavefronts at any size; 2 for the plane
passes; 0 leaves it to the lattice's size: windows on small lattices.  The forms
sum in another order and are held to the tolerance of the tests that compare
them on small lattices (1e-5 of each gradient plus 1e-7 of the largest one: a
term's rounding and its sum's spread grow alike with the nodes).  The forward
fields of a state are written by the step that reads it or recomputed by the
reverse step, with the same bits, so that the checkpoint interval does not
change a result."""
import numpy as np
import pytest

from paper_2005_04642_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU machines too
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2005_04642_gb300 import cmrt as cm  # noqa: E402

cm.load()


def _setup(nx, ny, wall, **kw):
    d = I.base_params(nx, ny, wall_y=wall, g_acc=(1e-5, -2e-5), **kw)
    rn = I.drops_field(nx, ny, [(0.5 * nx + 0.3, 0.5 * ny - 0.2)], [0.25 * min(nx, ny)], periodic_y=not wall)
    target = I.drops_field(nx, ny, [(0.5 * nx + 1.3, 0.5 * ny + 0.3)], [0.25 * min(nx, ny)], periodic_y=not wall)
    u = I.velocity_noise(nx, ny, 0.01, 5)
    return d, rn.astype(np.float32), u.astype(np.float32), target.astype(np.float32)


def _close(a, b):
    top = max(abs(x) for x in b)
    return all(abs(x - y) <= 1e-5 * abs(y) + 1e-7 * top for x, y in zip(a, b))


# kernels of a VJP: with the row wavefronts the unstreaming pass, forward fields,
# collision, tail and reduction; by windows forward fields, (collision,) window and
# reduction; the plane passes are eight between the unstreaming and the reduction
@pytest.mark.parametrize("n,fused,vjp", [(64, 1, 5), (64, 2, 10), (64, 0, 3), (160, 1, 5), (160, 2, 10), (160, 0, 4)])
def test_adjoint_fused_chooses_the_kernels_at_every_size(n, fused, vjp):
    d, rn, u, target = _setup(n, n, False, adjoint_fused=fused)
    lat = cm.Lattice(d, rn, u)
    lam = torch.ones((2, 9, n, n), device="cuda")
    before = lat.launches
    lat.step_vjp(lam)
    assert lat.launches - before == vjp
    # a sweep with every state kept: per step the step and the reverse step, whose
    # forward fields the step has written (not for the plane passes); two for the
    # objective, one reduction
    before = lat.launches
    lat.adjoint(3, target, ckpt_every=1)
    per_reverse = {0: 1 if n == 64 else 2, 1: 2, 2: 8}[fused]
    assert lat.launches - before == 3 * (1 + per_reverse) + 3
    lat.close()


# just above 400 000 nodes (fields written by windows), and above 700 000, where
# the row march writes them (16-byte and 4-byte copies)
@pytest.mark.parametrize("nx,ny,wall", [(700, 580, False), (700, 580, True), (1001, 701, False), (1024, 704, True)])
def test_sweep_by_row_wavefronts(nx, ny, wall):
    outs = []
    for fused, K in ((0, 1), (0, 3), (0, 8), (1, 3), (2, 3)):
        d, rn, u, target = _setup(nx, ny, wall, adjoint_fused=fused)
        lat = cm.Lattice(d, rn, u)
        J, g, grn = lat.adjoint(8, target, ckpt_every=K, want_rho_n0=True)
        outs.append((J, list(g.values()), grn.clone()))
        lat.close()
    J0, g0, r0 = outs[0]
    for J, g, r in outs[1:4]:
        assert J == J0 and g == g0
        assert torch.equal(r, r0)
    J2, g2, r2 = outs[4]
    assert J2 == J0
    assert _close(g0, g2), (g0, g2)
    assert (r0 - r2).abs().max() <= 1e-5 * r2.abs().max()


@pytest.mark.parametrize("nx,ny,wall", [(1000, 904, False), (1001, 904, True)])
def test_step_vjp_by_row_wavefronts(nx, ny, wall):
    lam = torch.from_numpy(np.random.default_rng(6).standard_normal((2, 9, ny, nx)).astype(np.float32)).cuda()
    outs = []
    for fused in (0, 2):
        d, rn, u, _ = _setup(nx, ny, wall, adjoint_fused=fused)
        lat = cm.Lattice(d, rn, u)
        v, g = lat.step_vjp(lam)
        outs.append((v.double(), g))
        lat.close()
    (v0, g0), (v2, g2) = outs
    assert _close(g0, g2), (g0, g2)
    assert (v0 - v2).abs().max() <= 1e-5 * v2.abs().max()

"""The forms of one pass that a size rule chooses between: windows of one node
per thread (small lattices, App. B's stencil, the reverse step) and the row
march (large lattices, batches), at the edges of their tiles.

Two forms of the forward step compute the same expressions, so their
populations must be equal bit for bit; the reverse step's forms sum in another
order and are held to the tolerance of the tests that compare its other forms
(1e-5 of each gradient).  Forms that no smaller lattice reaches are compared
with the FP64 oracle at the parity tests' bar for a few steps (2e-6 of the
largest population)."""
import numpy as np
import pytest

from oracle import cmrt_oracle as O
from paper_2005_04642_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU machines too
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2005_04642_gb300 import cmrt as cm  # noqa: E402

cm.load()


def _setup(nx, ny, wall, **kw):
    d = I.base_params(nx, ny, wall_y=wall, g_acc=(1e-5, -2e-5), **kw)
    rn, u = I.random_state_fields(nx, ny, seed=nx + 3 * ny, amplitude=0.02)
    return d, rn.astype(np.float32), u.astype(np.float32)


# own columns of a window: 26 or 24 (one node per thread), 88 or 120 (march);
# own rows 2, 4, 8, 10; widths that copy 16 bytes at a time and that do not
SHAPES = [(24, 8), (25, 9), (26, 10), (27, 11), (53, 21), (88, 40), (89, 5), (176, 23), (120, 64), (121, 12),
          (248, 31), (512, 66)]


@pytest.mark.parametrize("precision", [0, 1, 2], ids=["fp32", "bf16", "fp16"])
@pytest.mark.parametrize("wall", [False, True], ids=["periodic", "walls"])
def test_windows_and_march_give_the_same_bits(precision, wall):
    """A lattice of this size steps by windows; a batch member by the march."""
    members = [_setup(nx, ny, wall, precision=precision) for nx, ny in SHAPES]
    for pick in (slice(None), slice(5, 8), slice(8, 11)):  # 88- and 120-column strips
        b = cm.Batch(members[pick])
        b.step(3)
        for k, m in enumerate(members[pick]):
            lat = cm.Lattice(*m)
            lat.step(3)
            assert torch.equal(b.member(k).populations(), lat.populations()), (m[0]["nx"], m[0]["ny"])
            lat.close()
        b.close()


@pytest.mark.parametrize("nx,ny,wall,order", [(1024, 600, False, 2), (1024, 600, True, 2), (1001, 701, False, 2),
                                              (1001, 701, True, 2), (230, 400, False, 6), (230, 401, True, 6)])
def test_forms_of_larger_lattices_match_oracle(nx, ny, wall, order):
    """The march of a single lattice (16-byte and 4-byte copies) and the taller
    windows of App. B's stencil."""
    d = I.base_params(nx, ny, wall_y=wall, g_acc=(1e-5, -2e-5), stencil_order=order)
    rn = I.drops_field(nx, ny, [(0.3 * nx + 0.3, 0.45 * ny - 0.2), (1.5, 0.6 * ny + 0.4)], [0.2 * min(nx, ny), 40.0],
                       periodic_y=not wall)
    u = I.velocity_noise(nx, ny, 0.01, 7)
    lat = cm.Lattice(d, rn.astype(np.float32), u.astype(np.float32))
    lat.step(3)
    got = lat.populations().double().cpu().numpy()
    p = O.Params(**d)
    R, B = O.init_state(rn.astype(np.float32).astype(np.float64), *u.astype(np.float32).astype(np.float64), p)
    R, B = O.run(R, B, p, 3)
    ref = np.stack([R, B])
    assert np.abs(got - ref).max() <= 2e-6 * np.abs(ref).max()
    lat.close()


@pytest.mark.parametrize("nx,ny,wall", [(64, 64, False), (23, 300, True), (100, 101, False), (131, 90, True),
                                        (300, 260, False), (512, 400, True)])
def test_reverse_step_by_windows_matches_plane_passes(nx, ny, wall):
    """Sweeps whose lattices take the whole form (up to 9000 nodes) and the split
    one with 12 and 16 window rows, with recomputed and with written forward
    fields, and the step VJP, also in place."""
    rn = I.drops_field(nx, ny, [(0.5 * nx + 0.3, 0.5 * ny - 0.2)], [0.25 * min(nx, ny)], periodic_y=not wall)
    target = I.drops_field(nx, ny, [(0.5 * nx + 1.3, 0.5 * ny + 0.3)], [0.25 * min(nx, ny)], periodic_y=not wall)
    u = I.velocity_noise(nx, ny, 0.01, 5).astype(np.float32)
    lam = torch.from_numpy(np.random.default_rng(6).standard_normal((2, 9, ny, nx)).astype(np.float32)).cuda()
    outs = []
    for fused in (0, 2):
        d = I.base_params(nx, ny, wall_y=wall, g_acc=(1e-5, -2e-5), adjoint_fused=fused)
        lat = cm.Lattice(d, rn.astype(np.float32), u)
        v, gv = lat.step_vjp(lam)
        if fused == 0:
            same = lam.clone()
            g2 = cm.cmrt_step_vjp(lat.ctx, same.data_ptr(), same.data_ptr())
            assert torch.equal(same, v) and g2 == gv
        J, g, grn = lat.adjoint(6, target.astype(np.float32), ckpt_every=4, want_rho_n0=True)
        outs.append((J, list(g.values()), gv, grn.double(), v.double()))
        lat.close()
    (J0, g0, gv0, r0, v0), (J2, g2, gv2, r2, v2) = outs
    assert J0 == J2
    for a, b in ((g0, g2), (gv0, gv2)):
        top = max(abs(x) for x in b)
        assert all(abs(x - y) <= 1e-5 * abs(y) + 1e-7 * top for x, y in zip(a, b)), (a, b)
    assert (r0 - r2).abs().max() <= 1e-5 * r2.abs().max()
    assert (v0 - v2).abs().max() <= 1e-5 * v2.abs().max()


@pytest.mark.parametrize("precision", [1, 2], ids=["bf16", "fp16"])
def test_march_with_4_byte_copies_gives_the_bits_of_16_byte_ones(precision):
    """An odd width beyond the windows' range, a flow that is uniform along x: each
    column equals any column of a lattice whose width is a multiple of 4."""
    cols = []
    for nx in (757, 760):
        d = I.base_params(nx, 600, wall_y=False, g_acc=(1e-5, -2e-5), precision=precision)
        rn = np.repeat(np.tanh(np.sin(2 * np.pi * np.arange(600) / 600) * 20)[:, None], nx, 1).astype(np.float32)
        lat = cm.Lattice(d, rn, None)
        lat.step(3)
        p = lat.populations()
        assert torch.equal(p, p[..., :1].expand_as(p))
        cols.append(p[..., 0])
        lat.close()
    assert torch.equal(*cols)


@pytest.mark.parametrize("g", [1e-24, 1e-14, 1e-3, 1e19], ids=str)
@pytest.mark.parametrize("precision", [0, 2], ids=["fp32", "fp16"])
def test_diagnosed_speed_over_the_range_of_fp32(g, precision):
    """max|u| where |u|^2 is below, within and above FP32's range, against the
    fields' u: the two forms may round u by a few FP32 spacings differently."""
    d = I.base_params(40, 24, wall_y=False, g_acc=(g, -2.0 * g), precision=precision)
    lat = cm.Lattice(d, np.ones((24, 40), np.float32), None)
    f = lat.fields()
    want = float(torch.hypot(f["ux"].double(), f["uy"].double()).max())
    assert want >= g
    assert lat.diagnostics()["umax"] == pytest.approx(want, rel=1e-6, abs=0.0)
    lat.close()


# all widths copy 16 bytes at a time: strips of 88 own columns (96-column windows) and of 120
@pytest.mark.parametrize("precision", [0, 1, 2], ids=["fp32", "bf16", "fp16"])
@pytest.mark.parametrize("walls", [(False, False), (True, True), (False, True)], ids=["periodic", "walls", "mixed"])
@pytest.mark.parametrize("shapes", [[(88, 40), (176, 23), (256, 70), (84, 9)], [(120, 64), (240, 31), (112, 5)]],
                         ids=["window96", "window128"])
def test_batches_with_16_byte_copies_give_the_bits_of_windows(shapes, walls, precision):
    members = [_setup(nx, ny, walls[k % 2], precision=precision) for k, (nx, ny) in enumerate(shapes)]
    b = cm.Batch(members)
    b.step(3)
    for k, m in enumerate(members):
        lat = cm.Lattice(*m)
        lat.step(3)
        assert torch.equal(b.member(k).populations(), lat.populations()), (m[0]["nx"], m[0]["ny"])
        lat.close()
    b.close()


# App. B's stencil: lattices of one window's height (periodic rows that wrap inside
# it, walls), window heights chosen for the lattice's (33 and 40 rows), 22 and 24
# own columns
@pytest.mark.parametrize("nx,ny,wall", [(25, 1, False), (30, 2, False), (44, 3, True), (23, 5, False), (67, 31, True),
                                        (45, 32, False), (24, 32, True), (1900, 33, False), (1900, 40, False)])
def test_order6_windows_of_low_lattices_match_oracle(nx, ny, wall):
    d = I.base_params(nx, ny, wall_y=wall, g_acc=(1e-5, -2e-5), stencil_order=6)
    y, x = np.mgrid[0:ny, 0:nx]
    rn = np.tanh(3.0 * np.sin(2 * np.pi * x / nx + 0.3) * (1.0 if ny < 8 else np.cos(np.pi * y / ny) + 0.4))
    u = I.velocity_noise(nx, ny, 0.01, 7)
    lat = cm.Lattice(d, rn.astype(np.float32), u.astype(np.float32))
    lat.step(3)
    got = lat.populations().double().cpu().numpy()
    p = O.Params(**d)
    R, B = O.init_state(rn.astype(np.float32).astype(np.float64), *u.astype(np.float32).astype(np.float64), p)
    R, B = O.run(R, B, p, 3)
    ref = np.stack([R, B])
    assert np.abs(got - ref).max() <= 2e-6 * np.abs(ref).max()
    f, got = lat.fields(), lat.diagnostics()
    assert got["mass_r"] == pytest.approx(R.sum(), rel=2e-6) and got["mass_b"] == pytest.approx(B.sum(), rel=2e-6)
    assert got["umax"] == pytest.approx(float(torch.hypot(f["ux"].double(), f["uy"].double()).max()), rel=1e-6)
    if not wall:
        # the same rows again and again, on a lattice of windows with halo rows: the same bits
        k = 66 // ny + 1
        tall = cm.Lattice(dict(d, ny=k * ny), np.tile(rn, (k, 1)).astype(np.float32), np.tile(u, (1, k, 1)).astype(np.float32))
        tall.step(3)
        assert torch.equal(tall.populations(), lat.populations().tile(1, 1, k, 1))
        for name, v in tall.fields().items():
            assert torch.equal(v, f[name].tile(k, 1)), name
        tall.close()
    lat.close()

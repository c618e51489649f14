"""Edge sizes of the kernels' tiles, items and dispatch rules against plain FP64 references."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _sim(shape, dtype="f32", dims=3, **kw):
    from paper_1710_06829_gb300 import inputs
    from paper_1710_06829_gb300 import sim as S
    beta, delta = inputs.isotropic_theta(-0.05, -0.04, 0.02, 0.01)
    return S.Simulation(shape, [1.0, 1.0, 1.0], 0.4, beta, delta, dims=dims, dtype=dtype, **kw)


def _random_state(shape, dtype, seed=0):
    """Six seeded fields rounded to the dtype, as FP64 arrays."""
    from paper_1710_06829_gb300 import inputs
    np_t = np.float32 if dtype == "f32" else np.float64
    return [f.astype(np_t).astype(np.float64) for f in inputs.random_fields(shape, seed)]


# one row, one column group, a ragged last item (17 rows), several planes, more items than a wave
PROJECTION_SHAPES = [((4, 1, 1), 1), ((8, 17, 1), 2), ((12, 16, 5), 3), ((68, 33, 3), 3),
                     ((256, 130, 40), 3)]


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("shape,dims", PROJECTION_SHAPES)
def test_projections_match_direct_sums(shape, dims, dtype):
    """Plane-wave amplitude, energy moments and window energy against direct FP64 sums.  The sums
    have n terms of relative error a few eps, so n eps sum|term| bounds the difference; 1e-13
    sum|term| (about 500 eps) holds with room for the pairwise-like order used."""
    from paper_1710_06829_gb300 import inputs
    nx, ny, nz = shape
    f = _random_state(shape, dtype)
    sm = _sim(shape, dtype, dims)
    sm.set_state([torch.from_numpy(a) for a in f])
    for comp, k in ((0, (0.3, -0.7, 1.1)), (5, (2.9, 0.01, -3.0))):
        x, y, z = inputs.positions(shape, comp, [1.0, 1.0, 1.0])
        ref = np.sum(f[comp] * np.exp(-1j * (k[0] * x + k[1] * y + k[2] * z)))
        for _ in range(2):   # the block ticket is back at zero after the first launch
            got = sm.plane_wave(comp, k).cpu().numpy()
            assert abs(got[0] + 1j * got[1] - ref) <= 1e-13 * np.sum(np.abs(f[comp]))
    for axis in range(3):
        n = shape[axis]
        ref = np.zeros(3)
        for c in range(6):
            th = 2 * math.pi * inputs.positions(shape, c, [1.0, 1.0, 1.0])[axis] / n
            e = 0.5 * f[c] ** 2
            ref += [e.sum(), (e * np.cos(th)).sum(), (e * np.sin(th)).sum()]
        got = sm.energy_moments(axis).cpu().numpy()
        assert np.all(np.abs(got - ref) <= 1e-13 * ref[0])
    ref = 0.5 * sum(np.sum(np.take(a, range(-3, nx - 4), axis=2, mode="wrap") ** 2) for a in f)
    got = float(sm.energy(-3, nx - 1).cpu())
    assert abs(got - ref) <= 1e-13 * ref
    sm.close()


def test_plane_wave_of_denormals_and_non_finite_values():
    """The integer widening of the FP32 projection: denormal floats keep their values, an infinity or
    a NaN reaches the sums as the plain conversion would bring it there."""
    shape = (8, 20, 2)
    f = torch.zeros((2, 20, 8), dtype=torch.float32)
    f[1, 19, 5], f[0, 3, 2], f[1, 7, 0] = 3e-42, -1e-44, 2e-39
    sm = _sim(shape)
    for bad in (None, math.inf, math.nan):
        if bad is not None:
            f[0, 17, 6] = bad
        sm.set_state([None, None, f, None, None, None])
        re, im = sm.plane_wave(2, (0.0, 0.0, 0.0)).cpu().tolist()
        ref = float(f.double().sum())
        if bad is None:
            assert abs(re - ref) <= 1e-15 * abs(ref) and im == 0.0
        else:
            assert math.isnan(re) if math.isnan(ref) else re == ref
    sm.close()


@pytest.mark.parametrize("scale", [1.4e-45, 1e-42, 1e-38, 1e-36, 1e-30])
def test_plane_wave_of_tiny_fields(scale):
    """Fields of a few denormal steps up to small normal ones, with a phase, one column group of ordinary
    size among those of the second plane: tolerance of test_projections_match_direct_sums."""
    from paper_1710_06829_gb300 import inputs
    shape = (24, 35, 2)
    f = np.random.default_rng(12).integers(-40, 41, size=shape[::-1]).astype(np.float64) * scale
    f[1, 20, 4:8] *= 1e6
    f = f.astype(np.float32).astype(np.float64)
    sm = _sim(shape)
    sm.set_state([torch.from_numpy(f)] + [None] * 5)
    for k in ((0.3, -0.7, 1.1), (2.9, 0.01, -3.0)):
        x, y, z = inputs.positions(shape, 0, [1.0, 1.0, 1.0])
        ph = np.exp(-1j * (k[0] * x + k[1] * y + k[2] * z))
        for part in (f, np.where(np.arange(2)[:, None, None] == 0, f, 0.0)):   # both planes, one of them
            sm.set_state([torch.from_numpy(part)] + [None] * 5)
            got = sm.plane_wave(0, k).cpu().numpy()
            assert abs(got[0] + 1j * got[1] - np.sum(part * ph)) <= 1e-13 * np.sum(np.abs(part))
    sm.close()


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("shape,dims", [((4, 1, 1), 1), ((8, 3, 1), 2), ((260, 5, 7), 3), ((68, 130, 9), 3)])
def test_state_round_trip_is_exact(shape, dims, dtype, offset):
    """set_state / get_state through the padded layout, dense arrays that start on a 16-byte boundary
    and one element past it, a NULL component; one step after it equals the step from host memory
    (whose images come from another kernel)."""
    nx, ny, nz = shape
    tt = torch.float32 if dtype == "f32" else torch.float64
    f = [torch.from_numpy(a).to(tt) for a in _random_state(shape, dtype, 5)]
    f[3] = None
    dev = []
    for a in f:
        if a is None:
            dev.append(None)
            continue
        buf = torch.empty(a.numel() + offset, dtype=tt, device="cuda")[offset:].view(a.shape)
        buf.copy_(a)
        dev.append(buf)
    sm, ref = _sim(shape, dtype, dims), _sim(shape, dtype, dims)
    sm.set_state(dev)
    out = [torch.full((nx * ny * nz + offset,), 7.0, dtype=tt, device="cuda")[offset:].view(nz, ny, nx)
           for _ in range(6)]
    from paper_1710_06829_gb300 import _lib as L
    L.fdtd_get_state(sm.h, [t.data_ptr() for t in out], L.FDTD_MEM_DEVICE)
    torch.cuda.synchronize()
    for a, b in zip(f, out):
        assert torch.equal(b.cpu(), torch.zeros_like(b, device="cpu") if a is None else a)
    ref.set_state_host(f)
    sm.step(1)
    ref.step(1)
    for a, b in zip(sm.get_state(), ref.get_state()):
        assert torch.equal(a, b)
    sm.close()
    ref.close()


# one point, segments shorter than the minimum, a ragged last segment, rows that do not fill a
# block, empty rows under the cone, dt^2 S near 1 at the last points
NORM_CASES = [(1, (3, 1, 1), 0.9), (1, (4096, 1, 1), 0.9999), (2, (1, 7, 1), 0.9), (2, (67, 5, 1), 0.9),
              (2, (130, 129, 1), 0.9999), (3, (33, 2, 70), 0.95), (3, (70, 64, 3), 0.95)]


@pytest.mark.parametrize("weight,par", [(0, 0.0), (1, math.radians(30)), (1, math.radians(3)),
                                        (1, math.radians(120)), (2, 0.1)])
@pytest.mark.parametrize("dims,N,courant", NORM_CASES)
def test_norm_segments_and_weights_match_oracle(dims, N, courant, weight, par):
    """Row segments, cone starts and the angle table.  omega has a relative error of a few eps
    divided by sqrt(1 - dt^2 S), as in the plain formulas; rel 1e-11 covers it."""
    from oracle import dispersion as D
    from paper_1710_06829_gb300 import inputs
    from paper_1710_06829_gb300 import sim as S
    beta, delta = np.zeros((3, 3)), np.zeros(3)
    if dims > 1:
        beta, delta = inputs.isotropic_theta(-0.05, -0.04, 0.02, 0.01)
    dx = [1.0, 1.2, 0.9]
    dt = courant * D.dt_max(beta, delta, dx, dims)
    f, gb, gd, gdt = S.disp_norm(beta, delta, dt, dx, dims, N, weight, par)
    kind = (D.WEIGHT_UNIFORM, D.WEIGHT_CONE_X, D.WEIGHT_GAUSS_Y)[weight]
    rf, rgb, rgd, rgdt = D.norm_and_grad(beta, delta, dt, dx, N, dims, kind, par)
    got = np.r_[f, np.ravel(gb), gd, gdt]
    ref = np.r_[rf, np.ravel(rgb), rgd, rgdt]
    assert np.all(np.abs(got - ref) <= 1e-11 * np.abs(ref) + 1e-13 * max(1.0, abs(rf)))


@pytest.mark.parametrize("weight,par", [(0, 0.0), (1, math.radians(30))])
@pytest.mark.parametrize("e", [-250, -140, 140, 250])
def test_norm_of_wave_numbers_outside_the_float_range(e, weight, par):
    """Spacings of 1 and 2^e: the wave numbers of one axis lie outside single precision's range, in which
    the cone's test is made where it can be.  Yee's scheme; tolerance as above."""
    from oracle import dispersion as D
    from paper_1710_06829_gb300 import sim as S
    beta, delta, dx, N = np.zeros((3, 3)), np.zeros(3), [1.0, 2.0 ** e, 1.0], (40, 33, 1)
    dt = 0.9 * D.dt_max(beta, delta, dx, 2)
    f, gb, gd, gdt = S.disp_norm(beta, delta, dt, dx, 2, N, weight, par)
    rf, rgb, rgd, rgdt = D.norm_and_grad(beta, delta, dt, dx, N, 2, (D.WEIGHT_UNIFORM, D.WEIGHT_CONE_X)[weight], par)
    got, ref = np.r_[f, np.ravel(gb), gd, gdt], np.r_[rf, np.ravel(rgb), rgd, rgdt]
    assert np.all(np.abs(got - ref) <= 1e-11 * np.abs(ref) + 1e-13 * max(1.0, abs(rf)))


def test_norm_from_several_threads_and_streams():
    """More concurrent evaluations than scratch areas: every one returns its own value."""
    import threading

    from paper_1710_06829_gb300 import sim as S
    beta, delta = np.zeros((3, 3)), np.zeros(3)
    args = [(0.3 + 0.02 * i, [1.0, 1.0, 1.0], 2, (200 + i, 150, 1)) for i in range(8)]
    ref = [S.disp_norm(beta, delta, *a)[0] for a in args]
    bad = []

    def work(i):
        st = torch.cuda.Stream()
        for _ in range(20):
            if S.disp_norm(beta, delta, *args[i], stream=st)[0] != ref[i]:
                bad.append(i)
    th = [threading.Thread(target=work, args=(i,)) for i in range(len(args))]
    for t in th:
        t.start()
    for t in th:
        t.join()
    assert not bad


def _step_pair(shape, dtype, monkeypatch, steps=5, dims=3, **kw):
    """The state after `steps` steps with the tiled and with the reference-form kernels."""
    from paper_1710_06829_gb300 import sim as S
    f = [torch.from_numpy(a) for a in _random_state(shape, dtype, 11)]
    out = []
    for flag in ("1", "0"):
        monkeypatch.setenv("FDTD_FUSED", flag)
        sm = _sim(shape, dtype, dims, **kw)
        sm.set_state(f)
        src = None
        if not kw.get("batched"):
            src = S.Bunch(1.0, 0.9, 3.0, 2.0, 1.0, 2.0, 2.0)
        sm.step(steps, source=src)
        sm.sync()
        out.append(sm.get_state())
        sm.close()
    return out


# narrowest grids, last tiles of one column group or one row, ghosts of the last cells in the same
# and in a further tile, the fewest planes, more planes than a z-chunk
RAGGED = [(8, 4, 4), (60, 12, 5), (64, 9, 4), (68, 8, 7), (132, 31, 4), (124, 30, 40), (300, 20, 70)]


@pytest.mark.parametrize("sponge", [False, True])
@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("shape", RAGGED)
def test_ragged_tiles_step_bitwise_like_the_reference_form(shape, dtype, sponge, monkeypatch):
    if sponge and min(shape[1:]) < 4:
        pytest.skip("no room for the layers")
    kw = dict(absorb_cells=2, absorb_sigma=0.3) if sponge else {}
    for a, b in zip(*_step_pair(shape, dtype, monkeypatch, **kw)):
        assert torch.equal(a, b)


@pytest.mark.parametrize("shape", [(4, 2, 2), (4, 16, 3), (32, 3, 9), (64, 48, 33)])
def test_fp64_step_on_grids_inside_one_tile_and_whole_tiles(shape, monkeypatch):
    for a, b in zip(*_step_pair(shape, "f64", monkeypatch)):
        assert torch.equal(a, b)


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("shape", [(8, 1, 1), (12, 15, 17), (64, 16, 17), (8, 700, 600)])
def test_probe_loss_sums_the_plane(shape, dtype):
    """One value, a ragged block, more values than threads in a wave; added to what is there.  Sums of
    n positive terms in FP64: n eps relative, 1e-12 taken for up to 4e5."""
    from paper_1710_06829_gb300 import sim as S
    nx, ny, nz = shape
    f = _random_state(shape, dtype, 21)
    tt = torch.float32 if dtype == "f32" else torch.float64
    tgt = torch.from_numpy(np.random.default_rng(4).standard_normal((2, nz, ny))).to(tt).cuda()
    sm = _sim(shape, dtype, 1 if ny == 1 else 3)
    sm.set_state([torch.from_numpy(a) for a in f])
    loss = torch.full((1,), 3.0, dtype=torch.float64, device="cuda")
    ref = 3.0
    for s in range(2):
        sm.step(1, probe=S.Probe(2, nx - 1, tgt), loss=loss)
        ref += float(((sm.get_state()[2][:, :, nx - 1].double() - tgt[s].double()) ** 2).sum())
    assert abs(float(loss) - ref) <= 1e-12 * ref
    sm.close()


# narrowest plane, whole tiles, last tiles of one column group or one row, tall and wide planes
@pytest.mark.parametrize("nz,batched", [(1, False), (3, True), (1, None)])
@pytest.mark.parametrize("nx,ny", [(8, 4), (64, 16), (68, 17), (60, 33), (1000, 5), (12, 300)])
@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_planes_step_bitwise_like_the_reference_form(nx, ny, nz, batched, dtype, monkeypatch):
    """The 2D kernels on one plane (2D, and 3D one plane thick: batched None) and on a batch with its
    layers on y; the one-plane runs carry the bunch current."""
    kw = dict(batched=True, absorb_cells=2, absorb_sigma=0.3) if batched else {}
    for a, b in zip(*_step_pair((nx, ny, nz), dtype, monkeypatch, dims=3 if batched is None else 2, **kw)):
        assert torch.equal(a, b)


@pytest.mark.parametrize("shape,batched", [((1004, 701, 1), False), ((68, 33, 320), True),
                                           ((1004, 701, 1), None), ((512, 1368, 1), False)])
def test_large_fp64_planes_step_bitwise_like_the_reference_form(shape, batched, monkeypatch):
    """As above from 700000 cells on, where the FP64 kernel takes its large tile: ragged in both directions,
    a batch with layers, a 3D problem one plane thick, whole tiles."""
    kw = dict(batched=True, absorb_cells=2, absorb_sigma=0.3) if batched else {}
    for a, b in zip(*_step_pair(shape, "f64", monkeypatch, dims=3 if batched is None else 2, **kw)):
        assert torch.equal(a, b)


# one warp, a ragged warp, several blocks; particles of one cell moving across no, one or three faces
# and both ways along an axis (momenta along the cell's diagonal, or random), grids of a few cells, the
# per-cell mean of B (at least 2^20 particles and one per cell)
@pytest.mark.parametrize("sponge", [False, True])
@pytest.mark.parametrize("shape,n,kind", [
    ((8, 6, 5), 32, "diagonal"), ((8, 6, 5), 33, "random"), ((4, 4, 4), 700, "random"),
    ((12, 8, 6), 64, "still"), ((8, 8, 8), 96, "along"), ((16, 12, 10), 5000, "random"),
    ((32, 20, 16), 1 << 20, "random")])
def test_push_and_current_match_the_oracle(shape, n, kind, sponge):
    """Three cycles in FP64 against the oracle: every sum has at most n / cells + 60 terms a step, each
    with a few eps; 1e-10 of the largest value covers 2^20 particles on 10^4 cells."""
    from oracle import dispersion as D
    from oracle import fdtd as F
    from oracle import pic as P
    from paper_1710_06829_gb300 import inputs
    from paper_1710_06829_gb300 import sim as S
    if n > 100000 and sponge:
        pytest.skip("one large run is enough")
    nx, ny, nz = shape
    beta, delta = inputs.isotropic_theta(-0.05, -0.04, 0.02, 0.01)
    dx = [1.0, 1.1, 0.9]
    dt = 0.95 * D.dt_max(beta, delta, dx, 3)
    rng = np.random.default_rng(n)
    L = np.array([nx * dx[0], ny * dx[1], nz * dx[2]])[:, None]
    if kind == "random":
        x, u = rng.uniform(0, 1, (3, n)) * L, 2.0 * rng.standard_normal((3, n))
    else:   # all in one cell
        x = (rng.uniform(0, 1, (3, n)) + np.array([[nx - 1], [1], [0]])) * np.array(dx)[:, None]
        d = {"diagonal": (4.0, 4.0, -4.0), "still": (0.0, 0.0, 0.0), "along": (9.0, 0.1, 0.0)}[kind]
        u = np.repeat(np.array(d)[:, None], n, axis=1)
    x[:, 0] = 0.0
    f = [0.1 * a for a in inputs.random_fields(shape, 7)]
    kw = dict(absorb_cells=2, absorb_sigma=0.3) if sponge else {}
    sm = S.Simulation(shape, dx, dt, beta, delta, dtype="f64", **kw)
    sm.set_state([torch.from_numpy(a) for a in f])
    q = 1.0 / max(1, n // 100)
    sp = S.Species(torch.from_numpy(x.copy()).cuda(), torch.from_numpy(u.copy()).cuda(), q, -1.0)
    st, pt = F.State(f[:3], f[3:]), P.Particles(x, u, q, -1.0)
    fac = F.sponge_factor((nz, ny, nx), 2, 0.3) if sponge else None
    c = F.Coeffs(beta, delta, dx, dt)
    for _ in range(3):
        st = P.pic_step(st, [pt], c, fac)
    sm.pic_step(3, [sp])
    sm.sync()
    got = [t.cpu().numpy() for t in sm.get_state()]
    for a, b in zip(got, st.E + st.B):
        assert np.max(np.abs(a - b)) <= 1e-10 * max(np.max(np.abs(v)) for v in st.E + st.B)
    d = np.abs(sp.x.cpu().numpy() - pt.x)
    assert np.max(np.minimum(d, L - d)) <= 1e-9   # a position on the seam may sit at either end
    assert np.max(np.abs(sp.u.cpu().numpy() - pt.u)) <= 1e-9 * np.max(np.abs(pt.u)) + 1e-9
    sm.close()


@pytest.mark.parametrize("sponge", [False, True])
@pytest.mark.parametrize("shape", RAGGED + [(4, 2, 2), (4, 3, 5), (32, 3, 9), (64, 48, 33)])
def test_fp64_reverse_step_matches_the_reference_form(shape, sponge, monkeypatch):
    """lambda and the coefficient gradient of three recorded steps, with a probe on the last column.
    Per value about 40 FP64 operations a reverse step on terms of the field's size: 3 x 40 x 2^-53 =
    1.3e-14 of the largest value; 1e-13 taken, and for the gradient's sums of up to 4e5 terms 1e-11
    of the largest entry."""
    if sponge and min(shape[1:]) < 4:
        pytest.skip("no room for the layers")
    from paper_1710_06829_gb300 import sim as S
    kw = dict(absorb_cells=2, absorb_sigma=0.3) if sponge else {}
    f = [torch.from_numpy(a) for a in _random_state(shape, "f64", 12)]
    lam = [torch.from_numpy(a) for a in _random_state(shape, "f64", 13)]
    nx, ny, nz = shape
    tgt = torch.from_numpy(np.random.default_rng(3).standard_normal((3, nz, ny))).cuda()
    out = []
    for flag in ("1", "0"):
        monkeypatch.setenv("FDTD_FUSED", flag)
        sm = _sim(shape, "f64", **kw)
        sm.set_state(f)
        sm.step(3, record=True)
        sm.set_adjoint(lam)
        grad = torch.zeros(12, dtype=torch.float64, device="cuda")
        sm.step_adjoint(3, grad, probe=S.Probe(1, nx - 1, tgt))
        out.append((sm.get_adjoint(), grad.cpu()))
        sm.sync()
        sm.close()
    for a, b in zip(out[0][0], out[1][0]):
        assert float((a - b).abs().max()) <= 1e-13 * max(float(c.abs().max()) for c in out[1][0])
    assert float((out[0][1] - out[1][1]).abs().max()) <= 1e-11 * float(out[1][1].abs().max())


@pytest.mark.parametrize("shape,dims,kw", [
    ((64, 8, 1), 2, {}), ((64, 16, 1), 3, {}), ((128, 24, 2), 2, dict(batched=True)),
    ((192, 8, 17), 2, dict(batched=True)), ((64, 40, 70), 2, dict(batched=True)),
    ((128, 16, 9), 2, dict(batched=True, absorb_cells=3, absorb_sigma=0.3))])
def test_fp32_reverse_step_of_planes_matches_fp64(shape, dims, kw, monkeypatch):
    """lambda and the gradient of three recorded steps, with a probe on the last column, against the
    FP64 reference form on the same FP32 inputs.  Per value about 20 FP32 operations a step on terms
    of the field's size, forward and back: 6 x 20 x 2^-24 = 7e-6 of the largest value, 2e-5 taken;
    the gradient's terms carry that error with random signs, like the terms themselves: 1e-4 of
    the largest entry."""
    from paper_1710_06829_gb300 import sim as S
    f = [torch.from_numpy(a) for a in _random_state(shape, "f32", 14)]
    lam = [torch.from_numpy(a) for a in _random_state(shape, "f32", 15)]
    nx, ny, nz = shape
    tgt = torch.from_numpy(np.random.default_rng(4).standard_normal((3, nz, ny)).astype(np.float32)).cuda()
    out = []
    for flag, dtype, tt in (("1", "f32", torch.float32), ("0", "f64", torch.float64)):
        monkeypatch.setenv("FDTD_FUSED", flag)
        sm = _sim(shape, dtype, dims=dims, **kw)
        sm.set_state([t.to(tt) for t in f])
        sm.step(3, record=True)
        sm.set_adjoint([t.to(tt) for t in lam])
        grad = torch.zeros(12, dtype=torch.float64, device="cuda")
        sm.step_adjoint(3, grad, probe=S.Probe(1, nx - 1, tgt.to(tt)))
        out.append(([t.double() for t in sm.get_adjoint()], grad.cpu()))
        sm.sync()
        sm.close()
    for a, b in zip(out[0][0], out[1][0]):
        assert float((a - b).abs().max()) <= 2e-5 * max(float(c.abs().max()) for c in out[1][0])
    assert float((out[0][1] - out[1][1]).abs().max()) <= 1e-4 * float(out[1][1].abs().max())


@pytest.mark.parametrize("sponge", [False, True])
@pytest.mark.parametrize("n", [1 << 20, (1 << 20) + 77])
def test_push_of_many_particles_matches_that_of_few(n, sponge):
    """1000 charged particles alone, and beside n neutral ones that only drift: the second call takes
    the push for many particles (B once per cell, one large block an SM).  Positions of up to 32 cells
    differ by a few units of 2^-19 cells (B's rounding, three cycles); a deposit of charge 0.01 by as
    much of it, far below 1e-5 of fields of 0.3."""
    from paper_1710_06829_gb300 import inputs
    from paper_1710_06829_gb300 import sim as S
    shape = (32, 12, 16)
    rng = np.random.default_rng(8)
    ext = np.array(shape)[:, None]
    def species(m, q, qm):
        x = (rng.uniform(0, 0.999, (3, m)) * ext).astype(np.float32)
        u = rng.standard_normal((3, m)).astype(np.float32)
        return x, u, q, qm
    few, many = species(1000, 0.01, -1.0), species(n, 0.0, 0.0)
    f = [torch.from_numpy(0.1 * a).float() for a in inputs.random_fields(shape, 7)]
    out = []
    for sps in ([few], [few, many]):
        sm = _sim(shape, "f32", **(dict(absorb_cells=2, absorb_sigma=0.3) if sponge else {}))
        sm.set_state(f)
        sp = [S.Species(torch.from_numpy(x.copy()).cuda(), torch.from_numpy(u.copy()).cuda(), q, qm)
              for x, u, q, qm in sps]
        sm.pic_step(3, sp)
        sm.sync()
        out.append((sm.get_state(), sp))
        sm.close()
    big = max(float(t.abs().max()) for t in out[0][0])
    for a, b in zip(out[0][0], out[1][0]):
        assert float((a - b).abs().max()) <= 1e-5 * big
    L = torch.tensor(shape, dtype=torch.float64, device="cuda")[:, None]

    def far(a, b):   # a position on the seam may sit at either end
        d = (a.double() - b.double()).abs()
        return float(torch.minimum(d, L - d).max())
    a, b = out[0][1][0], out[1][1][0]
    assert far(a.x, b.x) <= 1e-4 and float((a.u - b.u).abs().max()) <= 1e-5 * float(a.u.abs().max())
    x, u = (torch.from_numpy(v).double().cuda() for v in many[:2])
    assert torch.equal(out[1][1][1].u, torch.from_numpy(many[1]).cuda())
    x = torch.remainder(x + 3 * 0.4 * u / torch.sqrt(1 + (u * u).sum(0)), L)
    assert far(out[1][1][1].x, x) <= 1e-4


@pytest.mark.parametrize("shape,dims,kw", [
    ((8, 4, 1), 3, {}), ((8, 5, 2), 3, {}), ((12, 9, 3), 3, {}), ((68, 33, 21), 3, {}),
    ((132, 7, 5), 2, dict(batched=True)), ((36, 20, 30), 3, dict(absorb_cells=4, absorb_sigma=0.3))])
def test_fp32_reverse_step_of_ragged_grids_matches_fp64(shape, dims, kw, monkeypatch):
    """As above, on grids without whole tiles: down to the smallest that the kernel of four cells a
    thread takes, one to three planes, layers."""
    test_fp32_reverse_step_of_planes_matches_fp64(shape, dims, kw, monkeypatch)


def test_fp64_grids_of_more_planes_than_chunks_on_one_grid_axis(monkeypatch):
    """More z-chunks than a grid's y axis has blocks (chunks of at most 64 planes, 65535 blocks): two
    recorded steps and the reverse steps against the reference form, whose kernels loop over planes.
    Tolerances as in test_fp64_reverse_step_matches_the_reference_form."""
    from paper_1710_06829_gb300 import sim as S
    shape = (4, 1, 64 * 65535 + 70)
    if torch.cuda.mem_get_info()[0] < 90 * 2 ** 30:
        pytest.skip("needs 90 GB of free device memory")
    gen = torch.Generator(device="cuda").manual_seed(9)
    f, lam = ([torch.randn(shape[::-1], generator=gen, device="cuda", dtype=torch.float64) for _ in range(6)]
              for _ in range(2))
    out = []
    for flag in ("1", "0"):
        monkeypatch.setenv("FDTD_FUSED", flag)
        sm = _sim(shape, "f64")
        sm.set_state(f)
        sm.step(2, record=True)
        state = sm.get_state()
        sm.set_adjoint(lam)
        grad = torch.zeros(12, dtype=torch.float64, device="cuda")
        sm.step_adjoint(2, grad)
        out.append((state, sm.get_adjoint(), grad))
        sm.sync()
        sm.close()
    for a, b in zip(out[0][0], out[1][0]):
        assert torch.equal(a, b)
    for a, b in zip(out[0][1], out[1][1]):
        assert float((a - b).abs().max()) <= 1e-13 * max(float(c.abs().max()) for c in out[1][1])
    assert float((out[0][2] - out[1][2]).abs().max()) <= 1e-11 * float(out[1][2].abs().max())


@pytest.mark.parametrize("sponge", [False, True])
@pytest.mark.parametrize("shape,per,extra", [((32, 32, 32), 32, 0), ((32, 16, 32), 64, 77)])
def test_push_of_many_particles_in_cell_order_matches_the_oracle(shape, per, extra, sponge):
    """FP32, at least 2^20 charged particles, whole warps in one cell: their currents are summed through
    the shared rows of all 24 warps of the large block.  By cell, particles at rest, moving along x,
    along the diagonal (over one to three faces, some and not others) and every way; extra particles
    shift the last warps off the cells.  Against the FP64 oracle on the same FP32 inputs: positions of up
    to 32 cells are rounded to 2^-20 of a cell where a particle moves by 0.4, so a face's sum is good to
    about 5e-6 of its terms, fields included; 5e-5 of the largest value taken."""
    from oracle import dispersion as D
    from oracle import fdtd as F
    from oracle import pic as P
    from paper_1710_06829_gb300 import inputs
    from paper_1710_06829_gb300 import sim as S
    nx, ny, nz = shape
    beta, delta = inputs.isotropic_theta(-0.05, -0.04, 0.02, 0.01)
    dx = [1.0, 1.0, 1.0]
    dt = 0.95 * D.dt_max(beta, delta, dx, 3)
    rng = np.random.default_rng(per)
    cells = nx * ny * nz
    c = np.repeat(np.arange(cells), per)
    n = c.size
    origin = np.array([c % nx, c // nx % ny, c // (nx * ny)], dtype=np.float64)
    x = (origin + rng.uniform(0.0, 0.999, (3, n))).astype(np.float32)
    way = rng.choice([-1.0, 1.0], (3, cells))[:, c]
    kinds = np.stack([np.zeros((3, n)), way * np.array([[4.0], [0.0], [0.0]]), 3.0 * way,
                      3.0 * rng.standard_normal((3, n))])
    u = np.take_along_axis(kinds, (c % 4)[None, None, :], axis=0)[0].astype(np.float32)
    if extra:
        x = np.concatenate([x[:, :1000], rng.uniform(0.0, 0.999, (3, extra)).astype(np.float32), x[:, 1000:]], axis=1)
        u = np.concatenate([u[:, :1000], np.zeros((3, extra), np.float32), u[:, 1000:]], axis=1)
    f = [(0.01 * a).astype(np.float32) for a in inputs.random_fields(shape, 8)]
    kw = dict(absorb_cells=4, absorb_sigma=0.3) if sponge else {}
    q = 1.0 / per
    sm = S.Simulation(shape, dx, dt, beta, delta, dtype="f32", **kw)
    sm.set_state([torch.from_numpy(a) for a in f])
    sp = S.Species(torch.from_numpy(x.copy()).cuda(), torch.from_numpy(u.copy()).cuda(), q, -1.0)
    sm.pic_step(1, [sp])
    sm.sync()
    got = [t.double().cpu().numpy() for t in sm.get_state()]
    sm.close()
    f64 = [a.astype(np.float64) for a in f]
    st, pt = F.State(f64[:3], f64[3:]), P.Particles(x.astype(np.float64), u.astype(np.float64), q, -1.0)
    fac = F.sponge_factor((nz, ny, nx), 4, 0.3) if sponge else None
    st = P.pic_step(st, [pt], F.Coeffs(beta, delta, dx, dt), fac)
    big = max(float(np.max(np.abs(v))) for v in st.E)
    assert big > 0.1   # the currents, not the fields of 0.01
    for a, b in zip(got, st.E + st.B):
        assert np.max(np.abs(a - b)) <= 5e-5 * big


@pytest.mark.parametrize("shape,dims,kw", [
    ((64, 8, 1), 2, {}), ((64, 16, 1), 3, {}), ((192, 8, 17), 2, dict(batched=True)),
    ((128, 24, 70), 2, dict(batched=True, absorb_cells=3, absorb_sigma=0.3))])
def test_fp32_reverse_step_of_planes_is_bitwise_that_of_the_3d_kernels(shape, dims, kw, monkeypatch):
    """lambda of the 2D kernel against the two-kernel 3D form, which forms every value in the same order."""
    from paper_1710_06829_gb300 import sim as S
    f = [torch.from_numpy(a) for a in _random_state(shape, "f32", 16)]
    lam = [torch.from_numpy(a) for a in _random_state(shape, "f32", 17)]
    nx, ny, nz = shape
    tgt = torch.from_numpy(np.random.default_rng(5).standard_normal((3, nz, ny)).astype(np.float32)).cuda()
    out = []
    for flag in ("0", "1"):
        monkeypatch.setenv("FDTD_ADJOINT_SPLIT", flag)
        sm = _sim(shape, "f32", dims=dims, **kw)
        sm.set_state(f)
        sm.step(3, record=True)
        sm.set_adjoint(lam)
        grad = torch.zeros(12, dtype=torch.float64, device="cuda")
        sm.step_adjoint(3, grad, probe=S.Probe(1, nx - 1, tgt))
        out.append((sm.get_adjoint(), grad))
        sm.sync()
        sm.close()
    for a, b in zip(out[0][0], out[1][0]):
        assert torch.equal(a, b)

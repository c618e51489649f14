"""Calls queued one behind the other without a synchronisation, as programs queue them, against the
same calls with the device idle before each: small grids, so that the kernels of several calls are
resident at once (dependent launches).  Everything is deterministic: the results are equal bit by bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

# the FP32 3D march, the FP64 3D pair of kernels, one plane and a batch in either precision
GRIDS = [((64, 16, 8), 3, "f32", {}), ((20, 12, 6), 3, "f32", dict(absorb_cells=2, absorb_sigma=0.3)),
         ((20, 12, 6), 3, "f64", {}), ((128, 48, 1), 2, "f32", {}), ((64, 24, 3), 2, "f32", dict(batched=True)),
         ((48, 40, 1), 2, "f64", {}), ((16, 9, 4), 2, "f64", dict(batched=True))]


def _runs(shape, dims, dtype, kw, body):
    """body(simulation, between) with nothing and with a synchronisation between its calls"""
    from paper_1710_06829_gb300 import inputs
    from paper_1710_06829_gb300 import sim as S
    beta, delta = inputs.isotropic_theta(-0.05, -0.04, 0.02, 0.01)
    f = [torch.from_numpy(a) for a in inputs.random_fields(shape, 31)]
    out = []
    for between in (lambda: None, torch.cuda.synchronize):
        sm = S.Simulation(shape, [1.0, 1.0, 1.0], 0.4, beta, delta, dims=dims, dtype=dtype, **kw)
        sm.set_state(f)
        out.append(body(sm, between))
        sm.sync()
        sm.close()
    return out


@pytest.mark.parametrize("shape,dims,dtype,kw", GRIDS)
def test_plane_waves_of_different_k_and_steps(shape, dims, dtype, kw):
    rng = np.random.default_rng(5)
    calls = [(int(rng.integers(6)), tuple(rng.uniform(-3, 3, 3))) for _ in range(24)]

    def body(sm, between):
        res = torch.zeros((len(calls), 2), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        for n, (comp, k) in enumerate(calls):
            sm.plane_wave(comp, k, out=res[n])
            between()
            if n % 3 == 2:
                sm.step(1)
                between()
        torch.cuda.synchronize()
        return res
    a, b = _runs(shape, dims, dtype, kw, body)
    assert torch.equal(a, b) and bool((a != 0).any())


@pytest.mark.parametrize("shape,dims,dtype,kw", GRIDS)
def test_steps_probes_and_reverse_steps(shape, dims, dtype, kw):
    from paper_1710_06829_gb300 import sim as S
    nx, ny, nz = shape
    tt = torch.float32 if dtype == "f32" else torch.float64
    n = 24
    tgt = torch.from_numpy(np.random.default_rng(6).standard_normal((n + 4, nz, ny))).to(tt).cuda()

    def body(sm, between):
        loss = torch.zeros(1, dtype=torch.float64, device="cuda")
        grad = torch.zeros(12, dtype=torch.float64, device="cuda")
        probe = S.Probe(1, nx - 1, tgt)
        src = None if kw.get("batched") else S.Bunch(1.0, 0.9, 3.0, 2.0, 1.0, 2.0, 2.0)
        sm.set_adjoint()
        torch.cuda.synchronize()
        for _ in range(n // 2):
            sm.step(1, source=src)
            between()
        for _ in range(n // 2):
            sm.step(1, probe=probe, loss=loss)
            between()
        state = sm.get_state()
        sm.step(4, record=True)
        between()
        for _ in range(4):
            sm.step_adjoint(1, grad, probe=probe)
            between()
        return [*state, *sm.get_adjoint(), loss, grad]
    a, b = _runs(shape, dims, dtype, kw, body)
    for x, y in zip(a, b):
        assert torch.equal(x, y)
    assert float(a[12]) > 0 and float(a[13].abs().max()) > 0


def test_norm_call_that_returns_an_error_leaves_no_kernel_behind():
    """A failed allocation of this thread is still recorded when the norm looks at its launches, so the
    call may report it; its kernels have ended all the same when it returns, since its scratch is the
    next call's."""
    from paper_1710_06829_gb300 import _lib as L
    from paper_1710_06829_gb300 import sim as S
    beta, delta = np.zeros((3, 3)), np.zeros(3)
    args = (beta, delta, 0.5, [1.0, 1.0, 1.0], 3, (256, 256, 256))
    st = torch.cuda.Stream()
    ref = S.disp_norm(*args, stream=st)
    with pytest.raises(L.FdtdError) as ei:   # 12 arrays of 8 TB
        S.Simulation((10000, 10000, 10000), [1.0, 1.0, 1.0], 0.4, beta, delta, dtype="f64")
    assert ei.value.status == L.FDTD_ENOMEM
    try:
        S.disp_norm(*args, stream=st)
    except L.FdtdError:
        pass
    assert st.query()
    assert S.disp_norm(*args, stream=st) == ref


def _captured(sm, stream, call):
    """call() captured as the handle's first of its kind; the graph"""
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        call(sm)
    return g


@pytest.mark.parametrize("shape,dims,dtype,kw", GRIDS)
def test_first_probe_step_under_stream_capture(shape, dims, dtype, kw):
    """Two steps with a probe and a plane-wave amplitude, captured as the first calls of a handle and
    replayed twice, against the same calls made directly."""
    from paper_1710_06829_gb300 import inputs
    from paper_1710_06829_gb300 import sim as S
    beta, delta = inputs.isotropic_theta(-0.05, -0.04, 0.02, 0.01)
    nx, ny, nz = shape
    f = [torch.from_numpy(a) for a in inputs.random_fields(shape, 32)]
    tt = torch.float32 if dtype == "f32" else torch.float64
    tgt = torch.from_numpy(np.random.default_rng(7).standard_normal((2, nz, ny))).to(tt).repeat(2, 1, 1).cuda()
    out = []
    for capture in (False, True):
        st = torch.cuda.Stream()
        loss = torch.zeros(1, dtype=torch.float64, device="cuda")
        amp = torch.zeros(2, dtype=torch.float64, device="cuda")
        sm = S.Simulation(shape, [1.0, 1.0, 1.0], 0.4, beta, delta, dims=dims, dtype=dtype, stream=st, **kw)
        sm.set_state(f)

        def call(sm):
            sm.step(2, probe=S.Probe(0, 1, tgt), loss=loss)
            sm.plane_wave(4, (0.3, -0.2, 0.1), out=amp)
        torch.cuda.synchronize()
        if capture:
            g = _captured(sm, st, call)
            with torch.cuda.stream(st):
                g.replay()
                g.replay()
        else:
            call(sm)
            call(sm)
        torch.cuda.synchronize()
        out.append([*sm.get_state(), loss, amp])
        sm.sync()
        sm.close()
    for a, b in zip(*out):
        assert torch.equal(a, b)


def test_first_cycle_of_many_particles_under_stream_capture():
    """As above for two PIC cycles with a particle per cell and more (the mean of B formed per cell).
    The current's additions have no fixed order: about 100 terms of 2e-5 a cell and cycle on fields of
    0.3, each rounded to 2^-24 of the sum: 4 x 100 x 2^-24 = 2.4e-5 of the largest value at the very
    most, 1e-5 taken, the roundings having random signs; positions of up to 32 cells by a few 2^-19."""
    from paper_1710_06829_gb300 import inputs
    from paper_1710_06829_gb300 import sim as S
    shape, n = (32, 20, 16), 1 << 20
    beta, delta = inputs.isotropic_theta(-0.05, -0.04, 0.02, 0.01)
    gen = torch.Generator(device="cuda").manual_seed(3)
    ext = torch.tensor(shape, device="cuda", dtype=torch.float32)[:, None]
    x = torch.rand((3, n), generator=gen, device="cuda") * 0.999 * ext
    u = torch.randn((3, n), generator=gen, device="cuda")
    f = [torch.from_numpy(0.1 * a) for a in inputs.random_fields(shape, 33)]
    out = []
    for capture in (False, True):
        st = torch.cuda.Stream()
        sm = S.Simulation(shape, [1.0, 1.0, 1.0], 0.4, beta, delta, dtype="f32", stream=st)
        sm.set_state(f)
        sp = S.Species(x.clone(), u.clone(), 2e-5, -1.0)

        def call(sm):
            sm.pic_step(2, [sp])
        torch.cuda.synchronize()
        if capture:
            g = _captured(sm, st, call)
            with torch.cuda.stream(st):
                g.replay()
                g.replay()
        else:
            call(sm)
            call(sm)
        torch.cuda.synchronize()
        out.append((sm.get_state(), sp))
        sm.sync()
        sm.close()
    big = max(float(a.abs().max()) for a in out[0][0])
    for a, b in zip(out[0][0], out[1][0]):
        assert float((a - b).abs().max()) <= 1e-5 * big
    d = (out[0][1].x - out[1][1].x).abs()
    assert float(torch.minimum(d, ext - d).max()) <= 1e-4
    assert float((out[0][1].u - out[1][1].u).abs().max()) <= 1e-4


@pytest.mark.parametrize("shape", [(64, 16, 8), (60, 14, 9)])
def test_temporal_blocking_keeps_the_problems_of_a_batch_apart(shape):
    """Pairs of steps on a batch: the bits of single steps, and an infinity in one problem stays there (a
    zero multiplier of a z difference would carry it to the neighbouring ones as NaN)."""
    from paper_1710_06829_gb300 import inputs
    from paper_1710_06829_gb300 import sim as S
    beta, delta = inputs.isotropic_theta(-0.05, -0.04, 0.02, 0.01)
    out = []
    for T, bad in ((1, False), (2, False), (2, True)):
        f = [torch.from_numpy(a) for a in inputs.random_fields(shape, 34)]
        if bad:
            f[0][3, 5, 7] = float("inf")
        sm = S.Simulation(shape, [1.0, 1.0, 1.0], 0.4, beta, delta, dims=2, dtype="f32", batched=True)
        sm.set_temporal_blocking(T, 3)
        sm.set_state(f)
        sm.step(5)
        out.append(sm.get_state())
        sm.close()
    for a, b, c in zip(*out):
        assert torch.equal(a, b)
        c = torch.cat([c[:3], c[4:]])
        assert torch.equal(torch.cat([a[:3], a[4:]]), c)


@pytest.mark.parametrize("shape,slab,sponge", [((60, 12, 20), 4, False), ((132, 15, 33), 5, True),
                                               ((8, 4, 9), 3, False), ((68, 9, 70), 0, False)])
def test_temporal_blocking_on_ragged_grids(shape, slab, sponge):
    """Pairs of steps give the bits of single steps on grids without whole tiles too."""
    from paper_1710_06829_gb300 import inputs
    from paper_1710_06829_gb300 import sim as S
    beta, delta = inputs.isotropic_theta(-0.05, -0.04, 0.02, 0.01)
    f = [torch.from_numpy(a) for a in inputs.random_fields(shape, 35)]
    kw = dict(absorb_cells=2, absorb_sigma=0.2) if sponge else {}
    out = []
    for T in (1, 2):
        sm = S.Simulation(shape, [1.0, 1.0, 1.0], 0.4, beta, delta, dtype="f32", **kw)
        sm.set_temporal_blocking(T, slab)
        sm.set_state(f)
        sm.step(5)
        sm.step(2)
        sm.sync()
        out.append(sm.get_state())
        sm.close()
    for a, b in zip(*out):
        assert torch.equal(a, b)


@pytest.mark.parametrize("name", ["disp_norm", "group_norm"])
def test_norm_call_while_another_thread_captures(name):
    """The call waits for its kernels, returns its value and leaves the capture as it was."""
    import threading

    from paper_1710_06829_gb300 import sim as S
    args = (np.zeros((3, 3)), np.zeros(3), 0.4, [1.0, 1.0, 1.0], 3, (60, 50, 40))
    ref = getattr(S, name)(*args)
    st, side, got = torch.cuda.Stream(), torch.cuda.Stream(), []
    x = torch.zeros(8, device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        x.add_(1)
        t = threading.Thread(target=lambda: got.append(getattr(S, name)(*args, stream=side)))
        t.start()
        t.join()
        x.add_(1)
    g.replay()
    torch.cuda.synchronize()
    assert got == [ref] and bool((x == 2).all())

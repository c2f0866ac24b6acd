"""The persistent FFT passes where their tiling can go wrong: more tiles than
the device holds at once (every CTA takes several, the next one's source
arriving meanwhile) with 16-, 8- and 4-byte staging and a ragged last tile, and
PML slabs whose width is not a multiple of the four cells the x pass moves."""
import numpy as np
import pytest

from paper_1705_04874_gb300 import synth
from conftest import cfl_dt, rel_l2, trace_errors

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def es():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_04874_gb300 import es as _es
    _es._load()
    return _es


# an FP32 derivative rounds its input, ~10 taps and ~4 log2 n butterflies at 1 % weight: a few 1e-7
@pytest.mark.parametrize("shape,axis", [((256, 510, 36), 2), ((510, 256, 34), 1), ((300, 128, 33), 1),
                                        ((128, 301, 35), 2), ((255, 63, 256), 0), ((250, 81, 48), 0)])
@pytest.mark.parametrize("shift", [1, -1])
def test_many_tiles_per_cta(es, orc, shape, axis, shift):
    import torch
    f = np.random.default_rng(sum(shape) + axis).standard_normal(shape).astype(np.float32)
    out = torch.empty(shape, device="cuda")
    es.es_derivative(torch.from_numpy(f).cuda(), axis, 10.0, shift, out)
    ref = orc.deriv(f.astype(np.float64), axis, 10.0, shift)
    assert rel_l2(out.cpu().numpy(), ref) < 5e-7


@pytest.mark.parametrize("nx,pml", [(32, 1), (32, 2), (48, 7), (64, 3), (80, 5)])
def test_slab_widths_that_are_not_whole_quads(es, orc, nx, pml):
    shape = (32, 32, nx)
    rho, cp, cs = synth.two_layer_model(shape=shape, water_cells=8)
    nt, dt = 80, cfl_dt(cp, 10.0)
    w = synth.ricker(nt, dt, 25.0)
    src = [dict(kind="moment", pos=(nx // 2, 15, 17), m=synth.explosive(), w=w)]
    rcv = orc.seabed_receivers(cs, pml, 4, 3)
    with es.Model(rho, cp, cs, dx=10.0, pml=pml) as m:
        m.source_set(src[0]["pos"], src[0]["m"], w)
        gpu = m.run(nt, dt, rcv)
        st = m.state_get()
    ref = orc.simulate(rho, cp, cs, dx=10.0, dt=dt, nt=nt, pml=pml, sources=src, receivers=rcv,
                       state=np.zeros((9,) + shape))
    assert trace_errors(gpu, ref["traces"]).max() < 1e-4
    for f in range(9):
        assert rel_l2(st[f], ref["state"][f]) < 1e-4, f


# every transform length of the convolution passes at both ends of its range (2 n <= length), the
# shortest axis they take and the one below, an axis past what one tile of CTAs holds
@pytest.mark.parametrize("n", [15, 16, 31, 33, 50, 51, 79, 81, 127, 129, 158, 161, 200, 201, 250, 251, 301, 312, 313, 512])
@pytest.mark.parametrize("axis,others", [(0, (7, 9)), (1, (5, 36)), (2, (6, 35))])
def test_convolution_lengths(es, orc, n, axis, others):
    """A derivative rounds its input, its taps and about 4 log2 (padded length)
    butterflies at 2 % weight: a few 1e-7; water-to-rock-like steps in the data."""
    import torch
    shape = {0: (others[0], others[1], n), 1: (others[0], n, others[1]), 2: (n, others[0], others[1])}[axis]
    rng = np.random.default_rng(n + axis)
    f = rng.standard_normal(shape).astype(np.float32)
    f[shape[0] // 2:] *= 50.0
    out = torch.empty(shape, device="cuda")
    for shift in (1, -1):
        es.es_derivative(torch.from_numpy(f).cuda(), axis, 10.0, shift, out)
        ref = orc.deriv(f.astype(np.float64), axis, 10.0, shift)
        assert rel_l2(out.cpu().numpy(), ref) < 5e-7


@pytest.mark.parametrize("shape", [(27, 30, 33), (66, 65, 97), (70, 27, 95)])
def test_run_on_convolution_axes(es, orc, shape):
    """A batch on three axes without a plan (odd nx; convolutions, direct sums and both) and PML, the
    first simulation against the oracle, the second against a run of its own."""
    pml, nt = 4, 100
    rho, cp, cs = synth.two_layer_model(shape=shape, water_cells=6)
    dt = cfl_dt(cp, 10.0)
    w = synth.ricker(nt, dt, 25.0)
    pos = np.array([[16, 15, 14], [14, 13, 15]], np.int32)
    mts = np.stack([synth.explosive(), synth.clvd()])
    rcv = orc.seabed_receivers(cs, pml, 3, 3)
    with es.Model(rho, cp, cs, dx=10.0, pml=pml) as m:
        m.batch_set(pos, mts, np.stack([w, w]))
        got = m.run(nt, dt, rcv)
    ref = orc.simulate(rho, cp, cs, dx=10.0, dt=dt, nt=nt, pml=pml,
                       sources=[dict(kind="moment", pos=tuple(pos[0]), m=mts[0], w=w)], receivers=rcv)["traces"]
    assert trace_errors(got[0], ref).max() < 1e-4
    with es.Model(rho, cp, cs, dx=10.0, pml=pml) as m:
        m.source_set(pos[1], mts[1], w)
        assert np.array_equal(m.run(nt, dt, rcv), got[1])


@pytest.mark.parametrize("shape,pml", [((19, 17, 96), 5), ((17, 19, 128), 3), ((48, 64, 45), 6), ((64, 48, 50), 5)])
def test_ragged_tiles_with_near_parts_in_tensor_memory(es, orc, shape, pml):
    """Lanes of one warp on either side of every branch between two reads of tensor memory: a last x tile of
    three lines, half a tile of columns (nx odd and even) and PML rows that start inside a warp's
    positions, on axes whose near parts wait there."""
    rho, cp, cs = synth.two_layer_model(shape=shape, water_cells=6)
    nt, dt = 60, cfl_dt(cp, 10.0)
    w = synth.ricker(nt, dt, 25.0)
    pos = (shape[2] // 2, shape[1] // 2, max(9, shape[0] // 2))
    rcv = orc.seabed_receivers(cs, pml, 3, 3)
    with es.Model(rho, cp, cs, dx=10.0, pml=pml) as m:
        m.source_set(pos, synth.explosive(), w)
        gpu = m.run(nt, dt, rcv)
        st = m.state_get()
    ref = orc.simulate(rho, cp, cs, dx=10.0, dt=dt, nt=nt, pml=pml, receivers=rcv, state=np.zeros((9,) + shape),
                       sources=[dict(kind="moment", pos=pos, m=synth.explosive(), w=w)])
    assert trace_errors(gpu, ref["traces"]).max() < 1e-4
    for f in range(9):
        assert rel_l2(st[f], ref["state"][f]) < 1e-4, f


ONE_TILE = [(16, 4, 4), (32, 8, 4), (48, 12, 4), (64, 16, 4), (64, 8, 8), (75, 5, 15), (75, 3, 25), (75, 15, 5), (125, 5, 25)]


@pytest.mark.parametrize("n,ra,rb", ONE_TILE)
@pytest.mark.parametrize("nx", [3, 33, 34, 64, 66])  # part of a tile, one or two columns of a second one, whole ones
def test_one_tile_per_cta(es, orc, n, ra, rb, nx):
    """The y and z passes that run one tile per CTA, both directions, stored and accumulated (the Laplacian
    along the other axes adds to what the first one stored).  Bounds as in test_many_tiles_per_cta; the second
    derivative's error is twice a derivative's."""
    import torch
    if nx == 64 and n == 64:
        pytest.skip("persistent")
    default = es.es_fft_plan(1, n)
    es.es_fft_plan_select(1, n, ra, rb)
    try:
        rng = np.random.default_rng(n + nx)
        for axis, shape in ((1, (5, n, nx)), (2, (n, 7, nx))):
            f = rng.standard_normal(shape).astype(np.float32)
            d = torch.from_numpy(f).cuda()
            out = torch.empty(shape, device="cuda")
            for shift in (1, -1):
                es.es_derivative(d, axis, 10.0, shift, out)
                assert rel_l2(out.cpu().numpy(), orc.deriv(f.astype(np.float64), axis, 10.0, shift)) < 5e-7
            es.es_laplacian(d, (10.0, 10.0, 10.0), out)
            want = sum(orc.deriv(orc.deriv(f.astype(np.float64), a, 10.0, -1), a, 10.0, 1) for a in range(3))
            assert rel_l2(out.cpu().numpy(), want) < 1e-6
    finally:
        es.es_fft_plan_select(1, n, *default)


@pytest.mark.parametrize("shape,pml", [((16, 32, 34), 4), ((48, 16, 61), 3), ((125, 75, 20), 5), ((75, 64, 62), 10)])
def test_runs_on_one_tile_passes(es, orc, shape, pml):
    """A batch with PML, sources and receivers in these passes: the first simulation against the oracle, the second
    against a run of its own."""
    nt = 60
    rho, cp, cs = synth.two_layer_model(shape=shape, water_cells=6)
    dt = cfl_dt(cp, 10.0)
    w = synth.ricker(nt, dt, 25.0)
    nz, ny, nx = shape
    pos = np.array([[nx // 2, ny // 2, max(8, nz // 3)], [nx // 2 - 1, ny // 2 - 1, max(9, nz // 3)]], np.int32)
    mts = np.stack([synth.explosive(), synth.clvd()])
    rcv = orc.seabed_receivers(cs, pml, 3, 3)
    with es.Model(rho, cp, cs, dx=10.0, pml=pml) as m:
        m.batch_set(pos, mts, np.stack([w, w]))
        got = m.run(nt, dt, rcv)
    ref = orc.simulate(rho, cp, cs, dx=10.0, dt=dt, nt=nt, pml=pml, receivers=rcv,
                       sources=[dict(kind="moment", pos=tuple(pos[0]), m=mts[0], w=w)])["traces"]
    assert trace_errors(got[0], ref).max() < 1e-4
    with es.Model(rho, cp, cs, dx=10.0, pml=pml) as m:
        m.source_set(pos[1], mts[1], w)
        assert np.array_equal(m.run(nt, dt, rcv), got[1])


# either side of the shortest convolution axes (64 cells, an odd x axis 96) and both ends of every transform's range
@pytest.mark.parametrize("n", [63, 65, 66, 78, 95, 97, 98, 126, 159, 162, 202, 252, 314, 511])
@pytest.mark.parametrize("axis,others", [(0, (7, 9)), (1, (5, 36)), (2, (6, 35))])
def test_quiet_half_beside_a_loud_one(es, orc, n, axis, others):
    """Half of every line is 50 times louder, in space a step along the transformed axis.  The near taps round
    locally; the far part's roundoff, at 2 % of the operator's weight and some 4 log2(1024) = 40 roundings,
    spreads over the line, so the quiet half sees 50 x 0.02 x 40 x 2^-24 = 2.4e-6 of its own derivative, and the
    few 1e-7 of its own rounding."""
    import torch
    shape = {0: (others[0], others[1], n), 1: (others[0], n, others[1]), 2: (n, others[0], others[1])}[axis]
    f = np.random.default_rng(3 * n + axis).standard_normal(shape).astype(np.float32)
    quiet, loud = [slice(None)] * 3, [slice(None)] * 3
    quiet[2 - axis], loud[2 - axis] = slice(8, n // 2 - 8), slice(n // 2, n)
    f[tuple(loud)] *= 50.0
    out = torch.empty(shape, device="cuda")
    for shift in (1, -1):
        es.es_derivative(torch.from_numpy(f).cuda(), axis, 10.0, shift, out)
        ref = orc.deriv(f.astype(np.float64), axis, 10.0, shift)
        got = out.cpu().numpy()
        assert rel_l2(got, ref) < 5e-7
        assert rel_l2(got[tuple(quiet)], ref[tuple(quiet)]) < 3e-6


@pytest.mark.parametrize("shape", [(13, 11, 75), (13, 11, 125), (13, 15, 66), (11, 13, 97), (13, 11, 127)])
def test_x_tiles_off_every_boundary(es, orc, shape):
    """Four simulations of an odd cell count (of 66 x 195 cells two of four) start 0, 4, 8 and 12 bytes past a
    16-byte boundary: each equals the single run, bit for bit, PML included."""
    pml, nt = 3, 40
    rho, cp, cs = synth.two_layer_model(shape=shape, water_cells=4)
    dt = cfl_dt(cp, 10.0)
    w = synth.ricker(nt, dt, 25.0)
    pos = (shape[2] // 2, shape[1] // 2, 6)
    rcv = orc.seabed_receivers(cs, pml, 3, 3)
    with es.Model(rho, cp, cs, dx=10.0, pml=pml) as m:
        m.source_set(pos, synth.explosive(), w)
        one, st = m.run(nt, dt, rcv), m.state_get()
    with es.Model(rho, cp, cs, dx=10.0, pml=pml) as m:
        m.batch_set(np.array([pos] * 4, np.int32), np.stack([synth.explosive()] * 4), np.stack([w] * 4))
        four, states = m.run(nt, dt, rcv), m.state_get()
    for k in range(4):
        assert np.array_equal(four[k], one) and np.array_equal(states[k], st), k
    ref = orc.simulate(rho, cp, cs, dx=10.0, dt=dt, nt=nt, pml=pml, receivers=rcv,
                       sources=[dict(kind="moment", pos=pos, m=synth.explosive(), w=w)])["traces"]
    assert trace_errors(one, ref).max() < 1e-4


# both ends of every transform of the convolution passes
@pytest.mark.parametrize("n,m", [(66, 160), (78, 160), (98, 256), (103, 256), (126, 256), (151, 320), (199, 400),
                                 (202, 500), (252, 625), (314, 1024), (511, 1024)])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_silence_far_from_a_pulse(es, orc, n, m, axis):
    """What a pulse leaves where its derivative is as good as zero, past the near taps (24).  An FFT of m points
    leaves a few 2^-24 of the pulse's norm over sqrt(m), times the norm of the kernel's far part, in every row:
    1.5 to 2.4 of them with this pulse, transforms and tables in 32 bits and a radix-free FFT on the host, so at
    most 4.  (A near part of 10 taps leaves 3 to 4 times as much, 5 at the least.)"""
    import torch
    rng = np.random.default_rng(7 * n + axis)
    x = np.arange(n)[:, None]
    f = np.exp(-((x - n // 2 - rng.uniform(-1, 1, 320)) / rng.uniform(2, 4, 320)) ** 2) * rng.uniform(0.5, 2, 320)
    f = np.where(abs(x - n // 2) <= 12, f, 0).astype(np.float32)
    a = np.moveaxis(f.reshape(n, 10, 32), 0, 2 - axis).copy()
    out = torch.empty(a.shape, device="cuda")
    quiet = abs(x[:, 0] - n // 2) > 26
    delta = np.moveaxis(np.eye(1, n)[0].reshape(n, 1, 1), 0, 2 - axis)
    for shift in (1, -1):
        c = np.moveaxis(orc.deriv(delta, axis, 10.0, shift), 2 - axis, 0).ravel()  # the circulant kernel
        far = np.sort(abs(c))[:-24]
        es.es_derivative(torch.from_numpy(a).cuda(), axis, 10.0, shift, out)
        err = out.cpu().numpy() - orc.deriv(a.astype(np.float64), axis, 10.0, shift)
        err = np.moveaxis(err, 2 - axis, 0)[quiet]
        rms = np.sqrt((f.astype(np.float64) ** 2).sum(0).mean())
        assert np.sqrt((err ** 2).mean()) < 4 * 2.0 ** -24 * rms * np.linalg.norm(far) / np.sqrt(m)

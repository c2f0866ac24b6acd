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

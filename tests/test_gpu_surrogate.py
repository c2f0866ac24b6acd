"""The learned surrogate on the GPU: its BF16/FP32 GEMM in every storage
order, its loss and gradients against the FP64 oracle (oracle/surrogate.py),
and the whole workflow on a small model -- solver catalog, training on the
GPU, error gate, serving with the solver as fallback -- where every served
seismogram is checked against the exact solver reference."""
import numpy as np
import pytest

from paper_1705_04874_gb300 import synth
from conftest import cfl_dt

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_04874_gb300 import es, surrogate
    es._load()
    return es, surrogate, torch


def _bf(torch, a):
    return torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda().to(torch.bfloat16)


@pytest.mark.parametrize("a_t", [False, True])
@pytest.mark.parametrize("b_nk", [False, True])
@pytest.mark.parametrize("split", [1, 3])
def test_gemm_all_layouts(env, a_t, b_nk, split):
    es, sur, torch = env
    rng = np.random.default_rng(int(a_t) * 4 + int(b_nk) * 2 + split)
    M, N, K = 200, 136, 328  # ragged against the 128 x 128 x 32 tiles
    A = rng.standard_normal((K, M) if a_t else (M, K)).astype(np.float32)
    B = rng.standard_normal((N, K) if b_nk else (K, N)).astype(np.float32)
    Ab, Bb = _bf(torch, A), _bf(torch, B)
    A64 = Ab.float().cpu().numpy().astype(np.float64)  # the BF16-rounded operands
    B64 = Bb.float().cpu().numpy().astype(np.float64)
    opA = A64.T if a_t else A64
    opB = B64.T if b_nk else B64
    C0 = rng.standard_normal((M, N)).astype(np.float32)
    C = torch.from_numpy(C0.copy()).cuda()
    sur.es_gemm_bf16(Ab, Bb, C, a_t=a_t, b_nk=b_nk, alpha=0.5, beta=-2.0, split_k=split)
    ref = 0.5 * opA @ opB - 2.0 * C0
    got = C.cpu().numpy()
    assert np.abs(got - ref).max() <= 2e-5 * np.abs(ref).max()


@pytest.mark.parametrize("M,N,K,split,beta", [(8, 8, 8, 1, 0.0), (128, 256, 64, 1, 0.0), (300, 520, 1000, 1, 1.5),
                                               (256, 1000, 4608, 6, -0.5), (130, 260, 136, 1, 0.0),
                                               (64, 4608, 8192, 16, 0.0), (2000, 4000, 200, 1, 0.5),
                                               (4096, 8192, 64, 1, 0.0)])
def test_tcgen05_gemm_k_major(env, M, N, K, split, beta):
    """Both operands K-major: the persistent tcgen05 kernel (TMA ring, two
    tensor-memory accumulators), single tiles, ragged edges in M, N and K,
    split-K, and grids of 256 and 1024 tiles (several per CTA)."""
    import ctypes
    es, sur, torch = env
    rng = np.random.default_rng(M + N + K + split)
    lda, ldb, ldc = K + 8, K + 16, N + 4  # leading dimensions past the matrix edge
    A = rng.standard_normal((M, lda)).astype(np.float32)
    B = rng.standard_normal((N, ldb)).astype(np.float32)
    Ab, Bb = _bf(torch, A), _bf(torch, B)
    A64 = Ab.float().cpu().numpy().astype(np.float64)[:, :K]
    B64 = Bb.float().cpu().numpy().astype(np.float64)[:, :K]
    C0 = rng.standard_normal((M, ldc)).astype(np.float32)
    C = torch.from_numpy(C0.copy()).cuda()
    vp = lambda t: ctypes.c_void_p(t.data_ptr())
    rc = sur._lib().es_gemm_bf16(M, N, K, vp(Ab), lda, 0, vp(Bb), ldb, 1, vp(C), ldc, ctypes.c_float(0.75),
                                 ctypes.c_float(beta), split, None)
    assert rc == 0
    sur.es_gemm_status()
    ref = 0.75 * A64 @ B64.T + beta * C0[:, :N]
    got = C.cpu().numpy()
    assert np.abs(got[:, :N] - ref).max() <= 2e-5 * np.abs(ref).max()
    assert np.array_equal(got[:, N:], C0[:, N:])  # columns past N untouched


def test_bounded_wait_times_out_and_the_context_survives(env):
    """The failure path of the tcgen05 GEMM's bounded waits, without a fault
    or a hang: a wait on a barrier phase that nothing completes gives up after
    50 ms, the status word reports ES_ERR_TIMEOUT once and is cleared, and the
    same context then runs a tcgen05 GEMM correctly."""
    import time
    es, sur, torch = env
    sur.es_gemm_status()  # starts clear
    t0 = time.perf_counter()
    sur.es_gemm_wait_probe(0.05)
    with pytest.raises(es.EsError) as err:
        sur.es_gemm_status()
    assert err.value.status == es.ES_ERR_TIMEOUT
    assert time.perf_counter() - t0 >= 0.05
    sur.es_gemm_status()  # read once, then clear
    rng = np.random.default_rng(1)
    A, B = _bf(torch, rng.standard_normal((136, 200))), _bf(torch, rng.standard_normal((264, 200)))
    C = torch.zeros((136, 264), device="cuda")
    sur.es_gemm_bf16(A, B, C, b_nk=True)
    sur.es_gemm_status()
    ref = A.float().cpu().numpy().astype(np.float64) @ B.float().cpu().numpy().astype(np.float64).T
    assert np.abs(C.cpu().numpy() - ref).max() <= 2e-5 * np.abs(ref).max()


def test_loss_and_gradients_match_oracle(env):
    es, sur, torch = env
    from oracle import surrogate as osur
    cfg = dict(nfreq=2, hidden=64, latent=16, n_rcv=4, nt=16)
    s = sur.Surrogate(cfg["n_rcv"], cfg["nt"], nfreq=2, hidden=64, latent=16, max_batch=16, seed=3)
    try:
        rng = np.random.default_rng(5)
        lay, P, F, D = osur.layout(**cfg)
        assert s.num_params() == P
        params = (rng.standard_normal(P) * 0.2).astype(np.float32)
        s.set_params(params)
        scale = [1.5, 0.7, 0.9, 1.1]
        s.set_output_scale(scale)
        B = 16
        pos = rng.uniform(-1, 1, (B, 3)).astype(np.float32)
        mt = rng.standard_normal((B, 6)).astype(np.float32)
        tgt = rng.standard_normal((B, D)).astype(np.float32)
        cu = lambda a: torch.from_numpy(a).cuda()
        loss, per, g = s.loss_grad(cu(pos), cu(mt), cu(tgt))
        # the oracle sees the parameters the GPU multiplies with (BF16-rounded weights)
        pb = torch.from_numpy(params).to(torch.bfloat16).float().numpy().astype(np.float64)
        pr = params.astype(np.float64).copy()
        for name in ("W1", "W2", "W3", "Wd"):
            o, shp = lay[name]
            pr[o:o + int(np.prod(shp))] = pb[o:o + int(np.prod(shp))]
        oloss, oper, og = osur.loss_and_grads(pr, cfg, pos, mt, tgt, scale)
        assert abs(loss - oloss) <= 2e-2 * oloss
        assert np.allclose(per.cpu().numpy(), oper, rtol=3e-2)
        g = g.cpu().numpy().astype(np.float64)
        # BF16 operands round to 2^-9 relative; the gradient of the first layer
        # sits behind five such roundings (dU, dA, dH2, dH1, x), the others behind fewer
        tol = {"W1": 6e-2, "b1": 6e-2}
        for name, (o, shp) in lay.items():
            n = int(np.prod(shp))
            a, b = g[o:o + n], og[o:o + n]
            assert np.linalg.norm(a - b) <= tol.get(name, 3e-2) * np.linalg.norm(b), name
        y = s.predict(cu(pos), cu(mt)).cpu().numpy()
        assert np.linalg.norm(y - osur.forward(pr, cfg, pos, mt, scale)["Y"]) <= 1e-2 * np.linalg.norm(y)
    finally:
        s.close()


def test_train_step_matches_oracle_adam(env):
    """One train step against the oracle's Adam step taken from its own FP64
    gradient (BF16-rounded weights).  The first Adam step moves a parameter by
    lr g / (|g| + eps), so wherever the gradient's sign is certain the GPU's
    update must equal the oracle's to FP32 rounding, and no parameter may move
    by more than lr.  The decoder has 96 rows (ragged 64-row tiles of the
    fused step).  Then predict() must run on the updated decoder: its K-major
    copy is refreshed by the step itself."""
    es, sur, torch = env
    from oracle import surrogate as osur
    cfg = dict(nfreq=2, hidden=64, latent=16, n_rcv=4, nt=16)
    s = sur.Surrogate(cfg["n_rcv"], cfg["nt"], nfreq=2, hidden=64, latent=16, max_batch=16, seed=3)
    try:
        rng = np.random.default_rng(11)
        lay, P, F, D = osur.layout(**cfg)
        params = (rng.standard_normal(P) * 0.2).astype(np.float32)
        s.set_params(params)
        scale = [1.5, 0.7, 0.9, 1.1]
        s.set_output_scale(scale)
        B, lr = 16, 2e-2
        pos = rng.uniform(-1, 1, (B, 3)).astype(np.float32)
        mt = rng.standard_normal((B, 6)).astype(np.float32)
        tgt = rng.standard_normal((B, D)).astype(np.float32)
        cu = lambda a: torch.from_numpy(a).cuda()
        s.predict(cu(pos), cu(mt))  # the K-major copy of the initial decoder exists before the step
        s.train_step(cu(pos), cu(mt), cu(tgt), lr)
        after = s.get_params().astype(np.float64)

        def bf16(x):
            out = np.asarray(x, np.float64).copy()
            r = torch.from_numpy(np.asarray(x, np.float32)).to(torch.bfloat16).float().numpy()
            for name in ("W1", "W2", "W3", "Wd"):
                o, shp = lay[name]
                out[o:o + int(np.prod(shp))] = r[o:o + int(np.prod(shp))]
            return out

        _, _, og = osur.loss_and_grads(bf16(params), cfg, pos, mt, tgt, scale)
        exp, _, _ = osur.adam_step(params.astype(np.float64), og, 0.0, 0.0, 1, lr)
        moved = after - params.astype(np.float64)
        assert np.abs(moved).max() <= lr * (1 + 1e-3)
        # The GPU's gradient is within tol * |g| of the oracle's (the bound of the gradient test), so
        # an element larger than that keeps its sign and must take the oracle's step exactly; below
        # it BF16 rounding may flip a sign, which at most 5 % of the elements may show.
        tol = {"W1": 6e-2, "b1": 6e-2}
        for name, (o, shp) in lay.items():
            n = int(np.prod(shp))
            g = og[o:o + n]
            dev = np.abs(after[o:o + n] - exp[o:o + n])
            sure = np.abs(g) > tol.get(name, 3e-2) * np.linalg.norm(g)
            assert not sure.any() or dev[sure].max() <= 1e-3 * lr, name
            nz = g != 0
            assert np.mean(dev[nz] <= 1e-3 * lr) >= 0.95, (name, np.mean(dev[nz] <= 1e-3 * lr))
        y = s.predict(cu(pos), cu(mt)).cpu().numpy()
        ref = osur.forward(bf16(after.astype(np.float32)), cfg, pos, mt, scale)["Y"]
        stale = osur.forward(bf16(np.concatenate([after[:lay["Wd"][0]], params[lay["Wd"][0]:]]).astype(np.float32)),
                             cfg, pos, mt, scale)["Y"]
        assert np.linalg.norm(ref - stale) > 5e-2 * np.linalg.norm(ref)  # the step moved the decoder visibly
        assert np.linalg.norm(y - ref) <= 1e-2 * np.linalg.norm(ref)
    finally:
        s.close()


@pytest.mark.parametrize("n_src", [40, 37])
def test_serve_trusted_sources(env, n_src):
    """Every location trusted: serve() predicts runs of consecutive sources
    straight into the caller's buffer (a ragged tail through a padded batch);
    the result equals predict() on the same inputs, bit for bit."""
    es, sur, torch = env
    s = sur.Surrogate(2, 16, nfreq=2, hidden=32, latent=8, max_batch=16, seed=2)
    try:
        rng = np.random.default_rng(n_src)
        pos_n = rng.uniform(-1, 1, (5, 3)).astype(np.float32)
        loc = rng.integers(0, 5, n_src)
        mts = rng.standard_normal((n_src, 6))
        buf = torch.full((n_src, 4, 2, 16), float("nan"), device="cuda")
        out, used = sur.serve(s, pos_n, np.ones(5, bool), loc, mts, None, None, 16, 0.0, np.zeros((2, 3), np.int32),
                              None, out=buf)
        assert out.data_ptr() == buf.data_ptr() and not used.any()
        for b in range(0, n_src, 16):
            n = min(16, n_src - b)
            k = (n + 7) // 8 * 8
            idx = np.concatenate([np.arange(b, b + n), np.full(k - n, b)])
            ref = s.predict(torch.from_numpy(pos_n[loc[idx]]).cuda(),
                            torch.from_numpy(mts[idx].astype(np.float32)).cuda())[:n]
            assert torch.equal(out[b:b + n].reshape(n, -1), ref), b
    finally:
        s.close()


def test_catalog_train_gate_serve(env):
    """Small marine model, 24 catalog locations: the surrogate learns their
    Green's functions from 144 solver runs (unit moment tensors), is trained
    on fresh random moment tensors every epoch, the gate keeps the locations it
    reproduces within 5 %, and every served seismogram (surrogate or solver)
    is within 5 % of the exact reference."""
    es, sur, torch = env
    shape = (48, 32, 32)
    rho, cp, cs = synth.marine_model(shape=shape, seed=4)
    pml, nt = 4, 256  # long enough for the full arrivals at every receiver
    dt = cfl_dt(cp, 10.0)
    wav = synth.ricker(nt, dt, 30.0)
    box = synth.reservoir_box(shape, pml)
    rng = synth.SplitMix64(6)
    locations = synth.latin_hypercube_positions(rng, box, 24)
    with es.Model(rho, cp, cs, dx=10.0, pml=pml) as m:
        rcv = m.seabed_receivers(2, 2)
        G = sur.green_catalog(m, locations, nt, dt, rcv, wav, per_batch=8)
        pos_n = sur.normalize_positions(locations, box)
        s = sur.Surrogate(len(rcv), nt, nfreq=3, hidden=128, latent=64, max_batch=48, seed=1)
        try:
            hist = sur.train(s, pos_n, G, epochs=200, lr=3e-3)
            assert hist[-1] < 1e-4 * hist[0]
            trusted, errs = sur.calibrate_gate(s, pos_n, G, n_val=3)
            assert trusted.mean() >= 0.75, errs.max(axis=1)
            # serve random sources at catalog locations
            loc = np.floor(synth.SplitMix64(9).uniform(40) * len(locations)).astype(int)
            mts = np.array([synth.random_dc(rng) for _ in loc])
            out, used_solver = sur.serve(s, pos_n, trusted, loc, mts, m, locations, nt, dt, rcv, wav)
            ref = sur.combine(G, loc, mts)
            # whole-seismogram relative L2 with each component divided by its RMS over the catalog
            sc = G.permute(2, 0, 1, 3, 4).reshape(4, -1).pow(2).mean(dim=1).sqrt().view(1, 4, 1, 1)
            d = ((out - ref) / sc).reshape(len(loc), -1).norm(dim=1) / (ref / sc).reshape(len(loc), -1).norm(dim=1)
            assert float(d.max()) < 0.05, float(d.max())
            assert used_solver.sum() == (~trusted[loc]).sum()
        finally:
            s.close()


def test_sources_away_from_the_catalog(env):
    """Sources at cells that are not catalog locations: their exact references
    come from fresh solver runs; the network is compared with the two baselines
    without one (the nearest catalog location, inverse-distance interpolation
    of the catalog); the position gate, calibrated on held-out cells, decides
    which of them the network may serve.  Every served seismogram -- network
    or solver fallback -- is within 5 % of its exact reference, and the
    fallback runs for the off-catalog sources the gate refuses."""
    es, sur, torch = env
    shape = (48, 32, 32)
    rho, cp, cs = synth.marine_model(shape=shape, seed=4)
    pml, nt = 4, 256
    dt = cfl_dt(cp, 10.0)
    wav = synth.ricker(nt, dt, 30.0)
    box = synth.reservoir_box(shape, pml)
    rng = synth.SplitMix64(6)
    locations = synth.latin_hypercube_positions(rng, box, 24)
    with es.Model(rho, cp, cs, dx=10.0, pml=pml) as m:
        rcv = m.seabed_receivers(2, 2)
        G = sur.green_catalog(m, locations, nt, dt, rcv, wav, per_batch=8)
        sc = sur.component_scale(G)
        s = sur.Surrogate(len(rcv), nt, nfreq=3, hidden=128, latent=64, max_batch=48, seed=1)
        try:
            sur.train(s, sur.normalize_positions(locations, box), G, epochs=200, lr=3e-3)
            trusted, _ = sur.calibrate_gate(s, sur.normalize_positions(locations, box), G, n_val=3)
            # held-out cells off the catalog
            cand = synth.random_positions(synth.SplitMix64(12), box, 64)
            _, dc = sur.nearest_locations(locations, cand)
            held = cand[dc[:, 0] > 0][:16]
            hmt = np.array([synth.random_dc(rng) for _ in held])
            truth = sur.solver_references(m, held, hmt, nt, dt, rcv, wav)
            _, hd = sur.nearest_locations(locations, held)
            e_net = sur.scaled_rel_l2(sur.predict_at(s, box, held, hmt), truth, sc)
            e_near = sur.scaled_rel_l2(sur.baseline_nearest(G, locations, held, hmt), truth, sc)
            e_idw = sur.scaled_rel_l2(sur.baseline_idw(G, locations, held, hmt), truth, sc)
            assert np.isfinite(e_net).all() and np.isfinite(e_near).all() and np.isfinite(e_idw).all()
            print(f"off-catalog: within 5 % {np.mean(e_net < 0.05):.3f}; median error network {np.median(e_net):.3f}, "
                  f"nearest location {np.median(e_near):.3f}, inverse-distance {np.median(e_idw):.3f}")
            d_star = sur.calibrate_position_gate(hd[:, 0], e_net)
            # a mix of catalog and off-catalog sources, not the held-out ones
            pos = np.concatenate([locations[:8], cand[dc[:, 0] > 0][16:24]])
            mts = np.array([synth.random_dc(rng) for _ in pos])
            out, used = sur.serve_positions(s, box, trusted, d_star, locations, pos, mts, m, nt, dt, rcv, wav)
            ref = sur.solver_references(m, pos, mts, nt, dt, rcv, wav)
            err = sur.scaled_rel_l2(out, ref, sc)
            assert err.max() < 0.05, err
            _, pd = sur.nearest_locations(locations, pos)
            assert used[pd[:, 0] > max(d_star, 0)].all()  # beyond the gate's distance: the solver
            assert used.any() and (~used[:8]).sum() == trusted[:8].sum()
        finally:
            s.close()


def test_decoder_step_inside_its_gradient_gemm(env):
    """The decoder takes its Adam step in the GEMM that forms the gradient, here with more 128 x 128
    tiles than SMs: 144 x 9824 (ragged row and column tiles, a 16-row remainder of a 32-row block), a batch
    of 24 (a part of a K slab).  Two steps against Adam in FP64 on the gradients that loss_grad
    returns.  The two FP32 accumulations of at most 24 products differ by about 1e-6 of their size,
    so where |g| > 0.1 rms in both steps a step m / sqrt(v) agrees to 1e-3.  Then both BF16 copies
    of the decoder equal those of a network that is given the parameters."""
    es, sur, torch = env
    args = dict(nfreq=2, hidden=64, latent=24, max_batch=24)
    n_rcv, nt, B, lr = 307, 8, 24, 1e-2
    D, K6 = 4 * n_rcv * nt, 6 * 24
    s, f = sur.Surrogate(n_rcv, nt, seed=3, **args), sur.Surrogate(n_rcv, nt, seed=4, **args)
    try:
        rng = np.random.default_rng(17)
        cu = lambda a: torch.from_numpy(a.astype(np.float32)).cuda()
        pos, mt = cu(rng.uniform(-1, 1, (B, 3))), cu(rng.standard_normal((B, 6)))
        tgt = cu(rng.standard_normal((B, D)))
        p = (rng.standard_normal(s.num_params()) * 0.2).astype(np.float32)
        s.set_params(p)
        wd = slice(len(p) - K6 * D, len(p))
        m = v = 0.0
        sure = True
        for t in (1, 2):
            before = s.get_params()[wd].astype(np.float64)
            g = s.loss_grad(pos, mt, tgt)[2].cpu().numpy()[wd].astype(np.float64)
            s.train_step(pos, mt, tgt, lr)
            after = s.get_params()[wd].astype(np.float64)
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            want = -lr * (m / (1 - 0.9 ** t)) / (np.sqrt(v / (1 - 0.999 ** t)) + 1e-8)
            sure = sure & (np.abs(g) > 0.1 * np.sqrt(np.mean(g * g)))
            assert sure.mean() > 0.5
            assert np.abs(after - before - want)[sure].max() <= 1e-3 * lr
        f.set_params(s.get_params())
        assert torch.equal(s.predict(pos, mt), f.predict(pos, mt))
        a, b = (x.loss_grad(pos, mt, tgt)[2][:wd.start] for x in (s, f))  # through the row-major copy
        assert float((a - b).norm()) <= 1e-5 * float(b.norm())
    finally:
        s.close()
        f.close()


@pytest.mark.parametrize("hidden, latent, B, nfreq", [(8, 8, 8, 0), (64, 64, 32, 9), (328, 40, 40, 3), (392, 136, 72, 16)])
def test_encoder_layers_at_ragged_sizes(env, hidden, latent, B, nfreq):
    """The 32 x 64 x 64 tiles of the layer kernel: less than one of each, exact ones, remainders of 8
    in every direction and more k-slabs than the ring holds, against the oracle's formulas in FP64
    with every operand rounded to BF16 where the GPU rounds it.  What is left are FP32 sums, about
    1e-6 off, and the BF16 roundings they flip: one in some 2^8 1e-5 of the values by 2^-8, 2e-4 of
    a norm per rounding, five of them on the way to the first layer, doubled."""
    es, sur, torch = env
    from oracle import surrogate as osur
    cfg = dict(nfreq=nfreq, hidden=hidden, latent=latent, n_rcv=4, nt=16)
    s = sur.Surrogate(4, 16, nfreq=nfreq, hidden=hidden, latent=latent, max_batch=B, seed=3)
    try:
        rng = np.random.default_rng(hidden)
        lay, P, F, D = osur.layout(**cfg)
        params = (rng.standard_normal(P) / np.sqrt(hidden)).astype(np.float32)
        s.set_params(params)
        scale = [1.5, 0.7, 0.9, 1.1]
        s.set_output_scale(scale)
        pos = rng.uniform(-1, 1, (B, 3)).astype(np.float32)
        mt = rng.standard_normal((B, 6)).astype(np.float32)
        tgt = rng.standard_normal((B, D)).astype(np.float32)
        cu = lambda a: torch.from_numpy(a).cuda()
        got = s.loss_grad(cu(pos), cu(mt), cu(tgt))[2].cpu().numpy().astype(np.float64)
        bf = lambda a: torch.from_numpy(np.asarray(a, np.float64)).float().to(torch.bfloat16).double().numpy()
        w = osur.unpack(params, lay)
        W1, W2, W3, Wd = (bf(w[k]) for k in ("W1", "W2", "W3", "Wd"))
        X = bf(osur.features(pos, nfreq, F))
        H1 = np.maximum(X @ W1 + w["b1"], 0)
        H2 = np.maximum(bf(H1) @ W2 + w["b2"], 0)
        A = bf(H2) @ W3 + w["b3"]
        m6 = mt.astype(np.float64)
        Z = bf((m6[:, :, None] * A[:, None, :]).reshape(B, -1))
        sc = np.repeat(scale, D // 4)
        den = np.sum((tgt / sc) ** 2, axis=1, keepdims=True)
        dU = bf(2 * (Z @ Wd - tgt / sc) / (B * den))
        dA = np.einsum("bc,bck->bk", m6, (dU @ Wd.T).reshape(B, 6, latent))
        dH2 = (bf(dA) @ W3.T) * (H2 > 0)
        dH1 = (bf(dH2) @ W2.T) * (H1 > 0)
        want = dict(Wd=Z.T @ dU, b3=dA.sum(0), W3=bf(H2).T @ bf(dA), b2=dH2.sum(0), W2=bf(H1).T @ bf(dH2),
                    b1=dH1.sum(0), W1=X.T @ bf(dH1))
        for name, (o, shp) in lay.items():
            a, b = got[o:o + int(np.prod(shp))], want[name].ravel()
            assert np.linalg.norm(a - b) <= 2e-3 * np.linalg.norm(b), name
    finally:
        s.close()


@pytest.mark.parametrize("B", [8, 64, 72])
def test_target_on_any_word_boundary(env, B):
    """A target off the 16-byte boundary gives the same loss and gradients to the last bit (D = 288 is
    a multiple of neither tile side; one split, so every sum has a fixed order)."""
    es, sur, torch = env
    s = sur.Surrogate(3, 24, nfreq=1, hidden=16, latent=8, max_batch=B, seed=3)
    try:
        g = torch.Generator().manual_seed(B)
        r = lambda *n: torch.randn(*n, generator=g).cuda()
        pos, mt, tgt = r(B, 3).clamp(-1, 1), r(B, 6), r(B, 4 * 3 * 24)
        shifted = torch.empty(tgt.numel() + 1, device="cuda")[1:].view_as(tgt).copy_(tgt)
        a, b = s.loss_grad(pos, mt, tgt), s.loss_grad(pos, mt, shifted)
        assert abs(a[0] - b[0]) <= 1e-6 * abs(a[0])  # the mean over samples is added in any order
        assert torch.equal(a[1], b[1]) and torch.equal(a[2], b[2])
    finally:
        s.close()


@pytest.mark.parametrize("rank, stage", [(0, 0), (1, 0), (0, 3), (1, 3), (0, 6), (1, 13), (0, 19), (1, 19)])
def test_a_pair_that_gives_up_awaits_its_copies(env, rank, stage):
    """The failure path of a CTA pair, without a fault or a hang: one CTA's producer stops (at the first
    k-block, within the ring of six, a turn later, at the last), every wait runs out within its bound,
    and the copies that only the other CTA had started are awaited too.  The status word reports it once,
    and the next product is right."""
    es, sur, torch = env
    sur.es_gemm_status()
    sur.es_gemm_pair_probe(rank, stage)
    with pytest.raises(es.EsError) as err:
        sur.es_gemm_status()
    assert err.value.status == es.ES_ERR_TIMEOUT
    rng = np.random.default_rng(stage)
    A, B = _bf(torch, rng.standard_normal((256, 1280))), _bf(torch, rng.standard_normal((512, 1280)))
    C = torch.zeros((256, 512), device="cuda")
    sur.es_gemm_bf16(A, B, C, b_nk=True)
    sur.es_gemm_status()
    ref = A.float().cpu().numpy().astype(np.float64) @ B.float().cpu().numpy().astype(np.float64).T
    assert np.abs(C.cpu().numpy() - ref).max() <= 2e-5 * np.abs(ref).max()


@pytest.mark.parametrize("M, N, K, split, beta", [
    (256, 77824, 1024, 1, 0.0),   # 608 tiles of 16 k-blocks: 64 for each of 152 SMs, the fewest that run on pairs
    (256, 77824, 960, 1, 0.0),    # 15 k-blocks: single CTAs
    (200, 77800, 1000, 1, 0.5),   # ragged rows, columns and K on pairs
    (1024, 20000, 1096, 1, 0.0),  # eight row tiles, several tiles per pair
    (250, 4600, 100000, 32, 1.0), # slices of K added by atomics
])
def test_products_large_enough_for_pairs(env, M, N, K, split, beta):
    """Products on either side of the rule that puts them on pairs of CTAs, against FP64.  K products of
    N(0, 1) operands summed in FP32 are within 2e-5 of the largest sum (about 6 sqrt(K))."""
    es, sur, torch = env
    g = torch.Generator(device="cuda").manual_seed(M + N)
    A = torch.randn((M, K), device="cuda", generator=g).bfloat16()
    B = torch.randn((N, K), device="cuda", generator=g).bfloat16()
    C = torch.randn((M, N), device="cuda", generator=g)
    want = beta * C.double()
    for n in range(0, N, 8192):
        want[:, n:n + 8192] += A.double() @ B[n:n + 8192].double().T
    sur.es_gemm_bf16(A, B, C, b_nk=True, beta=beta, split_k=split)
    sur.es_gemm_status()
    assert float((C - want).abs().max()) <= 2e-5 * float(want.abs().max())


@pytest.mark.parametrize("latent, n_rcv, nt, B", [
    (8, 3, 24, 768),      # the largest batch whose step stays in the gradient GEMM while the weights fit in L2
    (8, 3, 24, 776),      # the smallest past it: gradient and step apart
    (48, 37, 208, 440),   # 8.9 M weights: in the GEMM below 448
    (48, 37, 208, 448),   # and apart from there on; 288 rows and 30784 columns, ragged tiles of 64
])
def test_decoder_step_on_both_sides_of_its_rule(env, latent, n_rcv, nt, B):
    """One training step against Adam in FP64 on the gradient that loss_grad returns, where that is not tiny
    (|g| > 0.1 rms): the two FP32 sums of at most 776 products differ by about 1e-6 of their size, so the first
    step, lr g / |g|, agrees to 1e-3.  Then both BF16 copies equal those of a network given the parameters."""
    es, sur, torch = env
    args = dict(nfreq=1, hidden=16, latent=latent, max_batch=B)
    s, f = sur.Surrogate(n_rcv, nt, seed=3, **args), sur.Surrogate(n_rcv, nt, seed=4, **args)
    D, lr = 4 * n_rcv * nt, 1e-2
    try:
        g = torch.Generator().manual_seed(B)
        r = lambda *n: torch.randn(*n, generator=g).cuda()
        pos, mt, tgt = r(B, 3).clamp(-1, 1), r(B, 6), r(B, D)
        s.set_params((np.random.default_rng(B).standard_normal(s.num_params()) * 0.2).astype(np.float32))
        wd = slice(s.num_params() - 6 * latent * D, s.num_params())
        before = s.get_params()[wd].astype(np.float64)
        grad = s.loss_grad(pos, mt, tgt)[2].cpu().numpy()[wd].astype(np.float64)
        s.train_step(pos, mt, tgt, lr)
        after = s.get_params()[wd].astype(np.float64)
        m, v = 0.1 * grad, 0.001 * grad * grad
        want = -lr * (m / (1 - 0.9)) / (np.sqrt(v / (1 - 0.999)) + 1e-8)
        sure = np.abs(grad) > 0.1 * np.sqrt(np.mean(grad * grad))
        assert sure.mean() > 0.5
        assert np.abs(after - before - want)[sure].max() <= 1e-3 * lr
        f.set_params(s.get_params())
        assert torch.equal(s.predict(pos, mt), f.predict(pos, mt))
        a, b = (x.loss_grad(pos, mt, tgt)[2][:wd.start] for x in (s, f))  # through the row-major copy
        assert float((a - b).norm()) <= 1e-5 * float(b.norm())
    finally:
        s.close()
        f.close()


def test_encoder_layers_past_the_small_tiles(env):
    """Hidden layers of 1544 units and a batch of 1280: the second layer, its weight gradient and the gradient of
    its input (1000, 1225 and 1000 small tiles, 1544, 1280 and 1544 deep) each run through a general kernel and
    the element-wise pass, the other products in small tiles; same formulas and bound as above."""
    test_encoder_layers_at_ragged_sizes(env, 1544, 24, 1280, 3)


@pytest.mark.parametrize("n_rcv, nt", [(1, 8), (3, 24), (5, 40), (4, 64)])
@pytest.mark.parametrize("B", [8, 136])
def test_component_scales_across_column_blocks(env, n_rcv, nt, B):
    """Served outputs take their component's scale 32 columns at a time, or column by column in a block on a
    component's edge (components of 8, 72 and 200 columns; of 256, none).  Scales that are powers of two
    change nothing else, so the outputs are exact multiples."""
    es, sur, torch = env
    s = sur.Surrogate(n_rcv, nt, nfreq=1, hidden=16, latent=8, max_batch=B, seed=5)
    try:
        g = torch.Generator().manual_seed(B + nt)
        pos, mt = torch.randn(B, 3, generator=g).clamp(-1, 1).cuda(), torch.randn(B, 6, generator=g).cuda()
        one = s.predict(pos, mt)
        scale = [2.0, 0.25, 8.0, 0.5]
        s.set_output_scale(scale)
        want = one.view(B, 4, -1) * torch.tensor(scale, device="cuda")[None, :, None]
        assert torch.equal(s.predict(pos, mt).view(B, 4, -1), want)
    finally:
        s.close()


def test_batches_of_millions(env):
    """A small network serves 2.2 million sources at once (68,750 row tiles of the encoder) and takes the losses
    of 4.3 million (67,188 tiles of the loss): each sample's result is that of a batch of 64."""
    es, sur, torch = env
    for B in (2_200_000, 4_300_000):
        s = sur.Surrogate(1, 8, nfreq=0, hidden=8, latent=8, max_batch=B, seed=2)
        try:
            g = torch.Generator(device="cuda").manual_seed(1)
            pos = torch.rand((B, 3), device="cuda", generator=g) * 2 - 1
            mt = torch.randn((B, 6), device="cuda", generator=g)
            tgt = torch.randn((B, s.D), device="cuda", generator=g)
            ends = [slice(0, 64), slice(B - 64, B)]
            if B < 3_000_000:
                out = s.predict(pos, mt)
                for e in ends:
                    assert torch.equal(out[e], s.predict(pos[e].contiguous(), mt[e].contiguous()))
            else:
                per = s.loss_grad(pos, mt, tgt, grads=False)[1]
                for e in ends:
                    assert torch.equal(per[e], s.loss_grad(pos[e].contiguous(), mt[e].contiguous(), tgt[e].contiguous(),
                                                           grads=False)[1])
        finally:
            s.close()
            torch.cuda.empty_cache()

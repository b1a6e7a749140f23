"""The float32 pair loop (packed, 32 x 128 tiles, 16-coordinate stages) at the edges of its
tiles: target counts around 32, source counts around the groups of 64 and tiles of 128 and
the source ranges, coordinate counts around a stage, every number of scales, with and
without noise coefficients -- each predicted log-weight against the FP64 oracle within the
float32 bar of the step tests, 1e-5 relative, plus what the multi-scale combination
amplifies (`combination_err_ok`)."""
import numpy as np
import pytest

from ._helpers import combination_err_ok, oracle_problem, rel_err, sobol_inputs

pytestmark = pytest.mark.gpu

NOISE = dict(u=0.7, u_kappa=0.8, u_zero=0, v=1.3, v_kappa=0.5)


@pytest.mark.parametrize("r,n,N,noise", [(1, 2, 1, False), (2, 31, 2, False), (15, 33, 3, False), (16, 64, 4, False),
                                         (17, 65, 1, False), (31, 127, 2, False), (32, 129, 3, False),
                                         (33, 257, 2, False), (63, 320, 2, False), (64, 321, 1, False),
                                         (65, 1025, 2, False), (129, 577, 3, False), (8, 20000, 2, False),
                                         (5, 63, 2, True), (16, 129, 1, True), (49, 700, 4, True)])
def test_prediction_at_tile_edges(yy_lib, r, n, N, noise):
    from oracle import filter as F
    from paper_2509_16896_gb300 import binding
    nz = NOISE if noise else None
    R = 0.3 if r > 8 else 1.0
    f = binding.Filter(binding.make_config(model="cubic", r=r, n=n, dt=0.01, R=R, n_scales=N, precision="f32", noise=nz))
    poly, scr = sobol_inputs(r, 40 + r)
    f.init_nodes(poly, scr, np.zeros(r))
    u, _ = f.get_nodes()
    p = oracle_problem("cubic", r, n, 0.01, R, N, noise=nz)
    rng = np.random.default_rng(r * 1000 + n)
    centre = rng.standard_normal(r)
    # weights of a posterior: a few nats apart, some nodes without weight
    lw = (-2.0 * rng.random(n) - np.log(n)).astype(np.float32)
    lw[rng.random(n) < 0.05] = -np.inf
    lw[0] = 0.0
    f.set_state(centre, lw, 0.0, 1)
    f.predict()
    pred, off = f.get_log_weights()
    prep = F.prepare(p, u, centre)
    lw64 = lw.astype(np.float64)
    Lj = F.kernel_lse(p, prep, lw64)
    ref, _ = F.combine(p, Lj, lw64, prep.mask)
    got = pred.astype(np.float64) + off
    # a row whose combination is within float32 error of zero may clamp on one side only
    both = np.isfinite(got) == np.isfinite(ref)
    assert both.mean() >= 0.99, np.nonzero(~both)[0][:5]
    ok, kappa = combination_err_ok(got[both], ref[both], Lj[both], p.coef, lw64[both], 1e-5)
    print(f"r={r} n={n} N={N} noise={noise}: largest condition number {kappa:.1f}")
    assert ok


@pytest.mark.parametrize("r,n,N", [(128, 300, 2), (130, 1000, 3), (200, 2049, 1), (256, 777, 4), (1000, 513, 2)])
@pytest.mark.parametrize("spread", [0.0, 60.0, 3000.0, 1e5])
@pytest.mark.parametrize("prec", ["f32", "f32s"])
def test_long_rows_with_spread_weights(yy_lib, prec, r, n, N, spread):
    """Long rows leave out terms that are zero in float32 next to the row's largest: the
    weights of a restart, of a posterior a few thousand nats wide (whole groups of sources
    drop out) and of the large-scale model after an update (1e5 nats), with dead and masked
    sources among them, in the plain form and behind the float32 screen (terms below
    e^-(ln n + 20)), against the oracle, which takes every term.  A log-weight of
    magnitude L carries its own float32 rounding, so the bar is relative to max(1, |ref|)."""
    from oracle import filter as F
    from paper_2509_16896_gb300 import binding
    f = binding.Filter(binding.make_config(model="cubic", r=r, n=n, dt=0.01, R=0.3, n_scales=N, precision=prec))
    poly, scr = sobol_inputs(r, 50 + r)
    f.init_nodes(poly, scr, np.zeros(r))
    u, _ = f.get_nodes()
    p = oracle_problem("cubic", r, n, 0.01, 0.3, N)
    rng = np.random.default_rng(r + n + int(spread))
    lw = (-spread * rng.random(n)).astype(np.float32)
    lw[rng.random(n) < 0.1] = -np.inf
    lw[n // 2] = 0.0
    centre = rng.standard_normal(r)
    f.set_state(centre, lw, 0.0, 1)
    f.predict()
    pred, off = f.get_log_weights()
    prep = F.prepare(p, u, centre)
    lw64 = lw.astype(np.float64)
    Lj = F.kernel_lse(p, prep, lw64)
    ref, _ = F.combine(p, Lj, lw64, prep.mask)
    got = pred.astype(np.float64) + off
    both = np.isfinite(got) == np.isfinite(ref)
    assert both.mean() >= 0.99, np.nonzero(~both)[0][:5]
    ok, _ = combination_err_ok(got[both], ref[both], Lj[both], p.coef, lw64[both], 1e-5)
    assert ok


@pytest.mark.parametrize("r,n,N,R", [(1, 2, 1, 2.0), (1, 300, 4, 5.0), (2, 1024, 2, 4.0), (3, 33, 2, 1.0), (8, 257, 3, 1.0),
                                     (23, 255, 2, 0.3), (47, 129, 2, 0.3), (63, 500, 3, 0.3), (64, 321, 1, 0.3)])
@pytest.mark.parametrize("spread", [2.0, 200.0])
def test_float64_short_rows(yy_lib, r, n, N, R, spread):
    """The float64 form that picks its pairs in float32: against the oracle at the edges of its
    source tiles and row blocks, narrow and wide weights, dead sources among them, within the
    float64 bar (1e-10 relative plus the combination's condition number)."""
    from oracle import filter as F
    from paper_2509_16896_gb300 import binding
    f = binding.Filter(binding.make_config(model="cubic", r=r, n=n, dt=0.01, R=R, n_scales=N, precision="f64"))
    poly, scr = sobol_inputs(r, 60 + r)
    f.init_nodes(poly, scr, np.zeros(r))
    u, _ = f.get_nodes()
    p = oracle_problem("cubic", r, n, 0.01, R, N)
    rng = np.random.default_rng(100 * r + n)
    lw = -spread * rng.random(n)
    lw[rng.random(n) < 0.05] = -np.inf
    lw[0] = 0.0
    centre = rng.standard_normal(r)
    f.set_state(centre, lw, 0.0, 1)
    f.predict()
    pred, off = f.get_log_weights()
    prep = F.prepare(p, u, centre)
    Lj = F.kernel_lse(p, prep, lw)
    ref, _ = F.combine(p, Lj, lw, prep.mask)
    got = pred + off
    both = np.isfinite(got) == np.isfinite(ref)
    assert both.mean() >= 0.99, np.nonzero(~both)[0][:5]
    ok, _ = combination_err_ok(got[both], ref[both], Lj[both], p.coef, lw[both], 1e-10, eps=2.0 ** -53)
    assert ok


@pytest.mark.parametrize("r,n,N", [(1, 100, 1), (2, 1500, 3), (9, 300, 1), (33, 200, 3), (64, 150, 1)])
@pytest.mark.parametrize("kind", ["weights", "distances", "both"])
def test_float64_short_rows_large_magnitudes(yy_lib, kind, r, n, N):
    """Scores far beyond float32's resolution of a nat: log-weights of 3e11 and more nats, and
    distances of 1e12 nats between the nodes (a step much shorter than the box), where a row
    without weight of its own has no near source.  Against the oracle within the float64 bar."""
    from oracle import filter as F
    from paper_2509_16896_gb300 import binding
    dt = 0.01 if kind == "weights" else 1e-13
    f = binding.Filter(binding.make_config(model="cubic", r=r, n=n, dt=dt, R=1.0, n_scales=N, precision="f64"))
    poly, scr = sobol_inputs(r, 70 + r)
    f.init_nodes(poly, scr, np.zeros(r))
    u, _ = f.get_nodes()
    p = oracle_problem("cubic", r, n, dt, 1.0, N)
    rng = np.random.default_rng(1000 * r + n)
    lw = -2.0 * rng.random(n) if kind == "distances" else -1e11 * (3.0 + rng.random(n))
    lw[rng.random(n) < 0.5] = -np.inf
    lw[n // 3] = 0.0 if kind == "distances" else -3e11 - 12345.678
    centre = rng.standard_normal(r)
    f.set_state(centre, lw, 0.0, 1)
    f.predict()
    pred, off = f.get_log_weights()
    prep = F.prepare(p, u, centre)
    Lj = F.kernel_lse(p, prep, lw)
    ref, _ = F.combine(p, Lj, lw, prep.mask)
    got = pred + off
    both = np.isfinite(got) == np.isfinite(ref)
    assert both.mean() >= 0.99, np.nonzero(~both)[0][:5]
    ok, _ = combination_err_ok(got[both], ref[both], Lj[both], p.coef, lw[both], 1e-10, eps=2.0 ** -53)
    assert ok


@pytest.mark.parametrize("r,n,N,R", [(1, 1025, 2, 2.0), (1, 2100, 1, 5.0), (7, 1800, 3, 1.0), (31, 600, 2, 0.3),
                                     (48, 353, 4, 0.05), (64, 129, 2, 0.05)])
def test_float64_short_rows_source_tiles(yy_lib, r, n, N, R):
    """Several source tiles, the last one ragged (a tile holds 1024 sources of short rows, 128 of
    64 coordinates), from boxes with few pairs in reach to boxes with all of them."""
    test_float64_short_rows(yy_lib, r, n, N, R, 2.0)


@pytest.mark.parametrize("r,n,N,R,spread", [(64, 4096, 1, 1.0, 2.0), (65, 4100, 2, 0.3, 60.0), (100, 4500, 2, 0.3, 2.0),
                                            (100, 5000, 3, 0.1, 2.0), (127, 4097, 4, 1.0, 3000.0)])
def test_float32_screen_of_mid_rows(yy_lib, r, n, N, R, spread):
    """The float32 screen below 128 coordinates, from boxes in which nearly every pair drops out to
    boxes in which none does: the screen is what runs (its launches, at least three), and the
    predictions are the oracle's within the float32 bar."""
    from oracle import filter as F
    from paper_2509_16896_gb300 import binding
    f = binding.Filter(binding.make_config(model="cubic", r=r, n=n, dt=0.01, R=R, n_scales=N, precision="f32s"))
    poly, scr = sobol_inputs(r, 80 + r)
    f.init_nodes(poly, scr, np.zeros(r))
    u, _ = f.get_nodes()
    p = oracle_problem("cubic", r, n, 0.01, R, N)
    rng = np.random.default_rng(r + n)
    lw = (-spread * rng.random(n)).astype(np.float32)
    lw[rng.random(n) < 0.1] = -np.inf
    lw[n // 2] = 0.0
    centre = rng.standard_normal(r)
    f.set_state(centre, lw, 0.0, 1)
    before = f.launches()
    f.predict()
    assert f.launches() - before >= 3
    pred, off = f.get_log_weights()
    prep = F.prepare(p, u, centre)
    lw64 = lw.astype(np.float64)
    Lj = F.kernel_lse(p, prep, lw64)
    ref, _ = F.combine(p, Lj, lw64, prep.mask)
    got = pred.astype(np.float64) + off
    both = np.isfinite(got) == np.isfinite(ref)
    assert both.mean() >= 0.99, np.nonzero(~both)[0][:5]
    ok, _ = combination_err_ok(got[both], ref[both], Lj[both], p.coef, lw64[both], 1e-5)
    assert ok


@pytest.mark.parametrize("r,n,N", [(200, 512, 2), (200, 513, 2), (511, 512, 1), (512, 512, 3), (700, 100, 2)])
@pytest.mark.parametrize("spread", [0.0, 3000.0])
def test_long_rows_with_few_sources(yy_lib, r, n, N, spread):
    """Both sides of the rule that leaves the skipping form out where there are few sources."""
    test_long_rows_with_spread_weights(yy_lib, "f32", r, n, N, spread)


@pytest.mark.parametrize("prec", ["f32", "f32s"])
@pytest.mark.parametrize("r,flat,n,N,dt,R", [(130, 0, 1000, 2, 1e-2, 0.3), (1000, 0, 700, 3, 1e-4, 0.3),
                                             (1000, 500, 1281, 1, 1e-8, 0.3), (300, 150, 897, 1, 1e-9, 1.0),
                                             (256, 100, 897, 1, 1e-9, 1.0), (256, 100, 929, 1, 1e-9, 1.0),
                                             (256, 100, 961, 1, 1e-9, 1.0), (256, 100, 993, 1, 1e-9, 1.0), (130, 0, 16384, 2, 1e-2, 0.3),
                                             (130, 0, 20000, 1, 1e-3, 0.3), (256, 100, 20000, 1, 1e-8, 0.5)])
@pytest.mark.parametrize("spread", [0.0, 1.0, 30.0])
def test_skipping_leaves_every_bit(yy_lib, prec, r, flat, n, N, dt, R, spread):
    """Long rows leave out only terms that are zero in float32: the prediction is, bit for bit,
    that of the form with noise coefficients, which takes every pair, at coefficients of one
    (the metric is one, its determinant's logarithm zero; linear drift, whose preparation is the
    same code for both).  The last `flat` coordinates have a box of no width to speak of, so that
    the sum is all there when it is tested, and n is 32 k + 1, so that the last block of targets has
    a row that nothing else keeps.  Steps so short that scores are 1e10 nats and their float32
    rounding is thousands, log-weights from equal to 30 times that spread; ranges of up to 313
    groups of sources.  Behind the float32 screen terms below e^-(ln n + 20) of the row's sum are missing:
    2e-9 of it, so 1e-6 relative (N = 1: no combination of scales to amplify it)."""
    from paper_2509_16896_gb300 import binding
    if prec == "f32s" and N > 1:
        N = 1
    one = dict(u=1.0, u_kappa=0.0, u_zero=0, v=1.0, v_kappa=0.0)
    poly, scr = sobol_inputs(r, 90)
    rng = np.random.default_rng(r + n)
    centre = rng.standard_normal(r)
    lw = (-spread * r * R * R / (3.0 * dt) * rng.random(n)).astype(np.float32)
    lw[rng.random(n) < 0.3] = -np.inf
    lw[n // 2] = 0.0
    half = np.full(r, R)
    half[r - flat:] = R * 1e-9
    out = []
    for p, nz in ((prec, None), ("f32", one)):
        f = binding.Filter(binding.make_config(model="linear", r=r, n=n, dt=dt, R=R, n_scales=N, precision=p, noise=nz))
        f.init_nodes(poly, scr, np.zeros(r), halfwidth=half)
        f.set_state(centre, lw, 0.0, 1)
        f.predict()
        lp, off = f.get_log_weights()
        out.append((lp, off))
    (a, oa), (b, ob) = out
    assert oa == ob
    assert np.isfinite(b).mean() >= 0.5 or N == 2
    if prec == "f32":
        assert np.array_equal(a, b)
    else:
        fin = np.isfinite(b)
        assert np.array_equal(fin, np.isfinite(a))
        assert np.all(np.abs(a[fin] - b[fin]) <= 1e-6 * np.maximum(1.0, np.abs(b[fin])))


@pytest.mark.parametrize("r,n,N,prefix", [(129, 1000, 2, 1), (191, 2049, 1, 3), (257, 1500, 3, 2), (300, 1025, 2, 5),
                                          (1000, 1500, 3, 16)])
@pytest.mark.parametrize("spread", [0.0, 60.0])
def test_float32_screen_first_pass_lengths(yy_lib, r, n, N, prefix, spread):
    """The float32 screen of long ragged rows at explicit lengths of its first pass (up to all
    coordinates): the plain form's prediction within the terms the screen may leave out."""
    from paper_2509_16896_gb300 import binding
    poly, scr = sobol_inputs(r, 95)
    rng = np.random.default_rng(r + n)
    centre = rng.standard_normal(r)
    lw = (-spread * rng.random(n)).astype(np.float32)
    lw[rng.random(n) < 0.1] = -np.inf
    lw[n // 2] = 0.0
    out = []
    for prec in ("f32", "f32s"):
        f = binding.Filter(binding.make_config(model="cubic", r=r, n=n, dt=0.01, R=0.3, n_scales=N, precision=prec,
                                               screen_prefix=prefix))
        f.init_nodes(poly, scr, np.zeros(r))
        f.set_state(centre, lw, 0.0, 1)
        f.predict()
        lp, off = f.get_log_weights()
        out.append(lp.astype(np.float64) + off)
    assert rel_err(out[1], out[0]) <= 2e-6

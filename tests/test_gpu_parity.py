"""GPU parity: the CUDA path, called through the C ABI, against the float64 CPU oracle on the
same seeded inputs.  Bar: completion depths equal; potentials within 1e-4 relative of the
oracle state at the same depth; achieved two-sided residual <= tol; slot counts exactly those
of Eq. 6-8.  Float64 arithmetic must meet it with no exception.  The default arithmetic
(fp32, or float64 exponents with fp32 exponentials when a lane's cost/eps range is beyond
fp32, or the tensor-core cross term for bf16 inputs) may sit one audit away only when the
oracle's own residual at the disputed audit is within 1e-5 relative of tol (or the decay-scaled
bound of helpers.miss_allowed for very slow lanes); every such lane goes into the ledger that
tests/test_yy_parity_ledger.py bounds and writes out.  Pure fp32 arithmetic is held to the
same bar where its error model says it can meet it, and to its documented limits elsewhere."""
import os
import ctypes

import numpy as np
import pytest

from helpers import (LEDGER, check_accounting, check_against_oracle, close_entry, compare_lane, new_entry,
                     pot_err, run_gpu)
from paper_2607_24741_b200 import workloads as wl

pytestmark = pytest.mark.gpu

POT_TOL_F32 = 1e-4      # acceptance bar for fp32 pair arithmetic
POT_TOL_F64 = 1e-9      # float64 pair arithmetic: differences are summation order only
MARGIN_F32 = 2e-2       # pure fp32: a +-1 lane must have |r - tol|/tol below this at the disputed audit
MARGIN_AUTO = 1e-5      # default arithmetic: fp32 exponential error (2^-22) over a ~1%/cycle decay

CASES = {
    "tiny": dict(name="tiny"),
    "sensor_ragged": dict(name="sensor", W=16, n=200, m=264),
    "registration_small": dict(name="registration", W=4, n=1000),
    "sweep_small": dict(name="sweep", W=48, n=100, m=77, max_iter=3000),
    "feature_small": dict(name="feature", W=4, n=200, m=333, d=80),      # bf16 inputs, large-d kernels
}
DEEP_CASES = {
    "feature_tensor": dict(name="feature", W=4, n=256, m=320, d=128),    # bf16 inputs on the tensor cores
}


def _make(case):
    kw = dict(CASES[case] if case in CASES else DEEP_CASES[case]); name = kw.pop("name")
    return wl.make(name, **kw)


@pytest.mark.parametrize("case", list(CASES))
@pytest.mark.parametrize("mode", ["active", "masked"])
def test_f64_arithmetic_reproduces_oracle_exactly(oracle, case, mode):
    w = _make(case)
    W = w.shape[0]
    r = run_gpu(w, mode=mode, compute="f64")
    misses = check_against_oracle(oracle, w, r, range(W), pot_tol=POT_TOL_F64, exact_depth=True)
    assert misses == []
    check_accounting(oracle, r, W, mode)


@pytest.mark.parametrize("case", list(CASES))
def test_default_arithmetic_meets_the_bar(oracle, case):
    w = _make(case)
    W = w.shape[0]
    r = run_gpu(w, mode="active")
    check_against_oracle(oracle, w, r, range(W), pot_tol=POT_TOL_F32, exact_depth=False, floor=MARGIN_AUTO,
                         label=f"default arithmetic, {case}")
    check_accounting(oracle, r, W, "active")
    # the float getter is the float64 one rounded
    np.testing.assert_array_equal(r["f32"], r["f"].astype(np.float32))


@pytest.mark.parametrize("case", ["tiny", "sensor_ragged", "registration_small"])
@pytest.mark.parametrize("cost_form", [0, 1, 2])
def test_pure_fp32_arithmetic_where_it_suffices(oracle, case, cost_form):
    # scaled squared radius up to a few hundred: fp32 exponents are good to ~1e-5
    w = _make(case)
    W = w.shape[0]
    r = run_gpu(w, mode="active", compute="f32", cost_form=cost_form)
    misses = check_against_oracle(oracle, w, r, range(W), pot_tol=POT_TOL_F32, exact_depth=False, floor=MARGIN_F32,
                                  label=f"pure fp32 (forced), {case}, cost form {cost_form}")
    assert len(misses) <= max(1, W // 8)


def test_pure_fp32_limits_on_small_eps_lanes(oracle):
    # eps down to 0.01 on unit-variance 8-d clouds: cost/eps ~ 10^3 even for the closest pair, so
    # an fp32 exponent carries ~1e-4 and slow lanes amplify it.  This is why the default
    # arithmetic leaves fp32 for such batches; the pure fp32 numbers are recorded, not hidden.
    w = _make("sweep_small")
    W = w.shape[0]
    o = oracle.solve_batch(w.x, w.y, w.a, w.b, w.eps, w.tol, max_iter=w.max_iter)
    r = run_gpu(w, mode="active", compute="f32")
    dd = r["depth"].astype(np.int64) - o.depth
    e = pot_err(r["f"], r["g"], o.f, o.g, w.eps.astype(np.float64))
    print(f"[fp32 limits] lanes off: {np.count_nonzero(dd)}/{W}, max |depth diff| {np.abs(dd).max()}, "
          f"max potential error on equal-depth lanes {e[dd == 0].max():.2e}")
    assert np.abs(dd).max() <= 4 and e[dd == 0].max() <= 1e-3
    np.testing.assert_array_equal(r["status"], o.status)
    ra = run_gpu(w, mode="active")
    assert np.array_equal(ra["depth"], o.depth)


@pytest.mark.parametrize("case", ["tiny", "sweep_small"])
@pytest.mark.parametrize("compute", ["f32", "auto", "f64"])
def test_masked_equals_active_bitwise_and_static_matches_fixed_depth(oracle, case, compute):
    w = _make(case)
    W = w.shape[0]
    ra = run_gpu(w, mode="active", compute=compute)
    rm = run_gpu(w, mode="masked", compute=compute)
    rs = run_gpu(w, mode="static", compute=compute)
    # same update, screen, check, tolerance and completion times (logical-mask control)
    np.testing.assert_array_equal(ra["depth"], rm["depth"])
    np.testing.assert_array_equal(ra["f"], rm["f"]); np.testing.assert_array_equal(ra["g"], rm["g"])
    np.testing.assert_array_equal(ra["r_row"], rm["r_row"])
    # fixed-width control: same first-pass depths, every lane carried to l_max
    np.testing.assert_array_equal(ra["depth"], rs["depth"])
    lmax = int(ra["depth"].max())
    check_accounting(oracle, rs, W, "static"); check_accounting(oracle, rm, W, "masked")
    ref = oracle.solve_batch(w.x, w.y, w.a, w.b, w.eps, w.tol, max_iter=w.max_iter, fixed_cycles=lmax)
    done = ra["status"] == 1
    e = pot_err(rs["f"], rs["g"], ref.f, ref.g, w.eps.astype(np.float64))
    assert e[done].max() <= {"f32": 1e-3, "auto": POT_TOL_F32, "f64": POT_TOL_F64}[compute]
    assert np.all(rs["r_row"][done] <= w.tol)
    # removable slots R = W*l_max - sum l_t (Eq. 8)
    assert rs["stats"]["slots"] - ra["stats"]["slots"] == W * lmax - int(ra["depth"].sum())


@pytest.mark.parametrize("case,compute", [("sensor_ragged", "f32"), ("sweep_small", "mixed"), ("tiny", "f64")])
def test_early_exit_mask_arm_equals_the_mask_control_bitwise(oracle, case, compute):
    # the extra arm skips the pair work of frozen lanes: same bits as MASKED, but only the slots of ACTIVE
    w = _make(case)
    W = w.shape[0]
    rm = run_gpu(w, mode="masked", compute=compute)
    re = run_gpu(w, mode="masked_exit", compute=compute)
    np.testing.assert_array_equal(rm["depth"], re["depth"]); np.testing.assert_array_equal(rm["status"], re["status"])
    np.testing.assert_array_equal(rm["f"], re["f"]); np.testing.assert_array_equal(rm["g"], re["g"])
    np.testing.assert_array_equal(rm["r_row"], re["r_row"]); np.testing.assert_array_equal(rm["r_col"], re["r_col"])
    assert re["stats"]["slots"] == int(re["depth"].sum()) and rm["stats"]["slots"] == W * int(rm["depth"].max())
    np.testing.assert_array_equal(np.array(re["stats"]["widths"]), oracle.slot_counts(re["depth"].astype(np.int64))["widths"])


def test_rows_per_thread_follow_the_width_without_changing_bits():
    # Mixed arithmetic launches four rows per thread while the grid fills the GPU and two rows once it does
    # not; MASKED never shrinks and stays on the one-launch-per-leg kernels, while ACTIVE runs the 1024
    # lanes through the multi-cycle cluster kernel (two rows per thread, state in shared memory).  A row's
    # arithmetic depends neither on the thread that holds it nor on the rows that share its block, and
    # residual terms are summed as integers, so the two modes must agree bit for bit at full size.
    w = wl.make("sweep")
    ra = run_gpu(w, mode="active", compute="mixed", widths_cap=10)
    rm = run_gpu(w, mode="masked", compute="mixed", widths_cap=10)
    np.testing.assert_array_equal(ra["depth"], rm["depth"])
    np.testing.assert_array_equal(ra["f"], rm["f"]); np.testing.assert_array_equal(ra["g"], rm["g"])
    np.testing.assert_array_equal(ra["r_row"], rm["r_row"]); np.testing.assert_array_equal(ra["r_col"], rm["r_col"])


def test_packing_commutes_with_the_per_lane_map(oracle):
    # Eq. 2: a W-lane batch gives each lane what a one-lane batch gives it, bit for bit
    # (the arithmetic is fixed here: the automatic choice looks at the whole batch)
    w = wl.make("sweep", W=6, n=96, m=80, max_iter=2000)
    for compute in ("mixed", "f32"):
        r = run_gpu(w, mode="active", column_split=4, compute=compute)
        for t in (0, 3, 5):
            one = wl.Workload(w.name, w.x[t:t + 1], w.y[t:t + 1], w.a[t:t + 1], w.b[t:t + 1],
                              w.eps[t:t + 1], w.tol, w.max_iter)
            r1 = run_gpu(one, mode="active", column_split=4, compute=compute)
            assert r1["depth"][0] == r["depth"][t]
            np.testing.assert_array_equal(r1["f"][0], r["f"][t]); np.testing.assert_array_equal(r1["g"][0], r["g"][t])
        r2 = run_gpu(w, mode="active", column_split=4, compute=compute)      # run-to-run determinism
        np.testing.assert_array_equal(r2["f"], r["f"]); np.testing.assert_array_equal(r2["depth"], r["depth"])


@pytest.mark.parametrize("cs", [1, 4, 32])
def test_every_column_split_agrees_with_the_oracle(oracle, cs):
    w = wl.make("sensor", W=5, n=150, m=333)
    r = run_gpu(w, mode="active", compute="f64", column_split=cs)
    assert check_against_oracle(oracle, w, r, range(5), pot_tol=POT_TOL_F64, exact_depth=True) == []
    w3 = wl.make("registration", W=3, n=700)
    r3 = run_gpu(w3, mode="active", column_split=cs)
    check_against_oracle(oracle, w3, r3, range(3), pot_tol=POT_TOL_F32, exact_depth=False, floor=MARGIN_AUTO,
                         label=f"registration n=700, column split {cs}")


def test_audit_grid_screen_threshold_and_iteration_limit(oracle):
    w = wl.make("tiny")
    r4 = run_gpu(w, compute="f64", audit_every=4)
    assert np.all(r4["depth"] % 4 == 0)
    assert check_against_oracle(oracle, w, r4, range(8), pot_tol=POT_TOL_F64, exact_depth=True, audit_every=4) == []
    rs = run_gpu(w, compute="f64", tol_screen=5e-4)
    assert check_against_oracle(oracle, w, rs, range(8), pot_tol=POT_TOL_F64, exact_depth=True, tol_screen=5e-4) == []
    assert np.all(rs["r_row"] <= 5e-4)
    cap = int(np.median(r4["depth"]))
    rl = run_gpu(w, compute="f64", max_iter=cap)
    assert check_against_oracle(oracle, w, rl, range(8), pot_tol=POT_TOL_F64, exact_depth=True, max_iter=cap) == []
    assert set(rl["status"]) == {1, 2} and rl["depth"].max() == cap
    assert np.all(np.isnan(rl["r_col"][rl["status"] == 2]))
    check_accounting(oracle, rl, 8, "active")


def test_degenerate_shapes(oracle):
    one = wl.Workload("one", np.array([[[1.0, 2.0]]], np.float32), np.array([[[4.0, 6.0]]], np.float32),
                      np.ones((1, 1), np.float32), np.ones((1, 1), np.float32),
                      np.array([0.3], np.float32), 1e-6, 50)
    r = run_gpu(one, compute="f64")
    assert r["depth"][0] == 1 and r["f"][0, 0] + r["g"][0, 0] == pytest.approx(25.0, rel=1e-12)
    w = wl.make("sensor", W=1, n=3, m=5)                          # far below one tile
    r = run_gpu(w, compute="f64")
    assert check_against_oracle(oracle, w, r, [0], pot_tol=POT_TOL_F64, exact_depth=True) == []
    w = wl.make("sweep", W=300, n=8, m=9, max_iter=400)            # W beyond one scan block... of lanes
    r = run_gpu(w, compute="f64")
    assert check_against_oracle(oracle, w, r, [0, 17, 255, 299], pot_tol=POT_TOL_F64, exact_depth=True,
                                max_iter=400) == []
    check_accounting(oracle, r, 300, "active")


@pytest.mark.parametrize("compute", ["auto", "f32", "mixed"])
def test_degenerate_lanes_in_the_fast_arithmetics(oracle, compute):
    # the cases the method itself degenerates on, in the arithmetics and kernels a default batch runs
    # (lanes this small go through the multi-cycle kernels): single points, one point against many,
    # coincident clouds (zero cost on the diagonal) and a cloud collapsed to one location (all costs
    # equal: the product coupling is optimal and the first audit passes)
    rng = np.random.default_rng(11)
    f32 = np.float32

    def lanes(x, y, a, b, eps, tol=1e-4, max_iter=400, name="degenerate"):
        return wl.Workload(name, x.astype(f32), y.astype(f32), a.astype(f32), b.astype(f32), eps.astype(f32), tol, max_iter)

    def uniform(W, n):
        return np.full((W, n), 1.0 / n)

    W = 3
    cases = []
    # one point against one point
    cases.append(lanes(rng.normal(size=(W, 1, 2)), rng.normal(size=(W, 1, 2)), uniform(W, 1), uniform(W, 1),
                       np.array([0.3, 0.1, 1.0])))
    # one point against seven, and seven against one
    wts = rng.uniform(0.5, 1.5, size=(W, 7)); wts /= wts.sum(axis=1, keepdims=True)
    cases.append(lanes(rng.normal(size=(W, 1, 3)), rng.normal(size=(W, 7, 3)), uniform(W, 1), wts, np.array([0.3, 0.1, 1.0])))
    cases.append(lanes(rng.normal(size=(W, 7, 3)), rng.normal(size=(W, 1, 3)), wts, uniform(W, 1), np.array([0.3, 0.1, 1.0])))
    # the same cloud on both sides
    pts = rng.normal(size=(W, 9, 2))
    cases.append(lanes(pts, pts.copy(), uniform(W, 9), uniform(W, 9), np.array([0.5, 0.2, 0.1])))
    # every point of both clouds at one location
    spot = np.broadcast_to(rng.normal(size=(W, 1, 4)), (W, 6, 4)).copy()
    cases.append(lanes(spot, spot[:, :5].copy(), uniform(W, 6), uniform(W, 5), np.array([0.5, 0.2, 0.1])))
    for k, w in enumerate(cases):
        if compute == "f32":
            w.tol = 1e-3          # pure fp32 by name: its evaluation error is ~2e-6 absolute here (eps 0.05 .. 1)
        r = run_gpu(w, compute=compute)
        if compute == "auto" and k == 3:
            # the automatic choice follows the tolerance: lane 2 has a scaled squared radius of 60, which
            # is fp32 territory at a tolerance of 1e-3 (limit 512) and not at 1e-4 (limit 51)
            assert r["arith"] == "mixed"
            w.tol = 1e-3
            assert run_gpu(w, compute="auto")["arith"] == "f32"
            w.tol = 1e-4
        assert (r["status"] == 1).all(), (k, r["status"])
        assert check_against_oracle(oracle, w, r, list(range(W)), pot_tol=POT_TOL_F32, exact_depth=False,
                                    label=f"degenerate lanes, case {k}, {compute}") == [], k
    # collapsed clouds: all costs equal, so f = g = const solves the problem after one cycle
    assert (r["depth"] == 1).all(), r["depth"]


def test_step_runs_fixed_cycles_and_running_lanes_are_readable(oracle):
    import torch
    from paper_2607_24741_b200 import binding as B
    w = wl.make("tiny")
    dev = torch.device("cuda:0")
    t = lambda v: torch.from_numpy(v).to(dev)
    sb = B.SinkhornBatch(t(w.x), t(w.y), t(w.a), t(w.b), t(w.eps), w.tol, mode="static", compute="f64")
    sb.step(7)
    f, g = sb.potentials(f64=True)
    assert sb.active() == 8
    ref = oracle.solve_batch(w.x, w.y, w.a, w.b, w.eps, w.tol, fixed_cycles=7)
    # after 7 enqueued cycles the g-leg of cycle 7 has run: state (f7, g7)
    assert pot_err(f.cpu().numpy(), g.cpu().numpy(), ref.f, ref.g, w.eps.astype(np.float64)).max() <= POT_TOL_F64
    sb.drain(); assert sb.active() == 0
    sb.close()


def test_bad_inputs_are_reported_not_trapped():
    import torch
    from paper_2607_24741_b200 import binding as B
    w = wl.make("tiny")
    dev = torch.device("cuda:0")
    t = lambda v: torch.from_numpy(v).to(dev)
    a = w.a.copy(); a[2, 5] = 0.0
    sb = B.SinkhornBatch(t(w.x), t(w.y), t(a), t(w.b), t(w.eps), w.tol)
    with pytest.raises(B.SkbError) as e:
        sb.drain()
    assert e.value.code == 3
    sb.close()
    eps = w.eps.copy(); eps[1] = -1.0
    sb = B.SinkhornBatch(t(w.x), t(w.y), t(w.a), t(w.b), t(eps), w.tol)
    with pytest.raises(B.SkbError):
        sb.drain()
    sb.close()
    with pytest.raises(B.SkbError):
        B.SinkhornBatch(t(w.x), t(w.y), t(w.a), t(w.b), t(w.eps), -1.0)
    cfg = B.make_config(8, 64, 64, 2)
    cfg.workspace_bytes = 16
    h = ctypes.c_void_p()
    ws = torch.empty(1024, dtype=torch.uint8, device=dev)
    cfg.workspace = ws.data_ptr()
    rc = B.lib.sinkhorn_batch_create(t(w.x).data_ptr(), t(w.y).data_ptr(), t(w.a).data_ptr(), t(w.b).data_ptr(),
                                     t(w.eps).data_ptr(), 1e-3, ctypes.byref(cfg), ctypes.byref(h))
    assert rc == 4 and b"workspace too small" in B.lib.sinkhorn_batch_last_error(None)


def test_host_buffer_call_matches_device_call(oracle):
    import torch
    from paper_2607_24741_b200 import binding as B
    w = wl.make("sensor", W=8, n=128)
    r = run_gpu(w)
    W, n, m, d = w.shape
    cfg = B.make_config(W, n, m, d, max_iter=w.max_iter)
    need = B.sinkhorn_batch_host_workspace_bytes(cfg)
    ws = torch.empty(need, dtype=torch.uint8, device="cuda:0")
    cfg.workspace = ws.data_ptr(); cfg.workspace_bytes = need
    f = np.empty((W, n), np.float32); g = np.empty((W, m), np.float32)
    depth = np.empty(W, np.int32); status = np.empty(W, np.int32)
    rr = np.empty(W, np.float32); rc = np.empty(W, np.float32)
    slots = ctypes.c_longlong(0); cycles = ctypes.c_int(0)
    p = lambda v: v.ctypes.data_as(ctypes.c_void_p)
    code = B.lib.sinkhorn_batch_solve_host(p(w.x), p(w.y), p(w.a), p(w.b), p(w.eps), w.tol, ctypes.byref(cfg),
                                           p(f), p(g), p(depth), p(status), p(rr), p(rc),
                                           ctypes.byref(slots), ctypes.byref(cycles))
    assert code == 0
    np.testing.assert_array_equal(depth, r["depth"]); np.testing.assert_array_equal(f, r["f32"])
    np.testing.assert_array_equal(g, r["g32"]); assert slots.value == r["stats"]["slots"]


# ---- the five workloads at their full sizes, in the launch configuration the benchmark times
#      (ACTIVE, default arithmetic); the oracle runs one whole lane per host core
FULL = {
    "tiny": range(8),
    "sensor": range(256),                       # every lane: the oracle needs well under a second for all of them
    "feature": list(range(64)),
    "sweep": list(range(1024)),
}


@pytest.mark.parametrize("name", list(FULL))
def test_full_size_lanes_against_oracle(oracle, name):
    lanes = FULL[name]
    w = wl.make(name)
    W = w.shape[0]
    r = run_gpu(w, mode="active")
    check_against_oracle(oracle, w, r, lanes, pot_tol=POT_TOL_F32, exact_depth=False, floor=MARGIN_AUTO,
                         label=f"full size, {name}")
    # properties that hold at any size
    depth = r["depth"].astype(np.int64)
    assert np.all(r["status"] == 1) and np.all(r["r_row"] <= w.tol)
    assert r["stats"]["slots"] == depth.sum() and r["cycles"] == depth.max()
    np.testing.assert_array_equal(np.array(r["stats"]["widths"]), oracle.survivor_widths(depth))


class _Stored:
    """One lane of tests/golden/registration_n8192.npz in the shape compare_lane expects."""
    def __init__(self, z, i, prefix="", stride=1):
        k_ = lambda name: z[prefix + name][i]
        self.depth = int(k_("depth")); self.status = int(k_("status"))
        self.f, self.g = k_("f"), k_("g")
        self.f_prev, self.g_prev = k_("f_prev"), k_("g_prev")
        self.f_next, self.g_next = k_("f_next"), k_("g_next")
        tail = k_("hist")
        self.hist = np.full(self.depth, np.nan)
        k = min(len(tail), self.depth)
        self.hist[self.depth - k:] = tail[len(tail) - k:]
        self.r_row = float(k_("r_row"))
        self.stride = stride                 # potentials hold every stride-th point


def test_full_size_registration_against_stored_oracle(oracle):
    # One oracle lane at n = m = 8192 takes a quarter of an hour, so the oracle's results are stored
    # (tests/golden/make_registration_golden.py wrote them, calling the oracle only): twelve lanes with
    # their full potentials, the other twenty with every eighth point.  Every lane of the workload is
    # held to the oracle's depth; the float64 residual evaluation of the emitted state is cheap enough
    # to run here.
    z = np.load(os.path.join(os.path.dirname(__file__), "golden", "registration_n8192.npz"))
    w = wl.make("registration")
    W, n, m, d = w.shape
    assert int(z["n"]) == n and float(z["tol"]) == w.tol
    r = run_gpu(w, mode="active")
    depth = r["depth"].astype(np.int64)
    assert np.all(r["status"] == 1) and np.all(r["r_row"] <= w.tol) and np.all(depth > 50)
    assert r["stats"]["slots"] == depth.sum() and r["cycles"] == depth.max()
    np.testing.assert_array_equal(np.array(r["stats"]["widths"]), oracle.survivor_widths(depth))
    lanes = [int(t) for t in z["lanes"]]
    stored = [(t, _Stored(z, i)) for i, t in enumerate(lanes)]
    if "light_lanes" in z.files:
        stored += [(int(t), _Stored(z, i, "light_", int(z["stride"]))) for i, t in enumerate(z["light_lanes"])]
        assert sorted(t for t, _ in stored) == list(range(W))            # every lane of the workload
    entry = new_entry("full size, registration (stored oracle)", w, r, [t for t, _ in stored], w.tol, MARGIN_AUTO)
    misses = []
    for t, o in stored:
        assert abs(o.r_row - o.hist[-1]) <= 1e-15
        miss = compare_lane(oracle, w, r, t, o, pot_tol=POT_TOL_F32, exact_depth=False, tol=w.tol, entry=entry)
        if miss is not None:
            misses.append(miss)
    close_entry(entry, misses, MARGIN_AUTO)
    t = lanes[0]
    # one more oracle cycle from the emitted state still passes and lowers the row residual
    C = oracle.cost_matrix(w.x[t], w.y[t])
    f1 = oracle.f_leg(C, r["g"][t], w.a[t], float(w.eps[t])); g1 = oracle.g_leg(C, f1, w.b[t], float(w.eps[t]))
    row, col = oracle.marginals(C, f1, g1, float(w.eps[t]))
    rr0, _ = oracle.residuals(w.x[t], w.y[t], w.a[t], w.b[t], float(w.eps[t]), r["f"][t], r["g"][t])
    assert np.abs(row - w.a[t]).sum() < rr0


@pytest.mark.parametrize("seed", [2, 3])
def test_random_configurations(oracle, seed):
    # sixty random combinations of law, shape (down to one point, ragged, d = 1 .. 40), mode, audit
    # grid, column split, cost form, screen threshold and guard band, in float64 (exact depths, exact
    # accounting) and mixed arithmetic (the usual bar)
    rng = np.random.default_rng(seed)
    for it in range(60):
        name = str(rng.choice(["sensor", "sweep", "tiny", "registration"]))
        W = int(rng.choice([1, 2, 3, 7, 16, 33]))
        kw = dict(W=W, n=int(rng.choice([1, 2, 5, 31, 64, 100, 129, 300])), max_iter=int(rng.choice([50, 400, 1500])))
        if name != "registration":
            kw["m"] = int(rng.choice([1, 3, 8, 33, 64, 77, 128, 257]))
        if name in ("sensor", "sweep"):
            kw["d"] = int(rng.choice([1, 2, 3, 4, 6, 8, 15, 16, 24, 32, 40]))
        w = wl.make(name, **kw)
        mode = str(rng.choice(["active", "masked", "static", "masked_exit"]))
        compute = str(rng.choice(["f64", "mixed"]))
        opts = dict(mode=mode, compute=compute, audit_every=int(rng.choice([1, 1, 2, 5])),
                    column_split=int(rng.choice([0, 0, 1, 4, 32])), cost_form=int(rng.choice([0, 0, 1, 2])),
                    guard_band=float(rng.choice([0.0, -1.0, 0.5])))
        if rng.random() < 0.3:
            opts["tol_screen"] = float(w.tol * rng.choice([0.5, 2.0]))
        what = f"random configuration {seed}/{it}: {name} {kw} {opts}"
        r = run_gpu(w, **opts)
        exact = compute == "f64"
        if mode == "static":
            ref = oracle.solve_batch(w.x, w.y, w.a, w.b, w.eps, w.tol, fixed_cycles=r["cycles"])
            err = pot_err(r["f"], r["g"], ref.f, ref.g, w.eps.astype(np.float64)).max()
            assert err <= (POT_TOL_F64 if exact else POT_TOL_F32), (what, err)
            assert r["stats"]["slots"] == r["cycles"] * W, what
        else:
            misses = check_against_oracle(oracle, w, r, range(W), pot_tol=POT_TOL_F64 if exact else POT_TOL_F32,
                                          exact_depth=exact, floor=None if exact else MARGIN_AUTO, max_iter=kw["max_iter"],
                                          audit_every=opts["audit_every"], tol_screen=opts.get("tol_screen", 0.0), label=what)
            assert not exact or misses == [], what
            if exact:
                check_accounting(oracle, r, W, "active" if mode == "masked_exit" else mode)


def test_four_batches_running_on_four_streams():
    # one batch per stream, four arithmetics / kernel families, stepped in turn without any
    # synchronisation in between: every batch ends with the bits it has when it runs alone
    import torch
    from paper_2607_24741_b200 import binding as B
    dev = torch.device("cuda:0")
    t = lambda v: torch.from_numpy(v).to(dev)
    cases = [wl.make("tiny"), _make("sensor_ragged"), _make("sweep_small"), _make("feature_tensor")]
    alone = [run_gpu(w) for w in cases]
    batches = []
    try:
        for w in cases:
            x, y = t(w.x), t(w.y)
            if w.xy_dtype == "bf16":
                x, y = x.bfloat16(), y.bfloat16()
            torch.cuda.synchronize()
            batches.append(B.SinkhornBatch(x, y, t(w.a), t(w.b), t(w.eps), w.tol, max_iter=w.max_iter,
                                           stream=torch.cuda.Stream(dev)))
        for _ in range(450):
            for sb in batches:
                sb.step(7)
        for sb, ref in zip(batches, alone):
            sb.drain()
            f, g = sb.potentials(f64=True)
            depth, _ = sb.depths()
            np.testing.assert_array_equal(depth.cpu().numpy(), ref["depth"])
            np.testing.assert_array_equal(f.cpu().numpy(), ref["f"]); np.testing.assert_array_equal(g.cpu().numpy(), ref["g"])
            assert sb.check_guards() == -1
    finally:
        for sb in batches:
            sb.close()


def test_host_threads_that_launch_the_same_kernels_for_different_shapes():
    # shapes that run the same kernels with different amounts of shared memory (deep lanes by d, lanes of several blocks by
    # their number, spatial order by the dimension), each from a host thread of its own, again and again: no thread's launch
    # may fail for what another has set, and every batch ends with the bits it has alone
    import threading
    import torch
    from paper_2607_24741_b200 import binding as B
    dev = torch.device("cuda:0")
    t = lambda v: torch.from_numpy(v).to(dev)
    kws = [dict(name="feature", W=2, n=40, m=100, d=64), dict(name="feature", W=2, n=40, m=100, d=512),
           dict(name="feature", W=2, n=140, m=300, d=64), dict(name="feature", W=2, n=900, m=300, d=64),
           dict(name="sensor", W=2, n=140, m=300), dict(name="sensor", W=2, n=1000, m=300),
           dict(name="registration", W=1, n=1024), dict(name="registration", W=1, n=1024)]
    work, alone = [], []
    for i, kw in enumerate(kws):
        w = wl.make(**kw, max_iter=10)
        if i == len(kws) - 1:                                          # the same law in the plane
            w.x, w.y = np.ascontiguousarray(w.x[:, :, :2]), np.ascontiguousarray(w.y[:, :, :2])
        alone.append(run_gpu(w))
        x, y = t(w.x), t(w.y)
        work.append((x.bfloat16(), y.bfloat16(), t(w.a), t(w.b), t(w.eps)) if w.xy_dtype == "bf16" else (x, y, t(w.a), t(w.b), t(w.eps)))
    torch.cuda.synchronize()
    failed = []

    def run(i):
        try:
            for _ in range(30):
                sb = B.SinkhornBatch(*work[i], 1e-3, max_iter=10, stream=streams[i])
                sb.drain()
                with torch.cuda.stream(streams[i]):
                    f, _g = sb.potentials(f64=True)
                streams[i].synchronize()
                np.testing.assert_array_equal(f.cpu().numpy(), alone[i]["f"])
                sb.close()
        except Exception as e:                                          # noqa: BLE001 (reported below, from the main thread)
            failed.append((i, repr(e)[:300]))
    streams = [torch.cuda.Stream(dev) for _ in work]
    threads = [threading.Thread(target=run, args=(i,)) for i in range(len(work))]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert not failed, failed


# ---- the paper's guard: a stricter threshold inside, the reported tolerance outside ----------------
@pytest.mark.parametrize("case", list(CASES))
def test_guarded_thresholds_meet_the_reported_tolerance_without_slack(oracle, case):
    # Section "Screen, verify, and compact": screen and check run at 9.5e-4, the output is reported at
    # 1e-3.  Both sides get the guarded threshold; the float64 residual of every emitted state must then
    # be within the REPORTED tolerance with no allowance for the GPU's arithmetic.
    w = _make(case)
    W = w.shape[0]
    guard, reported = 9.5e-4, 1e-3
    r = run_gpu(w, mode="active", tol=guard)
    check_against_oracle(oracle, w, r, range(W), pot_tol=POT_TOL_F32, exact_depth=False, tol=guard, floor=MARGIN_AUTO,
                         label=f"guard arm 9.5e-4 -> 1e-3, {case}", report_tol=reported)
    check_accounting(oracle, r, W, "active")


# ---- tensor-core cross term (bf16 inputs, d a multiple of 64) ------------------------------------
# (bf16 products are exact in fp32 and accumulate in fp32, so the error model is the default
# arithmetic's: same margin, same potential bar; the acceptance bar for bf16 inputs, 5e-3, is far looser.)
@pytest.mark.parametrize("kw", [dict(W=3, n=200, m=333, d=64), dict(W=2, n=256, d=128), dict(W=2, n=129, m=640, d=512)])
def test_tensor_core_path_against_oracle(oracle, kw):
    w = wl.make("feature", **kw)
    W = w.shape[0]
    r = run_gpu(w, mode="active", compute="tensor")
    check_against_oracle(oracle, w, r, range(W), pot_tol=POT_TOL_F32, exact_depth=False, floor=MARGIN_AUTO,
                         label=f"tensor cores, {kw}")
    check_accounting(oracle, r, W, "active")
    # what AUTO picks for such inputs is this very path: bit-identical results
    ra = run_gpu(w, mode="active")
    np.testing.assert_array_equal(ra["f"], r["f"]); np.testing.assert_array_equal(ra["depth"], r["depth"])


def test_tensor_core_modes_and_compaction(oracle):
    w = wl.make("feature", W=6, n=256, d=128)
    ra = run_gpu(w, mode="active", compute="tensor")
    rm = run_gpu(w, mode="masked", compute="tensor")
    rs = run_gpu(w, mode="static", compute="tensor")
    np.testing.assert_array_equal(ra["depth"], rm["depth"]); np.testing.assert_array_equal(ra["depth"], rs["depth"])
    np.testing.assert_array_equal(ra["f"], rm["f"]); np.testing.assert_array_equal(ra["g"], rm["g"])
    assert len(set(ra["depth"].tolist())) > 1                    # lanes really leave at different depths
    check_accounting(oracle, ra, 6, "active"); check_accounting(oracle, rs, 6, "static")
    rx = run_gpu(w, mode="masked_exit", compute="tensor")         # frozen lanes' blocks return at once: same bits
    np.testing.assert_array_equal(rx["f"], rm["f"]); np.testing.assert_array_equal(rx["depth"], rm["depth"])
    assert rx["stats"]["slots"] == ra["stats"]["slots"]
    ref = oracle.solve_batch(w.x, w.y, w.a, w.b, w.eps, w.tol, max_iter=w.max_iter)
    np.testing.assert_array_equal(ra["depth"], ref.depth)
    assert pot_err(ra["f"], ra["g"], ref.f, ref.g, w.eps.astype(np.float64)).max() <= POT_TOL_F32


@pytest.mark.parametrize("kw", [dict(W=5, n=300, m=520, d=320), dict(W=2, n=140, m=2400, d=512)])
def test_tensor_core_pair_kernel_shapes_and_modes(oracle, kw):
    # 140 x 2400 streams its legs through the persistent CTA-pair kernel (d > 256): an odd number of row blocks
    # (one CTA of the last pair has no rows), more column tiles than units and, with so few lanes, row blocks whose
    # column tiles are shared out among many clusters.  300 x 520 stores its products and runs on chip.
    # Whatever the split, the bits must not depend on it: ACTIVE (shrinking batch) and MASKED (fixed batch) must agree exactly.
    w = wl.make("feature", **kw)
    W = w.shape[0]
    ra = run_gpu(w, mode="active", compute="tensor")
    rm = run_gpu(w, mode="masked", compute="tensor")
    np.testing.assert_array_equal(ra["depth"], rm["depth"])
    np.testing.assert_array_equal(ra["f"], rm["f"]); np.testing.assert_array_equal(ra["g"], rm["g"])
    check_against_oracle(oracle, w, ra, range(W), pot_tol=POT_TOL_F32, exact_depth=False, floor=MARGIN_AUTO,
                         label=f"tensor cores (CTA pairs), {kw}")
    check_accounting(oracle, ra, W, "active")
    rs = run_gpu(w, mode="static", compute="tensor")
    np.testing.assert_array_equal(ra["depth"], rs["depth"])
    check_accounting(oracle, rs, W, "static")
    rx = run_gpu(w, mode="masked_exit", compute="tensor")           # frozen lanes skipped, same bits
    np.testing.assert_array_equal(rx["f"], rm["f"]); np.testing.assert_array_equal(rx["g"], rm["g"])
    assert rx["stats"]["slots"] == ra["stats"]["slots"]


def test_tensor_core_pair_kernel_many_small_lanes(oracle):
    # many lanes with stored products, on chip: retirements move the products, and a few lanes are flagged at a time
    # (the pair kernel on these shapes: test_tensor_core_legs_that_stream)
    w = wl.make("feature", W=150, n=130, m=140, d=320)
    r = run_gpu(w, mode="active", compute="tensor")
    lanes = [0, 1, 73, 74, 75, 148, 149] + list(range(9, 150, 29))
    check_against_oracle(oracle, w, r, lanes, pot_tol=POT_TOL_F32, exact_depth=False, floor=MARGIN_AUTO,
                         label="tensor cores (CTA pairs), 150 small lanes")
    check_accounting(oracle, r, 150, "active")
    rm = run_gpu(w, mode="masked", compute="tensor")
    np.testing.assert_array_equal(rm["depth"], r["depth"]); np.testing.assert_array_equal(rm["f"], r["f"])


# Deep lanes whose legs are streamed by the tensor-core kernels: lanes too large for their products to be stored, and small ones in
# a workspace that has no room for those.  d <= 256: one CTA per row block; beyond: persistent CTA pairs, with an odd number of row
# blocks (300, 40: a CTA of the last pair without rows), a ring shorter than six stages (d = 320), more column tiles than units
# (2400 columns), few lanes (a row block's column tiles shared out among clusters) and many (every cluster walks several segments
# of different lanes; retirements move the tiled operand copies; the column check visits a few flagged lanes).
@pytest.mark.parametrize("roomy,kw", [
    (True, dict(W=2, n=1100, m=1030, d=64)), (True, dict(W=2, n=70, m=1101, d=128)), (True, dict(W=2, n=1029, m=600, d=256)),
    (True, dict(W=2, n=2049, m=90, d=192)), (True, dict(W=2, n=1300, m=1027, d=320)), (True, dict(W=3, n=40, m=2400, d=512)),
    (False, dict(W=3, n=200, m=333, d=64)), (False, dict(W=6, n=256, m=256, d=128)), (False, dict(W=2, n=129, m=640, d=256)),
    (False, dict(W=5, n=300, m=520, d=320)), (False, dict(W=3, n=1, m=129, d=64)), (False, dict(W=3, n=129, m=1, d=512)),
    (False, dict(W=150, n=130, m=140, d=320)), (False, dict(W=150, n=130, m=140, d=128))])
def test_tensor_core_legs_that_stream(oracle, monkeypatch, roomy, kw):
    import torch
    from paper_2607_24741_b200 import binding as B
    if not roomy:
        whole = B.sinkhorn_batch_workspace_bytes
        monkeypatch.setattr(B, "sinkhorn_batch_workspace_bytes", lambda cfg: whole(cfg) - 4 * cfg.W * cfg.n * cfg.m)
    w = wl.make("feature", **kw, max_iter=150)
    W = w.shape[0]
    if W > 2:
        w.eps = (w.eps * np.linspace(1.0, 3.0, W)).astype(np.float32)      # lanes leave at different depths
    t = lambda v: torch.from_numpy(v).to("cuda:0")
    sb = B.SinkhornBatch(t(w.x).bfloat16(), t(w.y).bfloat16(), t(w.a), t(w.b), t(w.eps), w.tol, compute="tensor", max_iter=w.max_iter)
    assert _launches_per_step(sb) > 3                                       # legs are streamed
    sb.close()
    ra = run_gpu(w, compute="tensor")
    rm = run_gpu(w, mode="masked", compute="tensor")
    np.testing.assert_array_equal(ra["depth"], rm["depth"])
    np.testing.assert_array_equal(ra["f"], rm["f"]); np.testing.assert_array_equal(ra["g"], rm["g"])
    lanes = range(W) if W < 10 else [0, 1, 73, 74, 75, 148, 149] + list(range(9, 150, 29))
    check_against_oracle(oracle, w, ra, lanes, pot_tol=POT_TOL_F32, exact_depth=False, floor=MARGIN_AUTO,
                         label=f"tensor cores, streamed, {kw}")
    check_accounting(oracle, ra, W, "active")
    rs = run_gpu(w, mode="static", compute="tensor")
    np.testing.assert_array_equal(ra["depth"], rs["depth"])
    check_accounting(oracle, rs, W, "static")
    rx = run_gpu(w, mode="masked_exit", compute="tensor")                   # frozen lanes skipped, same bits
    np.testing.assert_array_equal(rx["f"], rm["f"]); np.testing.assert_array_equal(rx["g"], rm["g"])
    assert rx["stats"]["slots"] == ra["stats"]["slots"]


def test_tensor_core_request_on_ineligible_input_is_refused():
    import torch
    from paper_2607_24741_b200 import binding as B
    w = wl.make("tiny")
    t = lambda v: torch.from_numpy(v).to("cuda:0")
    with pytest.raises(B.SkbError) as e:
        B.SinkhornBatch(t(w.x), t(w.y), t(w.a), t(w.b), t(w.eps), w.tol, compute="tensor")
    assert e.value.code == 2


@pytest.mark.parametrize("tol", [1e-2, 3e-4, 1e-4])
def test_other_tolerances_of_the_sweep_grid(oracle, tol):
    # the disagreement sweep runs the same lanes at five tolerances: depths, slots and potentials at each
    w = wl.make("sweep", W=24, n=100, m=77, max_iter=50000)
    r = run_gpu(w, mode="active", tol=tol)
    check_against_oracle(oracle, w, r, range(24), pot_tol=POT_TOL_F32, exact_depth=False, tol=tol, floor=MARGIN_AUTO,
                         label=f"sweep grid, tol {tol}")
    check_accounting(oracle, r, 24, "active")
    rs = run_gpu(w, mode="static", tol=tol)
    np.testing.assert_array_equal(rs["depth"], r["depth"])
    lmax = int(r["depth"].max())
    assert rs["stats"]["slots"] == 24 * lmax and r["stats"]["slots"] == int(r["depth"].sum())


def test_bounded_wait_gives_up_instead_of_hanging():
    # failure detection without a fault: a barrier nothing completes, a 5 ms budget
    import torch
    from paper_2607_24741_b200 import binding as B
    out = torch.zeros(3, dtype=torch.int32, device="cuda:0")
    rc = B.lib.sinkhorn_batch_selftest_bounded_wait(out.data_ptr(), 5.0, None)
    assert rc == 0
    torch.cuda.synchronize()
    gave_up, abort_flag, kclk = out.cpu().tolist()
    assert gave_up == 1 and abort_flag == 1
    assert 5e3 <= kclk <= 5e5           # ~10 M clocks budget: it neither returned at once nor spun for long
    # the context is still usable
    assert int(torch.arange(10, device="cuda:0").sum().item()) == 45


def test_guard_strips_report_an_overwritten_array_end():
    # the workspace check itself: intact after a solve, and a write just past the end of the last
    # array (made here, from the host side of the test) is reported with that strip's index
    import torch
    from paper_2607_24741_b200 import binding as B
    w = wl.make("tiny")
    dev = torch.device("cuda:0")
    t = lambda v: torch.from_numpy(v).to(dev)
    for compute in ("f64", "f32"):                  # explicit arithmetic: the layout ends where the workspace ends
        sb = B.SinkhornBatch(t(w.x), t(w.y), t(w.a), t(w.b), t(w.eps), w.tol, compute=compute, max_iter=w.max_iter)
        try:
            assert sb.check_guards() == -1           # right after create
            sb.drain()
            assert sb.check_guards() == -1
            assert sb.check_guards() == -1           # the check leaves the strips as they are
            last = sb.workspace.numel() - 1
            sb.workspace[last] ^= 0x40               # one bit of the last strip's last word
            bad = sb.check_guards()
            assert bad >= 40, bad                    # the last of several dozen strips
            sb.workspace[last] ^= 0x40
            assert sb.check_guards() == -1
            sb.workspace[last - 255] ^= 0x01         # first byte of the same strip: same index
            assert sb.check_guards() == bad
        finally:
            sb.close()


def test_very_wide_batch_and_rectangular_lanes(oracle):
    # more lanes than the planner has threads: its scans run in several chunks, holes and fillers
    # pair up across chunks
    w = wl.make("sweep", W=2500, n=8, m=9, max_iter=600)
    r = run_gpu(w, mode="active", compute="f64")
    lanes = [0, 1, 1023, 1024, 1025, 2047, 2048, 2499] + list(range(300, 2500, 211))
    assert check_against_oracle(oracle, w, r, lanes, pot_tol=POT_TOL_F64, exact_depth=True, max_iter=600) == []
    check_accounting(oracle, r, 2500, "active")
    rm = run_gpu(w, mode="masked", compute="f64")
    np.testing.assert_array_equal(rm["depth"], r["depth"]); np.testing.assert_array_equal(rm["f"], r["f"])
    # few sources, many targets (and the reverse): row blocks and column tiles of very different counts
    for n, m in ((5, 700), (700, 5)):
        w = wl.make("sensor", W=3, n=n, m=m)
        for compute in ("f64", "auto"):
            r = run_gpu(w, compute=compute)
            misses = check_against_oracle(oracle, w, r, range(3), pot_tol=POT_TOL_F64 if compute == "f64" else POT_TOL_F32,
                                          exact_depth=compute == "f64")
            assert misses == []


def test_widest_batch_the_interface_takes(oracle):
    # W = 65535 lanes (the interface's limit: one grid row per lane) of four points against five, in the
    # default arithmetic: the planner's scans run over 64 chunks, retirements and moves happen in every
    # cycle, and the widths shrink from 65535 to 1.  Depths of a sample of lanes against the oracle,
    # accounting identities (Eq. 6-8) over all of them.
    W = 65535
    w = wl.make("sweep", W=W, n=4, m=5, max_iter=20000)
    r = run_gpu(w, mode="active", widths_cap=30000)
    depth = r["depth"].astype(np.int64)
    assert np.all(r["status"] == 1) and r["left"] == 0
    assert r["stats"]["slots"] == int(depth.sum()) and r["cycles"] == int(depth.max())
    np.testing.assert_array_equal(np.array(r["stats"]["widths"]), oracle.survivor_widths(depth))
    lanes = [0, 1, 1023, 1024, 32767, 32768, 65534] + list(range(500, W, 4099))
    check_against_oracle(oracle, w, r, lanes, pot_tol=POT_TOL_F32, exact_depth=False, floor=MARGIN_AUTO, max_iter=20000,
                         label="widest batch, W = 65535")
    # the one-launch-per-leg path at this width: the column check's grid has no rows left for the guard
    # band's pool, which then runs as a launch of its own - same bits as ACTIVE
    rm = run_gpu(w, mode="masked", max_iter=20000, widths_cap=30000)
    np.testing.assert_array_equal(rm["depth"], r["depth"]); np.testing.assert_array_equal(rm["f"], r["f"])
    with pytest.raises(Exception):
        run_gpu(wl.make("sweep", W=W + 1, n=4, m=5, max_iter=10))       # one lane more is refused, not mis-launched


def test_mixed_arithmetic_with_a_useless_reference_estimate(oracle):
    # Clouds ten units apart at a small eps: starting from zero potentials, the first legs move
    # every potential by thousands of log2 units, so a reference point estimated from the old
    # potential is off by far more than the fp32 exponent range.  The kernel must notice and
    # repeat such a pass from scratch; otherwise every term flushes to zero and the lanes blow up.
    rng = np.random.default_rng(7)
    W, n, m, d = 6, 70, 90, 3
    x = rng.random((W, n, d), dtype=np.float32)
    y = rng.random((W, m, d), dtype=np.float32) + np.float32(10.0)
    a = rng.random((W, n), dtype=np.float32) + 0.5; a /= a.sum(1, keepdims=True)
    b = rng.random((W, m), dtype=np.float32) + 0.5; b /= b.sum(1, keepdims=True)
    eps = np.linspace(0.03, 0.2, W).astype(np.float32)
    w = wl.Workload("far_apart", x, y, a.astype(np.float32), b.astype(np.float32), eps, 1e-5, 5000)
    for mode in ("active", "static"):
        r = run_gpu(w, mode=mode, compute="mixed")
        assert (r["status"] == oracle.DONE).all()
        check_against_oracle(oracle, w, r, range(W), pot_tol=POT_TOL_F32, exact_depth=False, floor=MARGIN_AUTO,
                             label=f"clouds far apart, {mode}")


# ---- warm proposals and the audit of the proposal itself -------------------------------------------
@pytest.mark.parametrize("compute", ["f64", "auto"])
def test_warm_proposal_continues_a_cold_solve(oracle, compute):
    # Section "Initialization and repeated couplings".  A proposal that is the cold iteration's state after
    # j cycles must finish l_t - j cycles later at the same potentials (both sides get the same proposal).
    w = wl.make("sensor", W=6, n=150, m=170)
    j = 2
    part = oracle.solve_batch(w.x, w.y, w.a, w.b, w.eps, w.tol, fixed_cycles=j)
    warm = (part.f, part.g)
    r = run_gpu(w, compute=compute, warm=warm)
    tolp = POT_TOL_F64 if compute == "f64" else POT_TOL_F32
    check_against_oracle(oracle, w, r, range(6), pot_tol=tolp, exact_depth=compute == "f64", warm=warm,
                         floor=None if compute == "f64" else MARGIN_AUTO, label=f"warm proposal, {compute}")
    cold = run_gpu(w, compute=compute)
    np.testing.assert_array_equal(r["depth"] + j, cold["depth"])
    check_accounting(oracle, r, 6, "active")


@pytest.mark.parametrize("compute", ["f64", "mixed", "f32"])
@pytest.mark.parametrize("mode", ["active", "masked"])
def test_audit_of_the_proposal_measures_both_marginals(oracle, compute, mode):
    # With audit_initial the proposal itself gets the screen and the two-sided check.  Here the proposal
    # is a converged state whose g has been perturbed, so NEITHER marginal is current: the column residual
    # is far from rounding level and the column-check leg has to measure it.  Thresholds are chosen so
    # that some lanes pass at depth 0 (their output is the proposal, with the measured residuals) and the
    # others go on.
    w = wl.make("sensor", W=8, n=130, m=150)
    conv = oracle.solve_batch(w.x, w.y, w.a, w.b, w.eps, 1e-9, max_iter=2000)
    rng = np.random.default_rng(5)
    amp = np.linspace(0.002, 0.05, 8)[:, None] * w.eps[:, None].astype(np.float64)
    warm = (conv.f.copy(), conv.g + amp * rng.standard_normal(conv.g.shape))
    tol = 2e-2
    r = run_gpu(w, mode=mode, compute=compute, warm=warm, audit_initial=True, tol=tol)
    ref = {t: oracle.solve_lane(w.x[t], w.y[t], w.a[t], w.b[t], float(w.eps[t]), tol, f0=warm[0][t], g0=warm[1][t],
                                audit_initial=True) for t in range(8)}
    np.testing.assert_array_equal(r["depth"], [ref[t].depth for t in range(8)])
    zero = [t for t in range(8) if ref[t].depth == 0]
    assert 2 <= len(zero) <= 6                                   # the case really has both kinds of lane
    rel = {"f64": 1e-9, "mixed": 1e-5, "f32": 2e-4}[compute]
    for t in zero:
        # the proposal comes back as it went in (up to the rounding of scaling by 1/eps and back)
        np.testing.assert_allclose(r["f"][t], warm[0][t], rtol=1e-14, atol=0)
        np.testing.assert_allclose(r["g"][t], warm[1][t], rtol=1e-14, atol=0)
        assert ref[t].r_col > 1e-3 and ref[t].r_row > 1e-4       # both far above rounding level
        assert abs(r["r_col"][t] - ref[t].r_col) <= rel * ref[t].r_col + 1e-7
        assert abs(r["r_row"][t] - ref[t].r_row) <= rel * ref[t].r_row + 1e-7
    e = pot_err(r["f"], r["g"], np.stack([ref[t].f for t in range(8)]), np.stack([ref[t].g for t in range(8)]),
                w.eps.astype(np.float64))
    assert e.max() <= (POT_TOL_F64 if compute == "f64" else POT_TOL_F32)
    assert r["stats"]["slots"] == (int(r["depth"].sum()) if mode == "active" else 8 * int(r["depth"].max()))


def test_warm_start_is_refused_after_the_first_cycle():
    import torch
    from paper_2607_24741_b200 import binding as B
    w = wl.make("tiny")
    t = lambda v: torch.from_numpy(v).to("cuda:0")
    sb = B.SinkhornBatch(t(w.x), t(w.y), t(w.a), t(w.b), t(w.eps), w.tol)
    sb.step(1)
    z = torch.zeros(8, 64, dtype=torch.float64, device="cuda:0")
    with pytest.raises(B.SkbError) as e:
        sb.warm_start(z, z)
    assert e.value.code == 5
    sb.close()
    sb = B.SinkhornBatch(t(w.x), t(w.y), t(w.a), t(w.b), t(w.eps), w.tol)
    bad = z.clone(); bad[3, 7] = float("nan")
    sb.warm_start(bad, z)
    with pytest.raises(B.SkbError) as e:
        sb.drain()
    assert e.value.code == 3
    sb.close()


# ---- measurement aids must not disturb the solve ----------------------------------------------------
def _solve_plain(w, compute, mode="active"):
    r = run_gpu(w, mode=mode, compute=compute)
    return r


@pytest.mark.parametrize("case,compute", [("tiny", "auto"), ("sensor_ragged", "f32"), ("feature_small", "auto")])
def test_profiling_an_update_leg_leaves_the_solve_bit_identical(case, compute):
    import torch
    from paper_2607_24741_b200 import binding as B
    w = _make(case)
    plain = run_gpu(w, compute=compute)
    dev = torch.device("cuda:0")
    t = lambda v: torch.from_numpy(v).to(dev)
    x, y = t(w.x), t(w.y)
    if w.xy_dtype == "bf16":
        x, y = x.bfloat16(), y.bfloat16()
    sb = B.SinkhornBatch(x, y, t(w.a), t(w.b), t(w.eps), w.tol, compute=compute, max_iter=w.max_iter)
    sb.step(3)
    assert sb.profile_update(leg=0, reps=5) > 0.0
    assert sb.profile_update(leg=1, reps=2) > 0.0
    sb.drain()
    f, g = sb.potentials(f64=True); depth, status = sb.depths(); rr, rc = sb.residuals(); st = sb.stats()
    np.testing.assert_array_equal(depth.cpu().numpy(), plain["depth"])
    np.testing.assert_array_equal(f.cpu().numpy(), plain["f"]); np.testing.assert_array_equal(g.cpu().numpy(), plain["g"])
    np.testing.assert_array_equal(rr.cpu().numpy(), plain["r_row"])
    assert st["slots"] == plain["stats"]["slots"]
    with pytest.raises(B.SkbError) as e:                      # nothing is running any more
        sb.profile_update(leg=0, reps=1)
    assert e.value.code == 5
    sb.close()


@pytest.mark.parametrize("case,mode", [("sweep_small", "active"), ("sensor_ragged", "static"), ("registration_small", "active")])
def test_phase_timing_adds_up_and_changes_no_bit(case, mode):
    # Eq. 11: update legs (c_k), column check (H_check), planning and emission/compaction (H_compact)
    import torch
    from paper_2607_24741_b200 import binding as B
    w = _make(case)
    plain = run_gpu(w, mode=mode)
    dev = torch.device("cuda:0")
    t = lambda v: torch.from_numpy(v).to(dev)
    sb = B.SinkhornBatch(t(w.x), t(w.y), t(w.a), t(w.b), t(w.eps), w.tol, mode=mode, max_iter=w.max_iter)
    sb.set_profiling(True)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(); sb.drain(); e1.record(); torch.cuda.synchronize()
    wall = e0.elapsed_time(e1)
    st = sb.stats(widths_cap=100000)
    trace = sb.cycle_trace()
    f, g = sb.potentials(f64=True); depth, _ = sb.depths()
    sb.close()
    np.testing.assert_array_equal(depth.cpu().numpy(), plain["depth"])
    np.testing.assert_array_equal(f.cpu().numpy(), plain["f"]); np.testing.assert_array_equal(g.cpu().numpy(), plain["g"])
    ph = st["phase_ms"]
    assert ph["create"] > 0 and ph["f_leg"] > 0 and ph["g_leg"] > 0 and ph["plan"] > 0
    cyc = sum(ph[k] for k in ("f_leg", "column_check", "plan", "emit_move", "g_leg"))
    assert 0.5 * wall <= cyc <= wall                     # the rest is the gaps between the harvested chunks
    assert len(trace) >= st["cycles"] and abs(sum(trace) - ph["f_leg"] - ph["g_leg"]) <= 1e-3 * cyc + 1e-3
    assert plain["stats"]["phase_ms"]["f_leg"] == 0.0 and plain["stats"]["phase_ms"]["create"] > 0


def test_step_alone_follows_the_width_and_reports_device_errors():
    import time
    import torch
    from paper_2607_24741_b200 import binding as B
    w = wl.make("tiny")
    t = lambda v: torch.from_numpy(v).to("cuda:0")
    a = w.a.copy(); a[2, 5] = -1.0
    sb = B.SinkhornBatch(t(w.x), t(w.y), t(a), t(w.b), t(w.eps), w.tol)
    code = None
    for _ in range(200):                                  # no drain, no synchronising call
        try:
            sb.step(1)
        except B.SkbError as e:
            code = e.code
            break
        time.sleep(0.001)
    assert code == 3
    sb.close()
    # a good batch stepped to the end: the launches stop growing once the host has seen it finish
    ref = run_gpu(w)
    sb = B.SinkhornBatch(t(w.x), t(w.y), t(w.a), t(w.b), t(w.eps), w.tol)
    for _ in range(int(ref["depth"].max()) // 10 + 3):
        sb.step(10); time.sleep(0.002)
    torch.cuda.synchronize(); sb.step(1)
    before = sb.launch_count(); sb.step(50)
    assert sb.launch_count() == before                     # finished: further steps enqueue nothing
    depth, _ = sb.depths(); f, _g = sb.potentials(f64=True)
    np.testing.assert_array_equal(depth.cpu().numpy(), ref["depth"]); np.testing.assert_array_equal(f.cpu().numpy(), ref["f"])
    sb.close()


def test_two_batches_interleaved_on_one_stream(oracle):
    # Two handles sharing a stream, stepped alternately; one finishes long before the other.  An f-leg then
    # follows the OTHER batch's (possibly empty) kernels: every kernel of a cycle must still see complete
    # predecessors.
    import torch
    from paper_2607_24741_b200 import binding as B
    wa = wl.make("tiny"); wb = wl.make("sensor", W=12, n=300, m=260)
    t = lambda v: torch.from_numpy(v).to("cuda:0")
    ra, rb = run_gpu(wa), run_gpu(wb)
    sa = B.SinkhornBatch(t(wa.x), t(wa.y), t(wa.a), t(wa.b), t(wa.eps), wa.tol)
    sb = B.SinkhornBatch(t(wb.x), t(wb.y), t(wb.a), t(wb.b), t(wb.eps), wb.tol)
    for _ in range(int(ra["depth"].max()) + 2):
        sa.step(1); sb.step(1)
    torch.cuda.synchronize()
    for s, r in ((sa, ra), (sb, rb)):
        assert s.active() == 0
        f, g = s.potentials(f64=True); depth, _ = s.depths()
        np.testing.assert_array_equal(depth.cpu().numpy(), r["depth"])
        np.testing.assert_array_equal(f.cpu().numpy(), r["f"]); np.testing.assert_array_equal(g.cpu().numpy(), r["g"])
        s.close()


# ---- audit arms ---------------------------------------------------------------------------------------
@pytest.mark.parametrize("case", ["tiny", "sensor_ragged", "sweep_small"])
@pytest.mark.parametrize("every", [1, 4])
def test_full_check_arm_against_oracle(oracle, case, every):
    # no screen: every audited lane gets the two-sided check (tol_screen far above any residual); the oracle
    # runs with the same thresholds and the same audit grid
    w = _make(case)
    W = w.shape[0]
    r = run_gpu(w, mode="active", tol_screen=1e30, audit_every=every)
    check_against_oracle(oracle, w, r, range(W), pot_tol=POT_TOL_F32, exact_depth=False, tol_screen=1e30,
                         audit_every=every, floor=MARGIN_AUTO, label=f"full-check arm, every {every}, {case}")
    assert np.all(r["depth"] % every == 0)
    # every audit of every lane ran a column check: W*n*m per audit beyond the legs
    n, m = w.shape[1], w.shape[2]
    audits = int((r["depth"] // every).sum()) if every > 1 else int(r["depth"].sum())
    assert r["stats"]["pair_terms"] >= 2 * r["stats"]["slots"] * n * m + audits * n * m


def test_last_audit_reports_the_screen_of_the_previous_state(oracle):
    import torch
    from paper_2607_24741_b200 import binding as B
    w = wl.make("sensor", W=6, n=90, m=70)
    t = lambda v: torch.from_numpy(v).to("cuda:0")
    sb = B.SinkhornBatch(t(w.x), t(w.y), t(w.a), t(w.b), t(w.eps), 1e-7, mode="masked", compute="f64")
    sb.step(3)
    f, g = sb.potentials(f64=True)                       # state after 3 cycles
    sb.step(1)
    rr, rc, fl = sb.last_audit()                         # ... whose screen came out of the f-leg of cycle 4
    fh, gh, rr = f.cpu().numpy(), g.cpu().numpy(), rr.cpu().numpy()
    for k in range(6):
        want, _ = oracle.residuals(w.x[k], w.y[k], w.a[k], w.b[k], float(w.eps[k]), fh[k], gh[k])
        assert abs(rr[k] - want) <= 1e-6 * want
    assert (fl.cpu().numpy() == 0).all() and np.isnan(rc.cpu().numpy()).all()
    sb.close()
    w = wl.make("tiny")                                  # an ACTIVE batch of small lanes runs several cycles per launch
    act = B.SinkhornBatch(t(w.x), t(w.y), t(w.a), t(w.b), t(w.eps), w.tol, mode="active")
    act.step(2)
    with pytest.raises(B.SkbError) as e:
        act.last_audit()
    assert e.value.code == 5
    act.close()


# ---- large clouds ---------------------------------------------------------------------------------------
def test_sixteen_thousand_points_against_oracle_cycles(oracle):
    # n = m = 16384 (the size of the paper's largest Flash campaigns): the oracle's dense cost matrix is
    # 2 GB and one cycle takes it tens of seconds, so the comparison is on the state after two cycles
    w = wl.make("registration", W=1, n=16384)
    import torch
    from paper_2607_24741_b200 import binding as B
    t = lambda v: torch.from_numpy(v).to("cuda:0")
    sb = B.SinkhornBatch(t(w.x), t(w.y), t(w.a), t(w.b), t(w.eps), w.tol, mode="static")
    sb.step(2)
    f, g = sb.potentials(f64=True)
    sb.close()
    ref = oracle.solve_lane(w.x[0], w.y[0], w.a[0], w.b[0], float(w.eps[0]), w.tol, fixed_cycles=2)
    e = pot_err(f.cpu().numpy(), g.cpu().numpy(), ref.f[None], ref.g[None], w.eps.astype(np.float64))
    assert e.max() <= POT_TOL_F32


def test_limits_of_dimension_size_and_iteration_count(oracle):
    import torch
    from paper_2607_24741_b200 import binding as B
    t = lambda v: torch.from_numpy(v).to("cuda:0")
    # every padded dimension of the SIMT kernels (1 -> 2, 5 -> 8, 17 -> 32, 32), the first and the last
    # dimension of the large-d kernels (33, 1024), in the default arithmetic, against the oracle
    for d in (1, 5, 17, 32, 33, 100, 1024):
        w = wl.make("sensor", W=3, n=40, m=50, d=d)
        r = run_gpu(w)
        assert check_against_oracle(oracle, w, r, range(3), pot_tol=POT_TOL_F32, exact_depth=False, floor=MARGIN_AUTO,
                                    label=f"dimension limits, d = {d}") == [], d
    w = wl.make("sensor", W=3, n=40, m=50, d=1024)
    bad = B.make_config(3, 40, 50, 1025)
    assert B.sinkhorn_batch_workspace_bytes(bad) == 0                      # one dimension more is refused
    # bf16 inputs just past the tensor-core range (d = 576 > 512) fall back to the large-d SIMT kernels
    w = wl.make("feature", W=2, n=96, m=130, d=576)
    r = run_gpu(w)
    assert r["arith"] != "tensor"
    assert check_against_oracle(oracle, w, r, range(2), pot_tol=POT_TOL_F32, exact_depth=False, floor=MARGIN_AUTO,
                                label="bf16, d = 576") == []
    # bf16 storage on the small-d kernels, with every near-threshold audit escalated (the float64
    # re-evaluation reads the raw bf16 copies: vector loads where d is a multiple of 8, scalar otherwise)
    for d in (2, 12, 16):
        w = wl.make("feature", W=3, n=70, m=90, d=d)
        r = run_gpu(w, guard_band=0.5)
        assert check_against_oracle(oracle, w, r, range(3), pot_tol=POT_TOL_F32, exact_depth=False, floor=1e-6,
                                    label=f"bf16 inputs, d = {d}, guard band 0.5") == [], d
    # the largest cloud the interface takes (262143 points, fixed-point residual sums) against three points
    n_max = 262143
    w = wl.make("sweep", W=1, n=n_max, m=3, d=2, max_iter=10)
    sb = B.SinkhornBatch(t(w.x), t(w.y), t(w.a), t(w.b), t(w.eps), w.tol, mode="static", max_iter=10)
    sb.step(2)
    f, g = sb.potentials(f64=True)
    assert sb.check_guards() == -1
    sb.close()
    ref = oracle.solve_lane(w.x[0], w.y[0], w.a[0], w.b[0], float(w.eps[0]), w.tol, fixed_cycles=2)
    assert pot_err(f.cpu().numpy(), g.cpu().numpy(), ref.f[None], ref.g[None], w.eps.astype(np.float64)).max() <= POT_TOL_F32
    assert B.sinkhorn_batch_workspace_bytes(B.make_config(1, n_max + 1, 3, 2)) > 0          # sized ...
    with pytest.raises(B.SkbError):                                                          # ... but refused at create
        w1 = wl.make("sweep", W=1, n=n_max + 1, m=3, d=2, max_iter=10)
        B.SinkhornBatch(t(w1.x), t(w1.y), t(w1.a), t(w1.b), t(w1.eps), w1.tol)
    # one cycle allowed: every lane either passes its first audit or stops at the limit with depth 1
    w = wl.make("tiny", max_iter=1)
    r = run_gpu(w)
    ref = oracle.solve_batch(w.x, w.y, w.a, w.b, w.eps, w.tol, max_iter=1)
    np.testing.assert_array_equal(r["depth"], ref.depth); np.testing.assert_array_equal(r["status"], ref.status)
    assert (r["depth"] == 1).all() and r["stats"]["slots"] == 8
    # a tolerance nothing can miss (the L1 residual of unit-mass marginals is at most 2): depth 1 everywhere
    w = wl.make("sensor", W=5, n=30, m=20, tol=2.5)
    r = run_gpu(w)
    assert (r["depth"] == 1).all() and (r["status"] == 1).all()


def test_sixty_five_thousand_points_sampled_marginals():
    # n = m = 65536: far beyond what the oracle can hold (a 34 GB cost matrix), so the emitted state is
    # checked on sampled rows and columns, each computed from its definition in float64: after the last
    # g-leg every column marginal equals b_j (Eq. 4), and the sampled rows' deviations extrapolate to a
    # row residual below the tolerance the lane stopped at (Eq. 5).
    w = wl.make("registration", W=1, n=65536)
    r = run_gpu(w)
    assert r["status"][0] == 1 and r["r_row"][0] <= w.tol and r["depth"][0] > 50
    x, y = w.x[0].astype(np.float64), w.y[0].astype(np.float64)
    a, b, eps = w.a[0].astype(np.float64), w.b[0].astype(np.float64), float(w.eps[0])
    f, g = r["f"][0], r["g"][0]
    rng = np.random.default_rng(11)
    cols = rng.choice(65536, 48, replace=False)
    for j in cols:
        c = ((x - y[j]) ** 2).sum(1)
        assert abs(np.exp((f + g[j] - c) / eps).sum() - b[j]) <= 2e-5 * b[j]
    rows = rng.choice(65536, 256, replace=False)
    dev = 0.0
    for i in rows:
        c = ((y - x[i]) ** 2).sum(1)
        dev += abs(np.exp((f[i] + g - c) / eps).sum() - a[i])
    assert dev * (65536 / 256) <= 1.5 * w.tol          # a 256-row sample of an L1 norm: generous sampling slack


# ---- guard band: float64 escalation of near-threshold decisions -------------------------------------------
@pytest.mark.parametrize("case", ["tiny", "sweep_small", "sensor_ragged", "registration_small", "feature_small",
                                  "feature_tensor"])
def test_guard_band_decisions_come_from_the_float64_reevaluation(oracle, case):
    # Section 5's stress test: raw fp32 decisions near the threshold flip; an outward guard with float64
    # escalation removes the flips.  With a band of 50 % every audit within a factor 1.5 of the threshold is
    # decided from the float64 re-evaluation of the row residual, so the depths must be the oracle's to
    # within the acceptance bar's own band of 1e-6, in the multi-cycle kernels (ACTIVE) as in the
    # one-launch-per-leg path (MASKED), with identical bits.
    w = _make(case)
    W = w.shape[0]
    ra = run_gpu(w, mode="active", guard_band=0.5)
    rm = run_gpu(w, mode="masked", guard_band=0.5)
    np.testing.assert_array_equal(ra["depth"], rm["depth"])
    np.testing.assert_array_equal(ra["f"], rm["f"]); np.testing.assert_array_equal(ra["g"], rm["g"])
    np.testing.assert_array_equal(ra["r_row"], rm["r_row"])
    check_against_oracle(oracle, w, ra, range(W), pot_tol=POT_TOL_F32, exact_depth=False, floor=1e-6,
                         label=f"guard band 0.5, {case}")
    check_accounting(oracle, ra, W, "active")
    # the reported row residual of a lane decided by escalation IS the float64 value
    tol = w.tol
    for t in range(W):
        rr, _ = oracle.residuals(w.x[t], w.y[t], w.a[t], w.b[t], float(w.eps[t]), ra["f"][t], ra["g"][t])
        if ra["status"][t] == 1 and rr >= 0.51 * tol:           # inside the band when it stopped: escalated
            assert abs(ra["r_row"][t] - rr) <= 2e-7 * rr + 1e-10
    off = run_gpu(w, mode="active", guard_band=-1.0)              # switched off: still within the usual bar
    check_against_oracle(oracle, w, off, range(W), pot_tol=POT_TOL_F32, exact_depth=False, floor=MARGIN_AUTO,
                         label=f"guard band off, {case}")


# ---- finished lanes replaced by new problems ------------------------------------------------------------
@pytest.mark.parametrize("compute", ["f64", "mixed", "f32"])
def test_refill_keeps_the_width_up_and_every_lane_its_own_result(oracle, compute):
    # 40 problems through 12 slots: whenever slots are free, the next problems come in.  Lanes are
    # independent (Eq. 2), so every lane must end exactly as in a one-shot batch of all 40 (same bits:
    # a lane's arithmetic depends neither on its slot nor on when it came in), depths count the lane's own
    # cycles, and the slot identity of Eq. 7 holds over the whole run.
    import torch
    from paper_2607_24741_b200 import binding as B
    w = wl.make("sweep", W=40, n=96, m=80, max_iter=3000)
    S = 12
    ref = run_gpu(w, compute=compute, guard_band=-1.0 if compute == "f32" else 0.0)
    dev = torch.device("cuda:0")
    t = lambda v: torch.from_numpy(v).to(dev)
    x, y, a, b, eps = t(w.x), t(w.y), t(w.a), t(w.b), t(w.eps)
    sb = B.SinkhornBatch(x[:S], y[:S], a[:S], b[:S], eps[:S], w.tol, compute=compute, max_iter=w.max_iter,
                         lane_capacity=40, guard_band=-1.0 if compute == "f32" else 0.0)
    nxt, refills = S, 0
    while nxt < 40:
        sb.step(25)
        free = S - sb.active()
        if free > 0:
            c = min(free, 40 - nxt)
            first = sb.refill(x[nxt:nxt + c], y[nxt:nxt + c], a[nxt:nxt + c], b[nxt:nxt + c], eps[nxt:nxt + c])
            assert first == nxt
            nxt += c; refills += 1
    assert refills >= 3
    sb.drain()
    f, g = sb.potentials(f64=True); depth, status = sb.depths(); rr, rc = sb.residuals()
    st = sb.stats(widths_cap=100000); left = sb.active()
    sb.close()
    depth = depth.cpu().numpy(); assert depth.shape == (40,)
    np.testing.assert_array_equal(depth, ref["depth"]); np.testing.assert_array_equal(status.cpu().numpy(), ref["status"])
    np.testing.assert_array_equal(f.cpu().numpy(), ref["f"]); np.testing.assert_array_equal(g.cpu().numpy(), ref["g"])
    np.testing.assert_array_equal(rr.cpu().numpy(), ref["r_row"])
    assert left == 0 and st["slots"] == int(depth.sum()) == sum(st["widths"]) and max(st["widths"]) <= S
    if compute != "f32":            # (pure fp32 on these small-eps lanes has its recorded limits; the bit-identity above stands)
        lanes = [0, 5, 11, 12, 20, 33, 39]
        check_against_oracle(oracle, w, dict(ref, depth=depth), lanes, pot_tol=POT_TOL_F64 if compute == "f64" else POT_TOL_F32,
                             exact_depth=compute == "f64", floor=None if compute == "f64" else MARGIN_AUTO,
                             label=f"refilled lanes, {compute}")


def _launches_per_step(sb):
    # a step of one cycle (not a batch's first, which may rank its lanes) is three launches or fewer where the kernel matrix is on
    # chip, four or more where legs are streamed
    sb.step(1)
    before = sb.launch_count()
    sb.step(1)
    return sb.launch_count() - before


def test_a_deep_lane_has_the_same_bits_in_a_queue_and_in_one_batch_of_all_lanes():
    # products of deep lanes are stored up to a size, counted over all lanes that a batch can take in: 1025 lanes of
    # 1024 x 1024 are beyond it, in one batch and as a queue through eight slots
    import torch
    from paper_2607_24741_b200 import binding as B
    gen = torch.Generator(device="cuda:0"); gen.manual_seed(3)
    W, n, d, S, given = 1025, 1024, 64, 8, 20
    unit = lambda v: (v / v.norm(dim=2, keepdim=True)).bfloat16()
    x, y = (unit(torch.randn(W, n, d, generator=gen, device="cuda:0")) for _ in range(2))
    a = torch.full((W, n), 1.0 / n, device="cuda:0"); eps = torch.full((W,), 0.05, device="cuda:0")
    kw = dict(max_iter=3, compute="tensor")
    sb = B.SinkhornBatch(x, y, a, a, eps, 1e-7, **kw)
    assert _launches_per_step(sb) > 3
    sb.drain()
    f, g = (v[:given].cpu().numpy() for v in sb.potentials(f64=True))
    sb.close()
    sb = B.SinkhornBatch(x[:S], y[:S], a[:S], a[:S], eps[:S], 1e-7, lane_capacity=W, **kw)
    assert _launches_per_step(sb) > 3
    nxt = S
    while nxt < given:
        sb.drain()
        c = min(S, given - nxt)
        assert sb.refill(x[nxt:nxt + c], y[nxt:nxt + c], a[:c], a[:c], eps[:c]) == nxt
        nxt += c
    sb.drain()
    fq, gq = (v[:given].cpu().numpy() for v in sb.potentials(f64=True))
    assert sb.check_guards() == -1
    sb.close()
    np.testing.assert_array_equal(fq, f); np.testing.assert_array_equal(gq, g)


def test_deep_lanes_in_a_workspace_without_room_for_their_products(oracle):
    # a workspace smaller by the products is taken, on device and host buffers (the products are formed in every leg then); one
    # that lacks more is refused
    import torch
    from paper_2607_24741_b200 import binding as B
    w = wl.make("feature", W=3, n=200, m=260, d=64)
    t = lambda v: torch.from_numpy(v).to("cuda:0")
    x, y, a, b, eps = t(w.x).bfloat16(), t(w.y).bfloat16(), t(w.a), t(w.b), t(w.eps)
    dots, more = 4 * 3 * 200 * 260, 8 * 3 * (3 * 200 + 2 * 260)
    stream = torch.cuda.current_stream().cuda_stream
    cfg = B.make_config(3, 200, 260, 64, bf16=True, compute="tensor", stream=stream)
    need = B.sinkhorn_batch_workspace_bytes(cfg)
    ws = torch.empty(need, dtype=torch.uint8, device="cuda:0")
    cfg.workspace = ws.data_ptr()
    cfg.workspace_bytes = need - dots - more - 8192
    with pytest.raises(B.SkbError):
        B.sinkhorn_batch_create(x, y, a, b, eps, w.tol, cfg)
    full = run_gpu(w, compute="tensor")
    out = {}
    for room in (need, need - dots):
        cfg.workspace_bytes = room
        h = B.sinkhorn_batch_create(x, y, a, b, eps, w.tol, cfg)
        before = ctypes.c_longlong(0); after = ctypes.c_longlong(0)
        B.sinkhorn_batch_step(h, 1)
        B.lib.sinkhorn_batch_launch_count(h, ctypes.byref(before))
        B.sinkhorn_batch_step(h, 1)
        B.lib.sinkhorn_batch_launch_count(h, ctypes.byref(after))
        assert (after.value - before.value <= 3) == (room == need)
        B.sinkhorn_batch_drain(h)
        f = torch.zeros(3, 200, dtype=torch.float64, device="cuda:0"); g = torch.zeros(3, 260, dtype=torch.float64, device="cuda:0")
        assert B.lib.sinkhorn_batch_potentials_f64(h, B._ptr(f), B._ptr(g)) == 0
        depth = torch.zeros(3, dtype=torch.int32, device="cuda:0"); status = torch.zeros_like(depth)
        assert B.lib.sinkhorn_batch_depths(h, B._ptr(depth), B._ptr(status)) == 0
        bad = ctypes.c_int(-2)
        assert B.lib.sinkhorn_batch_check_guards(h, ctypes.byref(bad)) == 0 and bad.value == -1
        B.sinkhorn_batch_destroy(h)
        out[room] = f.cpu().numpy(), g.cpu().numpy(), depth.cpu().numpy()
    np.testing.assert_array_equal(out[need][0], full["f"]); np.testing.assert_array_equal(out[need][2], full["depth"])
    np.testing.assert_array_equal(out[need - dots][2], full["depth"])
    assert pot_err(*out[need - dots][:2], full["f"], full["g"], w.eps).max() <= 5e-6      # both within 3e-6 of the oracle's
    # host buffers
    host = B.sinkhorn_batch_host_workspace_bytes(cfg)
    ws = torch.empty(host, dtype=torch.uint8, device="cuda:0")
    cfg.workspace = ws.data_ptr()
    hx, hy, ha, hb, he = (v.cpu().contiguous() for v in (x, y, a, b, eps))
    ptr = lambda v: ctypes.c_void_p(v.data_ptr())
    for room, want in ((host, out[need]), (host - dots, out[need - dots])):
        cfg.workspace_bytes = room
        f = torch.zeros(3, 200); g = torch.zeros(3, 260)
        rc = B.lib.sinkhorn_batch_solve_host(ptr(hx), ptr(hy), ptr(ha), ptr(hb), ptr(he), ctypes.c_float(w.tol), ctypes.byref(cfg),
                                             ptr(f), ptr(g), None, None, None, None, None, None)
        assert rc == 0
        np.testing.assert_array_equal(f.numpy(), want[0].astype(np.float32)); np.testing.assert_array_equal(g.numpy(), want[1].astype(np.float32))


@pytest.mark.parametrize("n,m,d,kw", [(101, 90, 64, {}), (140, 131, 64, {}), (250, 255, 128, {}), (300, 200, 320, {}), (333, 300, 64, {}), (300, 600, 64, {}),
                                      (140, 131, 64, dict(guard_band=0.3, audit_every=3)), (333, 300, 64, dict(profiling=True))])
def test_deep_lanes_refilled_after_compaction(oracle, n, m, d, kw):
    # lanes with stored products come into slots that others have left or have been moved out of, in one block and in clusters
    # of several: every lane must end as in one batch of all of them, bit for bit
    import torch
    from paper_2607_24741_b200 import binding as B
    W, S = 22, 7
    w = wl.make("feature", W=W, n=n, m=m, d=d, max_iter=300)
    w.eps = np.random.default_rng(5).permutation(np.geomspace(0.03, 0.5, W)).astype(np.float32)
    t = lambda v: torch.from_numpy(v).to("cuda:0")
    x, y, a, b, eps = t(w.x).bfloat16(), t(w.y).bfloat16(), t(w.a), t(w.b), t(w.eps)
    profiling = kw.get("profiling", False)
    kw = {k: v for k, v in kw.items() if k != "profiling"}
    ref = run_gpu(w, **kw)
    assert ref["arith"] == "tensor" and len(set(ref["depth"])) > 5
    sb = B.SinkhornBatch(x[:S], y[:S], a[:S], b[:S], eps[:S], w.tol, max_iter=w.max_iter, lane_capacity=W, **kw)
    sb.set_profiling(profiling)
    nxt, partly = S, 0
    while nxt < W:
        sb.step(5)
        left = sb.active()
        c = min(S - left, W - nxt, 3)
        if c > 0:
            partly += left > 0
            assert sb.refill(x[nxt:nxt + c], y[nxt:nxt + c], a[nxt:nxt + c], b[nxt:nxt + c], eps[nxt:nxt + c]) == nxt
            nxt += c
    assert partly >= 3                                                  # refills next to lanes that were still running
    sb.drain()
    f, g = sb.potentials(f64=True); depth, status = sb.depths(); rr, _ = sb.residuals()
    assert sb.check_guards() == -1
    sb.close()
    if "audit_every" not in kw:                                         # (a lane's audits are on the batch's grid)
        np.testing.assert_array_equal(depth.cpu().numpy(), ref["depth"]); np.testing.assert_array_equal(status.cpu().numpy(), ref["status"])
        np.testing.assert_array_equal(f.cpu().numpy(), ref["f"]); np.testing.assert_array_equal(g.cpu().numpy(), ref["g"])
        np.testing.assert_array_equal(rr.cpu().numpy(), ref["r_row"])
        check_against_oracle(oracle, w, ref, range(0, W, 3), pot_tol=POT_TOL_F32, exact_depth=False, floor=MARGIN_AUTO,
                             label=f"refilled deep lanes, {n} x {m}")
    else:
        late = depth.cpu().numpy() - ref["depth"]
        assert (np.abs(late) < kw["audit_every"]).all() and (status.cpu().numpy() == ref["status"]).all(), late


@pytest.mark.parametrize("options", [dict(guard_band=0.5), dict(audit_every=4, guard_band=0.5), dict(profiling=True),
                                     dict(compute="mixed", audit_every=3, guard_band=0.5)],
                         ids=["guard", "grid4_guard", "profiled", "mixed_grid3_guard"])
def test_refill_combined_with_the_other_options(options):
    # refill together with an audit grid (new lanes come in on the grid), a guard band wide enough that
    # most audits escalate, and phase timing: every lane ends with the bits of a one-shot batch
    import torch
    from paper_2607_24741_b200 import binding as B
    dev = torch.device("cuda:0")
    t = lambda v: torch.from_numpy(v).to(dev)
    profiling = options.get("profiling", False)
    kw = {k: v for k, v in options.items() if k != "profiling"}
    every = kw.get("audit_every", 1)
    for name, shape, S in (("sweep", dict(W=40, n=96, m=80, max_iter=3000), 7), ("tiny", dict(W=24), 5)):
        w = wl.make(name, **shape)
        N = w.shape[0]
        ref = run_gpu(w, **kw)
        x, y, a, b, eps = t(w.x), t(w.y), t(w.a), t(w.b), t(w.eps)
        sb = B.SinkhornBatch(x[:S], y[:S], a[:S], b[:S], eps[:S], w.tol, max_iter=w.max_iter, lane_capacity=N, **kw)
        try:
            if profiling:
                sb.set_profiling(True)
            nxt = S
            while nxt < N:
                sb.step(12 * every)
                free = S - sb.active()
                if free > 0:
                    c = min(free, N - nxt)
                    sb.refill(x[nxt:nxt + c], y[nxt:nxt + c], a[nxt:nxt + c], b[nxt:nxt + c], eps[nxt:nxt + c])
                    nxt += c
            sb.drain()
            f, g = sb.potentials(f64=True); depth, status = sb.depths(); rr, _ = sb.residuals()
            slots = sb.stats(widths_cap=200000)["slots"]
            assert sb.check_guards() == -1
        finally:
            sb.close()
        np.testing.assert_array_equal(depth.cpu().numpy(), ref["depth"])
        np.testing.assert_array_equal(f.cpu().numpy(), ref["f"]); np.testing.assert_array_equal(g.cpu().numpy(), ref["g"])
        np.testing.assert_array_equal(rr.cpu().numpy(), ref["r_row"])
        assert slots == int(ref["depth"].sum())


def test_refill_is_refused_where_it_cannot_work():
    import torch
    from paper_2607_24741_b200 import binding as B
    w = wl.make("tiny")
    t = lambda v: torch.from_numpy(v).to("cuda:0")
    x, y, a, b, eps = t(w.x), t(w.y), t(w.a), t(w.b), t(w.eps)
    with pytest.raises(B.SkbError) as e:                          # only ACTIVE batches compact, so only they have free slots
        B.SinkhornBatch(x, y, a, b, eps, w.tol, mode="masked", lane_capacity=16)
    assert e.value.code == 2
    sb = B.SinkhornBatch(x[:4], y[:4], a[:4], b[:4], eps[:4], w.tol, lane_capacity=6)
    with pytest.raises(B.SkbError) as e:                          # no lane has finished yet
        sb.refill(x[4:6], y[4:6], a[4:6], b[4:6], eps[4:6])
    assert e.value.code == 5
    sb.drain()
    assert sb.refill(x[4:6], y[4:6], a[4:6], b[4:6], eps[4:6]) == 4
    with pytest.raises(B.SkbError) as e:                          # capacity of 6 lanes used up
        sb.refill(x[6:7], y[6:7], a[6:7], b[6:7], eps[6:7])
    assert e.value.code == 2
    sb.drain()
    depth, status = sb.depths()
    assert depth.shape[0] == 6 and (status.cpu().numpy() == 1).all()
    ref = run_gpu(w)
    np.testing.assert_array_equal(depth.cpu().numpy(), ref["depth"][:6])
    sb.close()


# ---- the plan as an output ------------------------------------------------------------------------------
@pytest.mark.parametrize("case", ["sensor_ragged", "registration_small", "sweep_small"])
def test_plan_application_against_the_oracle(oracle, case):
    import torch
    from paper_2607_24741_b200 import binding as B
    w = _make(case)
    W, n, m, d = w.shape
    dev = torch.device("cuda:0")
    t = lambda v: torch.from_numpy(v).to(dev)
    sb = B.SinkhornBatch(t(w.x), t(w.y), t(w.a), t(w.b), t(w.eps), w.tol, max_iter=w.max_iter)
    with pytest.raises(B.SkbError) as e:
        sb.apply_plan(t(w.y))
    assert e.value.code == 5                                   # lanes still running
    sb.drain()
    f, g = sb.potentials(f64=True)
    out_y = sb.apply_plan(t(w.y)).cpu().numpy()                # a_i times the barycentric image of x_i
    ones = sb.apply_plan(torch.ones(W, m, 1, device=dev)).cpu().numpy()
    sb.close()
    fh, gh = f.cpu().numpy(), g.cpu().numpy()
    for k in range(W):
        want = oracle.apply_plan(w.x[k], w.y[k], float(w.eps[k]), fh[k], gh[k], w.y[k])
        scale = np.abs(want).max()
        assert np.abs(out_y[k] - want).max() <= 2e-6 * scale           # same potentials: float32 output rounding
        np.testing.assert_allclose(ones[k, :, 0], want_row(oracle, w, k, fh[k], gh[k]), rtol=2e-6)
        ref = oracle.solve_lane(w.x[k], w.y[k], w.a[k], w.b[k], float(w.eps[k]), w.tol, max_iter=w.max_iter)
        mine = oracle.apply_plan(w.x[k], w.y[k], float(w.eps[k]), ref.f, ref.g, w.y[k])
        assert np.abs(out_y[k] - mine).max() <= 2e-3 * scale           # the oracle's own solve: potentials within 1e-4


def want_row(oracle, w, k, f, g):
    row, _ = oracle.marginals(oracle.cost_matrix(w.x[k], w.y[k]), f, g, float(w.eps[k]))
    return row


# ---- lanes whose kernel matrix stays on chip (mixed arithmetic) --------------------------------------
@pytest.mark.parametrize("n,m", [(16, 64), (17, 63), (64, 2), (65, 64), (128, 33), (129, 64), (64, 65), (65, 128), (129, 100),
                                 (64, 129), (65, 256), (512, 200), (513, 200), (64, 257), (300, 512), (513, 512)])
def test_kernel_matrix_lanes_at_the_edges_of_their_tiles(oracle, n, m):
    # first and last sizes of every tile shape and of the lanes that fit at all; one launch of many cycles
    # (drain), one of one cycle each (step), a logical mask and the one-launch-per-leg path (phase timing)
    # must give the same bits, whatever the lanes' K was formed from
    import torch
    from paper_2607_24741_b200 import binding as B
    w = wl.make("sweep", W=3, n=n, m=m, d=5, max_iter=120)
    r = run_gpu(w, compute="mixed")
    check_against_oracle(oracle, w, r, range(3), pot_tol=POT_TOL_F32, exact_depth=False, floor=MARGIN_AUTO, max_iter=120,
                         label=f"kernel matrix on chip, {n} x {m}")
    check_accounting(oracle, r, 3, "active")
    rm = run_gpu(w, compute="mixed", mode="masked")
    np.testing.assert_array_equal(rm["f"], r["f"]); np.testing.assert_array_equal(rm["r_row"], r["r_row"])
    t = lambda v: torch.from_numpy(v).to("cuda:0")
    for profiling in (False, True):
        sb = B.SinkhornBatch(t(w.x), t(w.y), t(w.a), t(w.b), t(w.eps), w.tol, compute="mixed", max_iter=120)
        sb.set_profiling(profiling)
        for _ in range(121):
            sb.step(1)
        assert sb.active() == 0
        f, g = sb.potentials(f64=True)
        np.testing.assert_array_equal(f.cpu().numpy(), r["f"]); np.testing.assert_array_equal(g.cpu().numpy(), r["g"])
        assert sb.check_guards() == -1
        sb.close()


@pytest.mark.parametrize("n,m", [(40, 128), (129, 100), (128, 129), (257, 256), (130, 257), (600, 512), (64, 513), (193, 600),
                                 (449, 1024), (1024, 520)])
def test_deep_lanes_on_chip_at_the_edges_of_their_tiles(oracle, n, m):
    # one block, clusters of 2 to 16 blocks, clusters with blocks that hold no rows, both ways of exchanging column sums;
    # launches of many cycles, of one cycle, of one leg, and a logical mask must give the same bits
    import torch
    from paper_2607_24741_b200 import binding as B
    w = wl.make("feature", W=3, n=n, m=m, d=64, max_iter=40)
    r = run_gpu(w)
    assert r["arith"] == "tensor"
    check_against_oracle(oracle, w, r, range(3), pot_tol=POT_TOL_F32, exact_depth=False, floor=MARGIN_AUTO, max_iter=40,
                         label=f"deep lanes on chip, {n} x {m}")
    check_accounting(oracle, r, 3, "active")
    rm = run_gpu(w, mode="masked")
    np.testing.assert_array_equal(rm["f"], r["f"]); np.testing.assert_array_equal(rm["r_row"], r["r_row"])
    t = lambda v: torch.from_numpy(v).to("cuda:0")
    for profiling in (False, True):
        sb = B.SinkhornBatch(t(w.x).bfloat16(), t(w.y).bfloat16(), t(w.a), t(w.b), t(w.eps), w.tol, max_iter=40)
        sb.set_profiling(profiling)
        for _ in range(41):
            sb.step(1)
        assert sb.active() == 0
        f, g = sb.potentials(f64=True)
        np.testing.assert_array_equal(f.cpu().numpy(), r["f"]); np.testing.assert_array_equal(g.cpu().numpy(), r["g"])
        assert sb.check_guards() == -1
        sb.close()


def test_last_audit_of_deep_lanes_follows_them_through_compaction():
    # lanes that others' retirement has moved report their own audit, as lanes that stay in place do
    import torch
    from paper_2607_24741_b200 import binding as B
    w = wl.make("feature", W=12, n=96, m=80, d=64)
    t = lambda v: torch.from_numpy(v).to("cuda:0")
    both = [B.SinkhornBatch(t(w.x).bfloat16(), t(w.y).bfloat16(), t(w.a), t(w.b), t(w.eps), w.tol, mode=m) for m in ("active", "masked")]
    seen = set()
    while both[0].active() > 0:
        for sb in both:
            sb.step(7)
        seen.add(both[0].active())
        running = (both[0].depths()[1] == 0).cpu().numpy()
        (ra, ca, fa), (rm, cm, fm) = (tuple(v.cpu().numpy() for v in sb.last_audit()) for sb in both)
        np.testing.assert_array_equal(ra[running], rm[running]); np.testing.assert_array_equal(fa[running], fm[running])
    assert len(seen - {0, 12}) > 0                                # lanes really left one after the other
    for sb in both:
        sb.close()


@pytest.mark.parametrize("light", [1.0, 2.0 ** -25, 2.0 ** -38, 2.0 ** -75])
def test_lanes_that_start_with_their_costs_absorbed(oracle, light):
    # four times the scaled squared radius on both sides of the 120 bits up to which a cold lane starts with zero potentials
    # absorbed, weights on both sides of the 2^-40 from which it does (and of the 2^-80 below which it never absorbs)
    rng = np.random.default_rng(11)
    f32 = np.float32
    W, n, m, d = 6, 70, 130, 5
    x = rng.uniform(-1, 1, (W, n, d)).astype(f32); y = rng.uniform(-1, 1, (W, m, d)).astype(f32)
    a = rng.uniform(0.5, 1.5, (W, n)); b = rng.uniform(0.5, 1.5, (W, m))
    a[1::2, 4] *= light; b[::2, 9:12] *= light
    rad = np.array([max(((x[t] - c) ** 2).sum(1).max(), ((y[t] - c) ** 2).sum(1).max())
                    for t in range(W) for c in [np.concatenate([x[t], y[t]]).mean(0)]])
    eps = (4.0 * 1.4426950408889634 * rad / np.array([20.0, 90.0, 118.0, 122.0, 200.0, 400.0])).astype(f32)
    w = wl.Workload("cold", x, y, (a / a.sum(1, keepdims=True)).astype(f32), (b / b.sum(1, keepdims=True)).astype(f32), eps, 1e-3, 300)
    for mode in ("active", "static"):
        r = run_gpu(w, mode=mode)
        if mode == "active":
            assert r["arith"] == "f32"
            check_against_oracle(oracle, w, r, range(W), pot_tol=POT_TOL_F32, exact_depth=False, floor=MARGIN_AUTO, max_iter=300,
                                 label=f"cold lanes, weights down to {light:.0e}")
    # a proposal replaces the zero potentials: two cycles, a restart from where they ended, and the rest
    first = run_gpu(w, max_iter=2)
    rest = run_gpu(w, warm=(first["f"], first["g"]))
    np.testing.assert_array_equal(np.where(first["status"] == 1, first["depth"], rest["depth"] + 2), run_gpu(w)["depth"])


@pytest.mark.parametrize("least", [2.0 ** -70, 2.0 ** -100, 2.0 ** -118])
@pytest.mark.parametrize("n,m", [(60, 64), (150, 100), (300, 200)])
def test_kernel_matrix_lanes_with_tiny_weights(oracle, n, m, least):
    # weights that span 30 orders of magnitude: plan entries of a light column are far below those of the others, and
    # a column whose entries fell out of the kernel matrix would come out wrong by O(eps)
    rng = np.random.default_rng(n)
    f32 = np.float32
    W, d = 3, 3
    a = rng.uniform(0.5, 1.5, (W, n)); b = rng.uniform(0.5, 1.5, (W, m))
    b[:, 5:9] *= least; a[1, 3] *= least; a[2, 7:20] *= 1e-20
    w = wl.Workload("light", rng.standard_normal((W, n, d)).astype(f32), (rng.standard_normal((W, m, d)) + 0.3).astype(f32),
                    (a / a.sum(1, keepdims=True)).astype(f32), (b / b.sum(1, keepdims=True)).astype(f32),
                    np.array([0.05, 0.3, 0.1], f32), 1e-4, 400)
    for mode in ("active", "masked"):
        r = run_gpu(w, compute="mixed", mode=mode)
        check_against_oracle(oracle, w, r, range(W), pot_tol=POT_TOL_F32, exact_depth=False, floor=MARGIN_AUTO, max_iter=400,
                             label=f"weights down to {least:.0e}, {n} x {m}, {mode}")
    rl = run_gpu(w, compute="mixed", mode="static", max_iter=6)                  # one launch per leg
    ref = oracle.solve_batch(w.x, w.y, w.a, w.b, w.eps, w.tol, max_iter=6)
    # in units of eps: 2^-22 per exponential, a few cycles
    err = np.abs(rl["g"] - ref.g).max(1) / w.eps
    assert err.max() <= 1e-5, err


@pytest.mark.parametrize("cycles", [2, 3, 5, 9, 30])
def test_kernel_matrix_lanes_whose_potentials_move_fast(oracle, cycles):
    # small regularisations, clouds apart: a cycle moves potentials by tens to hundreds of bits, so updates leave the
    # bands of the scalings in every way.  In units of eps the error is 2^-22 per exponential and cycle remembered
    rng = np.random.default_rng(5)
    f32 = np.float32
    W, n, m, d = 10, 100, 77, 4
    x = rng.standard_normal((W, n, d)).astype(f32); y = (rng.standard_normal((W, m, d)) * 0.7 + 0.5).astype(f32)
    a = rng.uniform(0.2, 1.8, (W, n)); b = rng.uniform(0.2, 1.8, (W, m))
    w = wl.Workload("fast", x, y, (a / a.sum(1, keepdims=True)).astype(f32), (b / b.sum(1, keepdims=True)).astype(f32),
                    np.geomspace(1e-3, 0.2, W).astype(f32), 1e-6, cycles)
    r = run_gpu(w, compute="mixed")
    ref = oracle.solve_batch(w.x, w.y, w.a, w.b, w.eps, w.tol, max_iter=cycles)
    err = np.maximum(np.abs(r["f"] - ref.f).max(1), np.abs(r["g"] - ref.g).max(1)) / w.eps
    assert err.max() <= 1e-6 * cycles + 2e-6, err


@pytest.mark.parametrize("n,m,d", [(150, 60, 5), (130, 100, 5), (70, 200, 5), (300, 300, 5), (300, 200, 64), (300, 500, 64), (600, 520, 64)])
def test_lanes_of_several_blocks_that_leave_the_band_again_and_again(oracle, n, m, d):
    # clouds two apart per dimension: some scaling of a column leaves 2^+-30 every four to seven cycles (counted with numpy in
    # float64), which one warp of one block finds first while others still look at the outcome of the exchange between blocks.
    # No wait may be reported to have run out, and the bits may not depend on how the cycles are shared out among launches.
    # (70 x 200 is a lane of one block, which has no exchange.)
    import torch
    from paper_2607_24741_b200 import binding as B
    rng = np.random.default_rng(n + m)
    W, cycles = 24, 60
    bf = lambda v: torch.from_numpy(v.astype(np.float32)).bfloat16().float().numpy()
    x = rng.standard_normal((W, n, d)); y = rng.standard_normal((W, m, d))
    if d == 64:
        x /= np.linalg.norm(x, axis=2, keepdims=True); y /= np.linalg.norm(y, axis=2, keepdims=True)
    x, y = (bf(x), bf(y + 2.0)) if d == 64 else (x.astype(np.float32), (y + 2.0).astype(np.float32))
    a = rng.uniform(0.1, 1.0, (W, n)); b = rng.uniform(0.1, 1.0, (W, m))
    eps = np.tile(np.float32([0.002, 0.01, 0.03, 0.05]), W // 4)
    w = wl.Workload("far apart", x, y, (a / a.sum(1, keepdims=True)).astype(np.float32), (b / b.sum(1, keepdims=True)).astype(np.float32),
                    eps, 1e-7, cycles, "bf16" if d == 64 else "f32")
    compute = "tensor" if d == 64 else "mixed"
    r = run_gpu(w, compute=compute)
    ref = oracle.solve_batch(w.x[:4], w.y[:4], w.a[:4], w.b[:4], w.eps[:4], w.tol, max_iter=cycles)
    err = np.maximum(np.abs(r["f"][:4] - ref.f).max(1), np.abs(r["g"][:4] - ref.g).max(1)) / w.eps[:4]
    # in units of eps: 2^-22 per exponential and cycle remembered; stored products are sums of d fp32 terms, off by up to
    # d 2^-24 |x| |y| each, twice that in the cost, which a leg (a soft minimum, so never more) hands on in every leg
    dot = 0.0 if d == 5 else 2.0 * d * 2.0 ** -24 * np.linalg.norm(x[:4], axis=2).max(1) * np.linalg.norm(y[:4], axis=2).max(1) / w.eps[:4]
    assert (err <= 1e-6 * cycles + 2e-6 + 2 * cycles * dot).all(), err
    t = lambda v: torch.from_numpy(v).to("cuda:0")
    xs, ys = (t(w.x).bfloat16(), t(w.y).bfloat16()) if d == 64 else (t(w.x), t(w.y))
    for run in (1, 7):
        sb = B.SinkhornBatch(xs, ys, t(w.a), t(w.b), t(w.eps), w.tol, compute=compute, max_iter=cycles)
        for _ in range(cycles // run + 1):
            sb.step(run)
        assert sb.active() == 0 and sb.check_guards() == -1
        f, g = sb.potentials(f64=True)
        np.testing.assert_array_equal(f.cpu().numpy(), r["f"]); np.testing.assert_array_equal(g.cpu().numpy(), r["g"])
        sb.close()


@pytest.mark.parametrize("kw", [dict(W=40, n=100, m=77, d=8), dict(W=24, n=64, m=64, d=2), dict(W=9, n=200, m=256, d=8), dict(W=5, n=300, m=500, d=8)])
@pytest.mark.parametrize("every,guard", [(1, 0.0), (4, 0.3)])
def test_static_batches_of_kernel_matrix_lanes_however_they_are_run(kw, every, guard):
    # the whole-cycle launches (the passed lanes wait and are caught up) against one launch per leg (phase timing), in
    # one drain, one cycle per call and a few cycles per call: same bits, same accounting; running lanes are
    # readable in between at the common cycle
    import torch
    from paper_2607_24741_b200 import binding as B
    w = wl.make("sweep", max_iter=150, tol=5e-3, **kw)
    t = lambda v: torch.from_numpy(v).to("cuda:0")
    args = [t(v) for v in (w.x, w.y, w.a, w.b, w.eps)]

    def run(step=0, profiling=False):
        sb = B.SinkhornBatch(*args, w.tol, mode="static", compute="mixed", max_iter=150, audit_every=every, guard_band=guard)
        sb.set_profiling(profiling)
        seen = {}
        while step and sb.active():
            sb.step(step)
            st = sb.stats()
            if st["cycles"] in (6, 12, 24, 48, 96):
                seen[st["cycles"]] = [v.cpu().numpy() for v in sb.potentials(f64=True)] + [st["slots"]]
                assert st["slots"] == w.shape[0] * st["cycles"]
        sb.drain()
        st = sb.stats(widths_cap=200)
        out = [v.cpu().numpy() for v in (*sb.potentials(f64=True), *sb.depths(), *sb.residuals(), *sb.last_audit())]
        assert sb.check_guards() == -1
        sb.close()
        return out + [np.array(st["widths"]), st["slots"], st["pair_terms"], st["cycles"]], seen
    ref, seen_ref = run(1, True)
    assert len(set(ref[2].tolist())) > 2 and (ref[3] != 0).all() and ref[-1] == ref[2].max()
    for step in (0, 1, 3, 24):
        got, seen = run(step)
        for a, b in zip(got, ref):
            np.testing.assert_array_equal(a, b)
        for k in seen:
            for a, b in zip(seen[k], seen_ref[k]):
                np.testing.assert_array_equal(a, b)


def test_last_audit_of_a_mask_does_not_depend_on_how_the_cycles_were_run():
    # lanes that froze earlier in a launch of many cycles are not screen-positive at its last audit
    import torch
    from paper_2607_24741_b200 import binding as B
    w = wl.make("sweep", W=40, n=100, m=77, tol=2e-2, max_iter=400)
    t = lambda v: torch.from_numpy(v).to("cuda:0")
    args = [t(v) for v in (w.x, w.y, w.a, w.b, w.eps)]
    for mode in ("masked", "masked_exit"):
        for cycles in (40, 160):
            out = []
            for step, profiling in ((1, True), (1, False), (cycles, False), (8, False)):
                sb = B.SinkhornBatch(*args, w.tol, mode=mode, compute="mixed", max_iter=400)
                sb.set_profiling(profiling)
                for _ in range(cycles // step):
                    sb.step(step)
                running = sb.depths()[1].cpu().numpy() == 0
                out.append([v.cpu().numpy() for v in sb.last_audit()])
                sb.close()
            assert 0 < running.sum() < 40 and np.isnan(out[0][1]).any()
            for rr, rc, fl in out[1:]:
                # (r_row of a lane that is frozen already is not a screen of anything: only the others')
                np.testing.assert_array_equal(rr[running], out[0][0][running])
                np.testing.assert_array_equal(rc, out[0][1]); np.testing.assert_array_equal(fl, out[0][2])


@pytest.mark.parametrize("n,m,d", [(1, 1, 1), (31, 65, 3), (2048, 64, 15), (2049, 63, 4), (4097, 65, 3), (100, 130, 17)])
def test_row_residual_over_the_whole_range_of_exponents(n, m, d):
    # blocks of 32, 64 and 128 rows at their edges, ragged tiles; entries from 2^-5000 to 2^40, a column of no weight
    # (g = -inf).  float64 sums stored as fp32: 2^-24 of the value, and m + d + 4 roundings of 2^-53 of an argument of up to 5000
    import torch
    from paper_2607_24741_b200 import binding as B
    rng = np.random.default_rng(n + 7 * m + d)
    x = rng.standard_normal((2, n, d)).astype(np.float32); y = rng.standard_normal((2, m, d)).astype(np.float32)
    a = rng.uniform(0.5, 1.5, (2, n)).astype(np.float32) / n
    eps = np.array([0.02, 0.5], np.float32)
    f = eps[:, None] * rng.uniform(-10.0, 10.0, (2, n)); g = eps[:, None] * rng.uniform(-10.0, 10.0, (2, m))
    cost = ((x.astype(np.float64)[:, :, None] - y.astype(np.float64)[:, None]) ** 2).sum(3)
    f += np.where(rng.random((2, n)) < 0.1, cost.min(2), 0.0)                # some rows with entries of the order of one
    if m > 1:
        g[:, m // 2] = -np.inf
    with np.errstate(under="ignore"):
        p = np.exp((f[:, :, None] + g[:, None] - cost) / eps.astype(np.float64)[:, None, None])
        ref = np.abs(p.sum(2) - a.astype(np.float64)).sum(1)
    t = lambda v: torch.from_numpy(v).to("cuda:0")
    r = B.sinkhorn_row_residual_static(t(x), t(y), t(a), t(f), t(g), t(eps)).cpu().numpy().astype(np.float64)
    np.testing.assert_allclose(r, ref, rtol=2.0 ** -24 + (m + d + 4) * 5000 * 2.0 ** -53 + 1e-11)


@pytest.mark.parametrize("n,d,dv", [(2700, 3, 3), (2600, 2, 1), (2600, 4, 4), (2600, 3, 5), (2564, 8, 3)])
def test_plan_application_by_tiles(oracle, n, d, dv):
    # enough row blocks for the tiles (81 of 32 and 64 rows), ragged ones, the widths of the values around those that the tiles are
    # made for; against the sums in float64.  fp32 results: 2^-24 of the value's own scale, 64-bit sums of m terms below that
    import torch
    from paper_2607_24741_b200 import binding as B
    rng = np.random.default_rng(n + d + dv)
    W, m = 2, 333
    x = rng.standard_normal((W, n, d)).astype(np.float32); y = (1.1 * rng.standard_normal((W, m, d))).astype(np.float32)
    a = np.full((W, n), 1.0 / n, np.float32); b = np.full((W, m), 1.0 / m, np.float32)
    eps = np.array([0.3, 0.6], np.float32)
    v = rng.standard_normal((W, m, dv)).astype(np.float32)
    t = lambda q: torch.from_numpy(q).to("cuda:0")
    sb = B.SinkhornBatch(t(x), t(y), t(a), t(b), t(eps), 1e-2, max_iter=40)
    sb.drain()
    f, g = (q.cpu().numpy() for q in sb.potentials(f64=True))
    out = sb.apply_plan(t(v)).cpu().numpy().astype(np.float64)
    sb.close()
    for k in range(W):
        cost = ((x[k].astype(np.float64)[:, None] - y[k].astype(np.float64)[None]) ** 2).sum(2)
        p = np.exp((f[k][:, None] + g[k][None] - cost) / float(eps[k]))
        want, size = p @ v[k].astype(np.float64), p @ np.abs(v[k]).astype(np.float64)
        assert (np.abs(out[k] - want) <= 2.0 ** -24 * np.abs(want) + 1e-11 * size).all()


# ---- large low-dimensional lanes in spatial order ----------------------------------------------------
def test_lanes_are_ranked_for_long_launches_of_wide_batches_only():
    # the ranking is one launch more, before a batch's first cycles; the results do not depend on it
    import torch
    from paper_2607_24741_b200 import binding as B
    t = lambda v: torch.from_numpy(v).to("cuda:0")
    for W, ranked in ((221, 0), (222, 1)):
        w = wl.make("sweep", W=W, n=20, m=30, d=4, max_iter=300)
        out = []
        for cycles, more in ((1, 0), (255, 0), (256, ranked)):
            sb = B.SinkhornBatch(t(w.x), t(w.y), t(w.a), t(w.b), t(w.eps), w.tol, max_iter=w.max_iter)
            count = [sb.launch_count()]
            for k in (cycles, cycles):
                sb.step(k)
                count.append(sb.launch_count())
            assert count[1] - count[0] - (count[2] - count[1]) == more, (W, cycles, count)
            sb.drain()
            out.append(sb.potentials(f64=True)[0].cpu().numpy())
            sb.close()
        np.testing.assert_array_equal(out[1], out[0]); np.testing.assert_array_equal(out[2], out[0])


@pytest.mark.parametrize("W,n,m,light", [(5, 20, 30, False), (6, 200, 256, False), (5, 300, 500, False), (160, 20, 30, False), (5, 20, 30, True)])
def test_a_masks_launch_ends_when_its_last_lane_has_passed(W, n, m, light):
    # drained lanes under a mask leave their launch together, in one block or in clusters, with lanes that stay in the log domain
    # (a weight below 2^-80) and with more lanes than are on the GPU at a time (whose launches stay short); same bits and
    # counts as without a mask, and what the last audit saw of lanes that froze long before it
    import torch
    from paper_2607_24741_b200 import binding as B
    w = wl.make("sweep", W=W, n=n, m=m, d=8, max_iter=700, tol=3e-3)
    if light:
        w.a[0, 3] = 2.0 ** -90
    t = lambda v: torch.from_numpy(v).to("cuda:0")
    out = []
    for mode in ("active", "masked"):
        sb = B.SinkhornBatch(t(w.x), t(w.y), t(w.a), t(w.b), t(w.eps), w.tol, mode=mode, max_iter=w.max_iter)
        before = sb.launch_count()
        sb.drain()
        launches = sb.launch_count() - before
        f, g = (v.cpu().numpy() for v in sb.potentials(f64=True))
        depth, status = (v.cpu().numpy() for v in sb.depths())
        assert sb.check_guards() == -1
        out.append((f, g, depth, status, launches, sb.stats()["cycles"]))
        if mode == "masked":
            rr, rc, fl = (v.cpu().numpy() for v in sb.last_audit())
            early = depth < depth.max()
            assert (rr[early] <= w.tol * 1.01).all() and not fl[early].any()
        sb.close()
    for a, b in zip(out[0][:4], out[1][:4]):
        np.testing.assert_array_equal(a, b)
    assert out[1][5] == out[0][5] == out[0][2].max()
    assert (out[1][4] <= 2 * 2 + 1) == (W < 148)           # two launches at most, each with its planner (and the ranking)


@pytest.mark.parametrize("n,m,Ws", [(40, 50, (330, 340, 400)), (100, 140, (140, 150, 300)), (140, 20, (735, 745))])
def test_kernels_of_128_and_255_registers_have_the_same_bits(n, m, Ws):
    # lanes whose matrix is in 32 registers a thread, or in half of the tensor memory, have two kernels, chosen by the mode and the number
    # of blocks; on both sides of each line STATIC, a mask and the plain batch give a lane the same bits
    import torch
    from paper_2607_24741_b200 import binding as B
    w = wl.make("sweep", W=max(Ws), n=n, m=m, d=4, max_iter=40)
    first = None
    for W in Ws:
        part = [torch.from_numpy(v[:W]).to("cuda:0") for v in (w.x, w.y, w.a, w.b, w.eps)]
        for mode in ("active", "static", "masked"):
            sb = B.SinkhornBatch(*part, 1e-9, mode=mode, max_iter=w.max_iter)      # (no lane passes: the common cycle of STATIC is theirs)
            sb.drain()
            f, g = (v.cpu().numpy() for v in sb.potentials(f64=True))
            assert (sb.depths()[0] == w.max_iter).all() and sb.check_guards() == -1
            sb.close()
            first = first or (f, g)
            k = len(first[0])
            np.testing.assert_array_equal(f[:k], first[0]); np.testing.assert_array_equal(g[:k], first[1])


@pytest.mark.parametrize("mode", ["active", "static", "masked"])
def test_a_drain_of_deep_lanes_waits_once_in_8192_cycles(mode):
    # a drain waits for a launch before it enqueues the next, so lanes of thousands of cycles must not be cut into many launches;
    # however they are cut, a lane's bits and the accounting are those of single steps.  (No lane passes: depth = max_iter.)
    import torch
    from paper_2607_24741_b200 import binding as B
    w = wl.make("sweep", W=3, n=30, m=20, d=4, max_iter=8300, tol=1e-12)
    t = lambda v: torch.from_numpy(v).to("cuda:0")
    out = []
    for step in (0, 700):
        sb = B.SinkhornBatch(t(w.x), t(w.y), t(w.a), t(w.b), t(w.eps), w.tol, mode=mode, max_iter=w.max_iter)
        before = sb.launch_count()
        while step and sb.active():
            sb.step(step)
        sb.drain()
        launches = sb.launch_count() - before
        f, g = (v.cpu().numpy() for v in sb.potentials(f64=True))
        s = sb.stats(widths_cap=9000)
        assert s["cycles"] == 8300 and s["slots"] == 3 * 8300 and list(s["widths"]) == [3] * 8300
        assert (sb.depths()[0] == 8300).all() and sb.check_guards() == -1
        out.append((f, g, launches))
        sb.close()
    assert out[0][2] <= (5 * 3 if mode == "static" else 2 * 3)      # (STATIC: 2048 cycles and three kernels a launch)
    np.testing.assert_array_equal(out[0][0], out[1][0]); np.testing.assert_array_equal(out[0][1], out[1][1])


def test_a_masks_launches_stay_short_however_many_cycles_are_asked_for():
    # under a logical mask lanes work until their launch ends: of 4096 cycles asked for, those past the launch in which the last
    # lane passes must be empty launches.  What a launch ran is not counted (Eq. 6-8 count to the last depth), so the launches are:
    # one of cycles and its planner for every 256
    import torch
    from paper_2607_24741_b200 import binding as B
    w = wl.make("tiny")
    t = lambda v: torch.from_numpy(v).to("cuda:0")
    for mode, most in (("masked", 256), ("masked_exit", 2048), ("active", 2048)):
        sb = B.SinkhornBatch(t(w.x), t(w.y), t(w.a), t(w.b), t(w.eps), w.tol, mode=mode, max_iter=w.max_iter)
        before = sb.launch_count()
        sb.step(4096)
        assert sb.active() == 0
        assert sb.launch_count() - before >= 2 * (4096 // most), mode
        assert sb.stats()["cycles"] == int(sb.depths()[0].max())
        sb.close()


@pytest.mark.parametrize("n,m,d", [(1024, 1024, 3), (1023, 1025, 3), (1055, 64, 2), (31, 1100, 4), (1024, 33, 1), (8193, 40, 3)])
def test_lanes_in_spatial_order(oracle, n, m, d):
    # sizes around the threshold, ragged boxes of 32, chunks of the ordering, every padded dimension; lanes of
    # several regularisations.  The mask control, which never changes its launch shape, must give the same bits, and a
    # warm proposal must find its way into the order.  (Clouds as wide as these mostly stay on the plain kernels: the
    # next test has the batches that are put into spatial order, and says so.)
    rng = np.random.default_rng(n + m + d)
    W = 3
    x = rng.standard_normal((W, n, d)); y = rng.standard_normal((W, m, d)) * 0.8 + 0.2
    a = rng.uniform(0.5, 1.5, (W, n)); b = rng.uniform(0.5, 1.5, (W, m))
    f32 = np.float32
    w = wl.Workload("spatial", x.astype(f32), y.astype(f32), (a / a.sum(1, keepdims=True)).astype(f32),
                    (b / b.sum(1, keepdims=True)).astype(f32), np.array([1.0, 0.2, 0.08], f32), 1e-3, 60)
    r = run_gpu(w, compute="f32")
    check_against_oracle(oracle, w, r, range(W), pot_tol=POT_TOL_F32, exact_depth=False, floor=MARGIN_AUTO, max_iter=60,
                         label=f"spatial order, {n} x {m}, d {d}")
    rm = run_gpu(w, compute="f32", mode="masked")
    np.testing.assert_array_equal(rm["f"], r["f"]); np.testing.assert_array_equal(rm["r_row"], r["r_row"])
    part = oracle.solve_batch(w.x, w.y, w.a, w.b, w.eps, w.tol, fixed_cycles=2)
    rw = run_gpu(w, compute="f32", warm=(part.f, part.g))
    check_against_oracle(oracle, w, rw, range(W), pot_tol=POT_TOL_F32, exact_depth=False, floor=MARGIN_AUTO, max_iter=60,
                         warm=(part.f, part.g), label=f"spatial order, warm, {n} x {m}, d {d}")
    # clouds far apart at a small eps: the first legs move potentials by far more than the estimate allows for
    far = wl.Workload("spatial_far", w.x, (w.y + f32(6.0)).astype(f32), w.a, w.b, np.array([0.9, 0.7, 0.5], f32), 1e-3, 12)
    rf = run_gpu(far, compute="f32")
    ref = oracle.solve_batch(far.x, far.y, far.a, far.b, far.eps, far.tol, max_iter=12)
    assert pot_err(rf["f"], rf["g"], ref.f, ref.g, far.eps.astype(np.float64)).max() <= POT_TOL_F32


def _cloud_pair(law, W, n, m, d, rng):
    if law == "sphere":
        x = rng.standard_normal((W, n, d)); x /= np.linalg.norm(x, axis=2, keepdims=True)
        y = rng.standard_normal((W, m, d)); y /= np.linalg.norm(y, axis=2, keepdims=True)
        return x, y + 0.01 * rng.standard_normal((W, m, d))
    if law == "flat":                                    # a sheet in more dimensions than it has
        x, y = rng.random((W, n, d)), rng.random((W, m, d))
        x[:, :, 2:] *= 0.01; y[:, :, 2:] *= 0.01
        return x, y
    return rng.random((W, n, d)), rng.random((W, m, d))


# (law, n, m, d, eps, spatial order expected): boxes of 32 points against the reach of eps
SPATIAL = [("sphere", 4096, 4000, 3, 0.01, True), ("sphere", 2500, 2047, 3, 0.01, True), ("sphere", 4096, 4096, 3, 0.1, False),
           ("cube", 2048, 1500, 2, 0.002, True), ("cube", 1024, 1025, 1, 0.002, True), ("cube", 2048, 2048, 2, 0.03, False),
           ("flat", 1800, 3001, 4, 0.003, True), ("sphere", 8193, 300, 3, 0.01, True), ("flat", 2048, 33, 3, 0.003, True), ("cube", 1500, 1500, 4, 0.02, False)]


@pytest.mark.parametrize("law,n,m,d,eps,expected", SPATIAL)
def test_spatial_order_is_taken_where_it_can_skip(oracle, law, n, m, d, eps, expected):
    # the choice follows the data (the ordering is one more set-up launch), and either way the state after a few cycles
    # is the oracle's; lanes of one batch are decided together
    import torch
    from paper_2607_24741_b200 import binding as B
    rng = np.random.default_rng(n + m)
    W = 2
    x, y = _cloud_pair(law, W, n, m, d, rng)
    f32 = np.float32
    a = rng.uniform(0.5, 1.5, (W, n)); b = rng.uniform(0.5, 1.5, (W, m))
    w = wl.Workload(law, x.astype(f32), y.astype(f32), (a / a.sum(1, keepdims=True)).astype(f32),
                    (b / b.sum(1, keepdims=True)).astype(f32), np.array([eps, 1.3 * eps], f32), 1e-3, 6)
    t = lambda v: torch.from_numpy(v).to("cuda:0")

    def run(**kw):
        sb = B.SinkhornBatch(t(w.x), t(w.y), t(w.a), t(w.b), t(w.eps), kw.pop("tol", w.tol), max_iter=6, **kw)
        launches, arith = sb.launch_count(), sb.arithmetic()
        sb.drain()
        f, g = (v.cpu().numpy() for v in sb.potentials(f64=True))
        assert sb.check_guards() == -1
        sb.close()
        return f, g, launches, arith
    f, g, launches, arith = run()
    assert arith == "f32"
    plain = run(column_split=1)
    assert launches - plain[2] == (2 if expected else 1)      # the estimate, the ordering
    ref = oracle.solve_batch(w.x, w.y, w.a, w.b, w.eps, w.tol, max_iter=6)
    e = w.eps.astype(np.float64)
    assert pot_err(f, g, ref.f, ref.g, e).max() <= POT_TOL_F32
    assert pot_err(plain[0], plain[1], ref.f, ref.g, e).max() <= POT_TOL_F32
    if expected:
        # a mask never changes its launch shape; a warm proposal finds its way into the order
        masked = run(mode="masked")
        np.testing.assert_array_equal(masked[0], f); np.testing.assert_array_equal(masked[1], g)
        part = oracle.solve_batch(w.x, w.y, w.a, w.b, w.eps, w.tol, fixed_cycles=2)
        rw = run_gpu(w, warm=(part.f, part.g), max_iter=4)
        assert pot_err(rw["f"], rw["g"], ref.f, ref.g, e).max() <= POT_TOL_F32
    # a cost form that the caller names, and looser tolerances, stay on the plain kernels
    for kw in (dict(cost_form=1), dict(cost_form=2), dict(tol=1e-2)):
        assert run(**kw)[2] == plain[2], kw


# (law, n, m, d, eps): groups of 16 rows and lists by warp at their edges; lists longer than what tensor memory holds (a
# large share of the pairs); outliers on both sides, whose potentials move by many bits in the first cycles
ONE_PASS = [("sphere", 1040, 1025, 3, 0.02), ("sphere", 1100, 2049, 3, 0.04), ("cube", 1031, 97, 2, 0.002), ("cube", 40, 1025, 1, 0.002),
            ("flat", 1500, 1100, 4, 0.004), ("outliers", 1300, 1300, 3, 0.01), ("sphere", 600, 513, 3, 0.01), ("cube", 530, 520, 2, 0.005)]


@pytest.mark.parametrize("law,n,m,d,eps", ONE_PASS)
def test_both_legs_in_one_pass(oracle, monkeypatch, law, n, m, d, eps):
    # lanes in spatial order whose g-legs take the column sums that the f-leg's pass has left, over enough cycles for lists to be
    # kept and made again, against the oracle; in a workspace without room for the lists each leg goes over the pairs by itself, and
    # lanes that come in later, move or stay under a mask have the bits of one batch
    import torch
    from paper_2607_24741_b200 import binding as B
    rng = np.random.default_rng(n + m + d)
    W, cycles, f32 = 3, 30, np.float32
    x, y = _cloud_pair("sphere" if law == "outliers" else law, W, n, m, d, rng)
    if law == "outliers":
        for c in (x, y):
            far = rng.random(c.shape[:2]) < 0.05
            c[far] = rng.uniform(-1.0, 1.0, (int(far.sum()), d))
    a = rng.uniform(0.5, 1.5, (W, n)); b = rng.uniform(0.5, 1.5, (W, m))
    w = wl.Workload(law, x.astype(f32), y.astype(f32), (a / a.sum(1, keepdims=True)).astype(f32),
                    (b / b.sum(1, keepdims=True)).astype(f32), (eps * np.array([1.0, 1.15, 1.3])).astype(f32), 1e-3, cycles)
    ref = oracle.solve_batch(w.x, w.y, w.a, w.b, w.eps, w.tol, max_iter=cycles)
    e = w.eps.astype(np.float64)
    r = run_gpu(w)
    assert r["arith"] == "f32"
    # these kernels did run: lanes in spatial order are ordered by one more launch at create, and groups of 16 have their lists (a
    # record of 512 bytes: the cycle they are from, in word 38, and the lengths for four warps, whole steps of 32, in words 40 to 43)
    t = lambda v: torch.from_numpy(v).to("cuda:0")
    at_create = []
    monkeypatch.setattr(B, "torch", _ZeroedWorkspace())
    for kw in ({}, dict(column_split=1)):
        sb = B.SinkhornBatch(t(w.x), t(w.y), t(w.a), t(w.b), t(w.eps), w.tol, max_iter=cycles, **kw)
        at_create.append(sb.launch_count())
        if not kw:
            sb.step(1)
            torch.cuda.synchronize()
            words = sb.workspace[:sb.workspace.numel() // 256 * 256].view(torch.int32).view(-1, 64)
            length = words[(words[:, 38] == 1) & (words[:, 40:44] % 32 == 0).all(1) & (words[:, 40:44] <= m + 96).all(1) & (words[:, 40:44] >= 0).all(1), 40:44]
            assert len(length) >= W * ((n + 15) // 16)
            if (n, m) == (1100, 2049):
                assert int(length.max()) > 256               # more than what tensor memory holds
        sb.close()
    monkeypatch.undo()
    assert at_create[0] - at_create[1] == 2                  # the estimate, the ordering
    np.testing.assert_array_equal(r["depth"], ref.depth)
    assert pot_err(r["f"], r["g"], ref.f, ref.g, e).max() <= POT_TOL_F32
    rm = run_gpu(w, mode="masked")
    np.testing.assert_array_equal(rm["f"], r["f"]); np.testing.assert_array_equal(rm["g"], r["g"])
    # values of the last audit
    sb = B.SinkhornBatch(*(torch.from_numpy(v).to("cuda:0") for v in (w.x, w.y, w.a, w.b, w.eps)), w.tol, max_iter=cycles)
    sb.step(2)
    assert (sb.last_audit()[0] > 0).all()
    sb.close()
    # one slot after the other, then two at a time: later lanes in slots that others have used
    sb = B.SinkhornBatch(t(w.x[:2]), t(w.y[:2]), t(w.a[:2]), t(w.b[:2]), t(w.eps[:2]), w.tol, max_iter=cycles, lane_capacity=W)
    while sb.active() == 2:
        sb.step(1)
    sb.refill(t(w.x[2:]), t(w.y[2:]), t(w.a[2:]), t(w.b[2:]), t(w.eps[2:]))
    sb.drain()
    f, g = sb.potentials(f64=True)
    np.testing.assert_array_equal(f.cpu().numpy(), r["f"]); np.testing.assert_array_equal(g.cpu().numpy(), r["g"])
    assert sb.check_guards() == -1
    sb.close()
    if min(n, m) < 1000:                                  # (the lists are small beside what an automatic batch is sized for)
        return
    whole = B.sinkhorn_batch_workspace_bytes
    monkeypatch.setattr(B, "sinkhorn_batch_workspace_bytes", lambda cfg: whole(cfg) - 256)
    rs = run_gpu(w)
    np.testing.assert_array_equal(rs["depth"], ref.depth)
    assert pot_err(rs["f"], rs["g"], ref.f, ref.g, e).max() <= POT_TOL_F32
    assert not np.array_equal(rs["f"], r["f"])               # (other arithmetic, to rounding)


def test_one_pass_under_the_other_modes_and_between_its_cycles(oracle):
    # STATIC over more than the first cycles, the mask that skips frozen lanes, audits on a grid, and timed dry launches between
    # cycles (whose lists are thrown away or the same): the bits, depths and audits of one plain solve
    from paper_2607_24741_b200 import binding as B
    n, m, cycles = 1300, 1100, 90
    w = _sphere_lanes(4, n, m, [0.05, 0.03, 0.012, 0.01], cycles)
    r = run_gpu(w)
    assert r["arith"] == "f32" and (r["depth"] < cycles).any() and (r["depth"] == cycles).any()
    rx = run_gpu(w, mode="masked_exit")
    for k in ("f", "g", "depth", "status", "r_row"):
        np.testing.assert_array_equal(rx[k], r[k])
    # (12 cycles: no lane has passed, so STATIC's common cycle is max_iter)
    few, static = run_gpu(w, max_iter=12), run_gpu(w, mode="static", max_iter=12)
    assert (few["depth"] == 12).all()
    np.testing.assert_array_equal(static["f"], few["f"]); np.testing.assert_array_equal(static["g"], few["g"])
    ref = oracle.solve_batch(w.x, w.y, w.a, w.b, w.eps, w.tol, max_iter=cycles, audit_every=7)
    grid = run_gpu(w, audit_every=7)
    np.testing.assert_array_equal(grid["depth"], ref.depth)
    assert pot_err(grid["f"], grid["g"], ref.f, ref.g, w.eps.astype(np.float64)).max() <= POT_TOL_F32
    for when in (0, 1, 2, 9):
        sb = B.SinkhornBatch(*_parts(w, slice(0, 4)), w.tol, max_iter=cycles)
        for k in range(12):
            if k % 10 == when:
                sb.profile_update(leg=0, reps=2); sb.profile_update(leg=1, reps=2)
            sb.step(1)
        sb.drain()
        f, g = (v.cpu().numpy() for v in sb.potentials(f64=True))
        np.testing.assert_array_equal(f, r["f"]); np.testing.assert_array_equal(g, r["g"])
        np.testing.assert_array_equal(sb.residuals()[0].cpu().numpy(), r["r_row"])
        assert sb.check_guards() == -1
        sb.close()


def _sphere_lanes(W, n, m, eps, cycles, seed=5):
    # lanes on a noisy unit sphere, uneven weights: at eps 0.01 to 0.03 they go into spatial order
    rng, f32 = np.random.default_rng(seed), np.float32
    x, y = _cloud_pair("sphere", W, n, m, 3, rng)
    a = rng.uniform(0.5, 1.5, (W, n)); b = rng.uniform(0.5, 1.5, (W, m))
    return wl.Workload("sphere", x.astype(f32), y.astype(f32), (a / a.sum(1, keepdims=True)).astype(f32),
                       (b / b.sum(1, keepdims=True)).astype(f32), np.asarray(eps, f32), 1e-3, cycles)


def _parts(w, lanes):
    import torch
    return [torch.from_numpy(np.ascontiguousarray(v[lanes])).to("cuda:0") for v in (w.x, w.y, w.a, w.b, w.eps)]


@pytest.mark.parametrize("first", [0, 3])
def test_a_lane_that_is_not_finite_leaves_its_neighbours_alone(first):
    # one pass: a lane whose points are finite but too far apart for fp32 comes in through a queue (create's radius test does not
    # see it) and takes the place of lane `first`, before another's arrays or before the end of all.  Its sums are NaN in the second cycle; no
    # part of them may go into another lane's totals or beyond the last one's, so the others' bits are those they have beside
    # a lane that is fine
    from paper_2607_24741_b200 import binding as B
    eps = np.full(5, 0.01, np.float32)
    eps[first] = 0.06
    w = _sphere_lanes(5, 1040, 1050, eps, 150)
    out = []
    for broken in (False, True):
        late = _parts(w, slice(4, 5))
        if broken:
            late[1][0, 5] = 1.0e20
            late[1][0, 6] = -1.0e20
        sb = B.SinkhornBatch(*_parts(w, slice(0, 4)), w.tol, max_iter=w.max_iter, lane_capacity=5)
        while sb.active() == 4:
            sb.step(1)
        assert sb.active() == 3
        sb.refill(*late)
        sb.drain()
        f, g = (v.cpu().numpy() for v in sb.potentials(f64=True))
        depth, status = (v.cpu().numpy() for v in sb.depths())
        assert sb.check_guards() == -1
        sb.close()
        assert depth[first] < depth[[k for k in range(4) if k != first]].min()
        assert status[4] == (B.LANE_NONFINITE if broken else B.LANE_ITER_LIMIT)
        out.append((f[:4], g[:4], depth[:4]))
    for p, q in zip(*out):
        np.testing.assert_array_equal(p, q)


@pytest.mark.parametrize("W,slots,n,m,cycles", [(3, 1, 600, 530, 40), (264, 66, 8192, 8192, 2)])
def test_a_queue_of_lanes_in_spatial_order_has_the_bits_of_one_batch(W, slots, n, m, cycles):
    # whether lanes of 513 to 1023 points are in spatial order, and whether there are lists, must not depend on the slots: a queue
    # through one slot, and one whose slots' lists are small where those of all its lanes are 2.2 GiB
    import torch
    from paper_2607_24741_b200 import binding as B
    if W < 100:
        w = _sphere_lanes(W, n, m, np.full(W, 0.01), cycles)
        parts = lambda a, b: _parts(w, slice(a, b))
    else:                                                  # (made on the GPU: 50 MB of points)
        gen = torch.Generator("cuda:0").manual_seed(1)
        c = torch.randn(2, W, n, 3, device="cuda:0", generator=gen)
        c /= c.norm(dim=3, keepdim=True)
        flat = torch.full((W, n), 1.0 / n, device="cuda:0")
        every = (c[0], c[1], flat, flat, torch.full((W,), 0.01, device="cuda:0"))
        parts = lambda a, b: [v[a:b].contiguous() for v in every]
    sb = B.SinkhornBatch(*parts(0, W), 1e-3, max_iter=cycles)
    sb.drain()
    whole = sb.potentials(f64=True)
    sb.close()
    del sb
    sb = B.SinkhornBatch(*parts(0, slots), 1e-3, max_iter=cycles, lane_capacity=W)
    for k in range(slots, W, slots):
        while sb.active():
            sb.step(4)
        sb.refill(*parts(k, min(k + slots, W)))
    sb.drain()
    queue = sb.potentials(f64=True)
    assert sb.check_guards() == -1
    sb.close()
    assert torch.equal(queue[0], whole[0]) and torch.equal(queue[1], whole[1])


class _ZeroedWorkspace:
    # stands in for torch in the binding: workspaces start as zeros
    def __getattr__(self, name):
        import torch
        return torch.zeros if name == "empty" else getattr(torch, name)


def test_an_f_leg_that_outruns_its_lists_is_noted(oracle, monkeypatch):
    # one pass: lists are chosen with phi from before the f-leg; where the leg raises it by more than they have room for (outliers in the first
    # cycle, two to six bits: beyond, rows start over), fewer columns may take the totals.  What is missing without that is at
    # most 2^-20 of a total and cannot be told from rounding in the potentials, so the note itself is looked for: integers by
    # lane, of this cycle and of the next, by themselves in 256 bytes
    import torch
    from paper_2607_24741_b200 import binding as B
    monkeypatch.setattr(B, "torch", _ZeroedWorkspace())
    W, n = 4, 1500
    w = _sphere_lanes(W, n, n, np.full(W, 0.01), 1)
    rng = np.random.default_rng(8)
    for c in (w.x, w.y):
        far = rng.random(c.shape[:2]) < 0.1
        c[far] = rng.uniform(-1.0, 1.0, (int(far.sum()), 3))
    sb = B.SinkhornBatch(*_parts(w, slice(0, W)), w.tol, max_iter=w.max_iter)
    sb.step(1)
    torch.cuda.synchronize()
    words = sb.workspace[:sb.workspace.numel() // 256 * 256].view(torch.int32).view(-1, 64)
    some, none = (words > 64) & (words < 1 << 24), words == 0
    alone = none[:, 2 * W:].all(1) & (some[:, :W].all(1) & none[:, W:2 * W].all(1) | none[:, :W].all(1) & some[:, W:2 * W].all(1))
    assert int(alone.sum()) == 1
    sb.drain()
    f, g = (v.cpu().numpy() for v in sb.potentials(f64=True))
    sb.close()
    ref = oracle.solve_batch(w.x, w.y, w.a, w.b, w.eps, w.tol, max_iter=1)
    assert pot_err(f, g, ref.f, ref.g, w.eps.astype(np.float64)).max() <= POT_TOL_F32


def test_a_half_box_without_points_has_no_largest_potential(monkeypatch):
    # one pass: the source's largest potentials are kept for halves of a box of 32; that of the last box is empty where n mod 32 is 1 to 16,
    # and must not hold its box's pairs up with what was there before.  Its value is minus infinity (-3e38) in both buffers, as
    # are the two of an empty half's record and the upper corner of its box: seven words a lane of a workspace that was zero
    import torch
    from paper_2607_24741_b200 import binding as B
    monkeypatch.setattr(B, "torch", _ZeroedWorkspace())
    w = _sphere_lanes(3, 1040, 1056, [0.01, 0.01, 0.01], 50)
    warm = [torch.zeros(3, k, dtype=torch.float64, device="cuda:0") for k in (1040, 1056)]
    for cycles, first in ((0, None), (0, warm), (7, None)):
        sb = B.SinkhornBatch(*_parts(w, slice(0, 3)), w.tol, max_iter=w.max_iter)
        if first:
            sb.warm_start(*first)
        sb.step(cycles)
        torch.cuda.synchronize()
        words = sb.workspace[:sb.workspace.numel() // 4 * 4].view(torch.float32)
        assert int((words == torch.tensor(-3.0e38, device="cuda:0")).sum()) == 3 * 7
        sb.close()


@pytest.mark.parametrize("mode", ["masked", "static"])
def test_a_frozen_lane_keeps_its_lists(mode):
    # one pass: the first lane (a flat kernel) passes after one cycle, in which the potentials of its heavy targets rise by three bits, so
    # that the pass which finds it done calls for new lists.  It works on under a mask, and must not make them again in
    # every cycle.  What a group's lists were made from is kept as a count of cycles, so
    # a lane that makes its lists in cycle k writes the number k once for every group of 16 points
    import torch
    from paper_2607_24741_b200 import binding as B
    n, cycles = 2048, range(98, 118)                       # (lengths of lists are multiples of 32)
    w = _sphere_lanes(3, n, 2048, [400.0, 0.01, 0.01], 200)
    w.b[0, ::16] *= 8.0
    w.b[0] /= w.b[0].astype(np.float64).sum()
    sb = B.SinkhornBatch(*_parts(w, slice(0, 3)), w.tol, mode=mode, max_iter=w.max_iter)
    sb.step(cycles[0] - 1)
    depth = sb.depths()[0].cpu().numpy()
    assert depth[0] == 1 and (mode == "static" or not depth[1:].any())
    made = []
    for k in cycles:
        sb.step(1)
        assert sb.stats()["cycles"] == k
        words = sb.workspace[:sb.workspace.numel() // 4 * 4].view(torch.int32)
        made.append(int((words == k).sum()) >= n // 16)
    sb.close()
    assert sum(made) <= 4, made                            # (the other lanes' lists hold for a dozen cycles and more by then)


def test_a_lanes_bits_do_not_depend_on_the_width_of_its_launches():
    # one pass: column launches of ten lanes have blocks of 64 columns, those of three lanes blocks of 32; in the first cycles some columns
    # are low and go over the pairs, which must leave their neighbours in a block to the totals.  Outliers on both sides, a
    # ragged last box; one batch, a queue through three slots, lanes by themselves
    from paper_2607_24741_b200 import binding as B
    W, n, m = 10, 1030, 4001
    assert (m + 63) // 64 * 3 < 592 <= (m + 63) // 64 * W          # (the rule of the launch)
    w = _sphere_lanes(W, n, m, np.linspace(0.01, 0.02, W), 16)
    rng = np.random.default_rng(2)
    for c in (w.x, w.y):
        far = rng.random(c.shape[:2]) < 0.05
        c[far] = rng.uniform(-1.0, 1.0, (int(far.sum()), 3))
    whole = run_gpu(w)
    assert whole["arith"] == "f32"
    sb = B.SinkhornBatch(*_parts(w, slice(0, 3)), w.tol, max_iter=w.max_iter, lane_capacity=W)
    for k in range(3, W, 3):
        while sb.active():
            sb.step(4)
        sb.refill(*_parts(w, slice(k, min(k + 3, W))))
    sb.drain()
    f, g = (v.cpu().numpy() for v in sb.potentials(f64=True))
    assert sb.check_guards() == -1
    sb.close()
    np.testing.assert_array_equal(f, whole["f"]); np.testing.assert_array_equal(g, whole["g"])
    for k in (0, W - 1):
        one = run_gpu(wl.Workload("one", *(np.ascontiguousarray(v[k:k + 1]) for v in (w.x, w.y, w.a, w.b, w.eps)), w.tol, w.max_iter))
        np.testing.assert_array_equal(one["f"][0], whole["f"][k]); np.testing.assert_array_equal(one["g"][0], whole["g"][k])


@pytest.mark.parametrize("cost_form", [0, 1, 2])
def test_large_radii_in_fp32_take_differences_whatever_the_size(oracle, cost_form):
    # scaled squared radius of 1000 to 3000, asked for in fp32: cost_form 0 and 2 must be the difference form with
    # two-part potentials.  Per cycle its error is a few ulp of the settled terms, the expanded form's an ulp of the radius
    rng = np.random.default_rng(3)
    W, n, m, d, cycles = 3, 1100, 1030, 3, 4
    f32 = np.float32
    x = rng.standard_normal((W, n, d)); x /= np.linalg.norm(x, axis=2, keepdims=True)
    y = x[:, rng.permutation(n)[:m]] + 0.02 * rng.standard_normal((W, m, d))
    w = wl.Workload("radius", x.astype(f32), y.astype(f32), np.full((W, n), 1 / n, f32), np.full((W, m), 1 / m, f32),
                    np.array([2e-3, 1e-3, 7e-4], f32), 1e-3, cycles)
    r = run_gpu(w, compute="f32", cost_form=cost_form, max_iter=cycles)
    ref = oracle.solve_batch(w.x, w.y, w.a, w.b, w.eps, w.tol, max_iter=cycles)
    e = w.eps.astype(np.float64)
    err = np.maximum(np.abs(r["f"] - ref.f).max(1), np.abs(r["g"] - ref.g).max(1)) / e
    radius = 1.4427 / e * 1.1
    assert (err <= (radius * 2.0 ** -22 * cycles if cost_form == 1 else 2e-5)).all(), (cost_form, err, radius)


# ---- float64 pair sums by column tiles ---------------------------------------------------------------
@pytest.mark.parametrize("n,m,d,dv", [(1, 1, 1, 1), (63, 65, 4, 4), (64, 64, 5, 5), (65, 128, 16, 16), (130, 63, 17, 3), (40, 70, 32, 16),
                                      (33, 50, 33, 2), (4097, 20, 3, 3)])
def test_pair_sums_in_float64_at_the_edges_of_their_tiles(oracle, n, m, d, dv):
    # plan application and the row residual of given potentials: tile edges, the last tiled dimension and the first
    # beyond, both value widths, both block sizes of the residual.  Both are float64 sums rounded once to fp32:
    # 2^-24 relative, plus the potentials' own rounding (1e-16 of C / eps = 1e3 in an exponent) far below it
    import torch
    from paper_2607_24741_b200 import binding as B
    w = wl.make("sweep", W=2, n=n, m=m, d=d, max_iter=7)
    t = lambda v: torch.from_numpy(v).to("cuda:0")
    args = [t(v) for v in (w.x, w.y, w.a, w.b, w.eps)]
    sb = B.SinkhornBatch(*args, w.tol, compute="f64", max_iter=7)
    sb.drain()
    f, g = sb.potentials(f64=True)
    v = torch.randn(2, m, dv, device="cuda:0", generator=torch.Generator("cuda:0").manual_seed(n + m))
    out = sb.apply_plan(v).cpu().numpy()
    sb.close()
    fr, gr = f.cpu().numpy(), g.cpu().numpy()
    # the residual of potentials that are not a solution's, so that it is far from its rounding
    f2 = f + 0.3 * args[4][:, None].double() * torch.sin(1.0 + torch.arange(n, device="cuda:0", dtype=torch.float64))
    rr = B.sinkhorn_row_residual_static(args[0], args[1], args[2], f2, g, args[4]).cpu().numpy()
    f2[0, n // 2] = float("inf")                       # an infinite potential: its lane's residual is not finite, the other's is
    bad = B.sinkhorn_row_residual_static(args[0], args[1], args[2], f2, g, args[4]).cpu().numpy()
    assert not np.isfinite(bad[0]) and bad[1] == rr[1]
    f2[0, n // 2] = 0.0
    for k in range(2):
        want = oracle.apply_plan(w.x[k], w.y[k], float(w.eps[k]), fr[k], gr[k], v[k].cpu().numpy())
        scale = np.abs(want).max()
        np.testing.assert_allclose(out[k], want, rtol=2.0 ** -23, atol=1e-9 * scale)
        fk = fr[k] + 0.3 * float(w.eps[k]) * np.sin(1.0 + np.arange(n))
        res, _ = oracle.residuals(w.x[k], w.y[k], w.a[k], w.b[k], float(w.eps[k]), fk, gr[k])
        assert abs(rr[k] - res) <= 2.0 ** -23 * res + 1e-12


@pytest.mark.parametrize("eps", [1e-2, 1e-3])
@pytest.mark.parametrize("offset,outlier", [(0.0, 0.0), (1e2, 0.0), (1e4, 0.0), (1e5, 0.0), (1e4, 1e2)])
def test_pair_sums_do_not_depend_on_where_the_clouds_lie(oracle, offset, outlier, eps):
    # clouds far from the origin, and a block whose first point is far from all others: the cost is a difference,
    # so both calls must be as tight as for centred clouds.  Bound: the fp32 result's 2^-24, and arguments good to
    # 2^-32 (k f is below 2^21 here: its own rounding, 2^-32, is of that size too)
    import torch
    from paper_2607_24741_b200 import binding as B
    rng = np.random.default_rng(11)
    W, n, m, d = 2, 130, 150, 3
    f32 = np.float32
    x = (offset + 0.3 * rng.standard_normal((W, n, d))).astype(f32)
    y = (offset + 0.3 * rng.standard_normal((W, m, d))).astype(f32)
    x[:, 0] += f32(outlier)
    y[:, 70] -= f32(outlier)
    a, b = np.full((W, n), 1.0 / n, f32), np.full((W, m), 1.0 / m, f32)
    e = np.full(W, eps, f32)
    t = lambda v: torch.from_numpy(v).to("cuda:0")
    args = [t(v) for v in (x, y, a, b, e)]
    sb = B.SinkhornBatch(*args, 1e-9, compute="f64", max_iter=9)
    sb.drain()
    f, g = sb.potentials(f64=True)
    v = (0.5 + rng.random((W, m, 2))).astype(f32)
    out = sb.apply_plan(t(v)).cpu().numpy()
    sb.close()
    f2 = f + 0.3 * eps * torch.sin(1.0 + torch.arange(n, device="cuda:0", dtype=torch.float64))
    rr = B.sinkhorn_row_residual_static(args[0], args[1], args[2], f2, g, args[4]).cpu().numpy()
    for k in range(W):
        want = oracle.apply_plan(x[k], y[k], float(e[k]), f[k].cpu().numpy(), g[k].cpu().numpy(), v[k])
        np.testing.assert_allclose(out[k], want, rtol=2.0 ** -23, atol=0.0)
        res, _ = oracle.residuals(x[k], y[k], a[k], b[k], float(e[k]), f2[k].cpu().numpy(), g[k].cpu().numpy())
        assert abs(rr[k] - res) <= 2.0 ** -23 * res + 2.0 ** -31

"""Adaptive DOP 8(5) on small Henon-Heiles ensembles (a pipeline of warps, two lanes per orbit)
against the one-thread-per-orbit form, which the same orbits take inside an ensemble padded with
FORBIDDEN orbits beyond the pipeline's size.  Step counts, rejections and statuses are equal.  The
forms sum in another order, which moves a step size by about 1e-8 of itself (the error estimate is
a small difference), a step's result by 1e-8 of the local error below 1e-7; states and vectors are
held to 1e-9 of their norm at equal times: at t = 12, and for orbits that froze earlier after the
shift of their last step's time (states by f(x) dt, vectors within |J| |w| |dt|, |J| < 10)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2507_00622_gb300 import chs  # noqa: E402

PAD = 15000


def _run(n, pad, k, calls=1, t_final=12.0, tol=1e-8, h_max=0.0, h0=0.05, **kw):
    S = chs.System(chs.HENON_HEILES, 2)
    rng = np.random.default_rng(n + k)
    m = max(n, pad)
    ics = np.full((4, m), 0.01)
    ics[:, :n] = rng.uniform(-0.33, 0.33, (4, n))
    ics[2:, :n:5] *= 2.4  # some escape
    if n > 8:
        ics[0, 7] = np.nan
    st = np.full(m, chs.ORBIT_FORBIDDEN, dtype=np.int32)
    st[:n] = 0
    w = np.zeros((k * 4, m))
    w[:, :n] = rng.uniform(-1, 1, (k * 4, n))
    ens = chs.DeviceEnsemble.empty(m, 4, k)
    abi = ens.abi(with_ld=False)
    par = dict(n_dev=k, integrator=chs.DOP853, **kw)
    chs.chs_ensemble_init(S.h, chs.params(0.05, 1, **par), abi, torch.from_numpy(ics).cuda(),
                          torch.from_numpy(st).cuda(), torch.from_numpy(w).cuda())
    f64 = dict(dtype=torch.float64, device="cuda")
    t, h = torch.zeros(m, **f64), torch.full((m,), h0, **f64)
    el, em = torch.zeros(m, **f64), torch.zeros(m, **f64)
    rej = torch.zeros(m, dtype=torch.int64, device="cuda")
    for _ in range(calls):
        n_steps = 1_000_000 if calls == 1 else 9
        chs.chs_integrate_adaptive(S.h, chs.params(0.05, n_steps, **par), chs.Adaptive(t_final, tol, tol, h_max), abi,
                                   t, h, el, em, rej)
    torch.cuda.synchronize()
    out = dict(x=ens.x, w=ens.w, dh=ens.dh_max, n_exec=ens.n_exec, status=ens.status, t=t, rej=rej, em=em)
    return {f: v.cpu().numpy()[..., :n] for f, v in out.items()}


def _close(a, b):
    for f in ("n_exec", "rej", "status"):
        np.testing.assert_array_equal(a[f], b[f], err_msg=f)
    ok = np.isfinite(b["x"]).all(axis=0)
    assert np.array_equal(ok, np.isfinite(a["x"]).all(axis=0))
    np.testing.assert_allclose(a["t"], b["t"], rtol=1e-6)
    dt = (a["t"] - b["t"])[ok]
    x = b["x"][:, ok]
    f = np.stack([x[2], x[3], -x[0] * (1 + 2 * x[1]), -x[1] - x[0] ** 2 + x[1] ** 2])
    assert (np.abs(a["x"][:, ok] - x - f * dt) / np.abs(x).max(axis=0)).max() < 1e-9
    w = b["w"][:, ok]
    assert (np.abs(a["w"][:, ok] - w) / np.abs(w).max(axis=0) - 10 * np.abs(dt)).max() < 1e-9


@pytest.mark.parametrize("k", [1, 2, 3, 4])
@pytest.mark.parametrize("n", [1, 17, 400])
def test_adaptive_pipeline_matches_one_thread_form(k, n):
    kw = dict(escape_r2=4.0, sample_every=7)
    a, b = _run(n, 0, k, **kw), _run(n, PAD, k, **kw)
    _close(a, b)
    if n == 400:
        assert {chs.ORBIT_OK, chs.ORBIT_ESCAPED, chs.ORBIT_NONFINITE} <= set(a["status"].tolist())
        assert (a["rej"] > 0).any()


@pytest.mark.parametrize("kw", [dict(sample_every=1), dict(sample_every=0, renorm=False),
                                dict(sample_every=5, early_exit=True, sali_threshold=0.6),
                                dict(sample_every=4, dh_limit=3e-9), dict(sample_every=6, clock_budget=1),
                                dict(sample_every=10, h_max=0.11), dict(sample_every=10, tol=0.0)])
def test_adaptive_pipeline_checks_and_controls(kw):
    base = dict(escape_r2=4.0)
    base.update(kw)
    _close(_run(150, 0, 2, **dict(base)), _run(150, PAD, 2, **dict(base)))


@pytest.mark.parametrize("h0", [1e-310, 1e-160, 1e-12])
def test_adaptive_pipeline_tiny_first_step(h0):
    """Steps that start far below the state's rounding grow tenfold until the error estimate, then
    all rounding, limits them: step counts may differ, the results at t_final agree to the tolerance."""
    a, b = (_run(150, pad, 2, h0=h0, sample_every=10) for pad in (0, PAD))
    ok = (a["status"] == 0) & (b["status"] == 0) & (np.abs(b["x"]).max(axis=0) < 1.0)
    assert ok.sum() > 90
    assert (a["t"][ok] == 12.0).all() and (b["t"][ok] == 12.0).all()
    assert np.abs(a["x"][:, ok] - b["x"][:, ok]).max() < 1e-6


def test_adaptive_pipeline_resumes_exactly():
    one = _run(90, 0, 3, escape_r2=4.0, sample_every=7)
    many = _run(90, 0, 3, calls=40, escape_r2=4.0, sample_every=7)
    for f in one:
        np.testing.assert_array_equal(one[f], many[f], err_msg=f)

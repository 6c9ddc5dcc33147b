"""Plain launches on Henon-Heiles ensembles of up to 2^20 cells deal the orbits that run out to the
warps in dense groups; an explicit block size (RK4) and the work queue (DOP853) run thread t on orbit t.
Every orbit takes the same steps, so everything is the same bit for bit: for statuses that leave full,
ragged, empty and single-orbit groups, every way an orbit freezes, and runs split into calls."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2507_00622_gb300 import chs  # noqa: E402


def _statuses(n, kind):
    rng = np.random.default_rng(n)
    st = np.zeros(n, np.int32)
    if kind == "scattered":
        st[rng.random(n) < 0.25] = chs.ORBIT_FORBIDDEN
        st[rng.random(n) < 0.02] = chs.ORBIT_PREDICTED_REGULAR
    elif kind == "blocks":  # whole mask words and chunks without an orbit
        st[(np.arange(n) // 1500) % 3 == 1] = chs.ORBIT_FORBIDDEN
    elif kind == "last":
        st[:-1] = chs.ORBIT_FORBIDDEN
    elif kind == "none":
        st[:] = chs.ORBIT_FORBIDDEN
    return st


def _run(n, k, plain, steps, kind, integrator, splits=1, **kw):
    rng = np.random.default_rng(n + k)
    ics = rng.uniform(-0.35, 0.35, (4, n))
    ics[2:, ::5] *= 2.2  # some escape
    ics[0, n // 2] = np.nan
    S = chs.System(chs.HENON_HEILES, 2)
    dp = integrator == chs.DOP853
    dt = 0.1 if dp else 0.01
    ens = chs.DeviceEnsemble.empty(n, 4, k)
    ens.ld.zero_()
    abi = ens.abi(with_ld=kw.get("ld_p", 0.0) > 0)
    par = dict(n_dev=k, seed=3, integrator=integrator, **kw)
    if plain and not dp:
        par["block_threads"] = 128
    chs.chs_ensemble_init(S.h, chs.params(dt, 1, **par), abi, torch.from_numpy(ics).cuda(),
                          torch.from_numpy(_statuses(n, kind)).cuda())
    work = chs.compact_work(n)
    for i in range(splits):
        prm = chs.params(dt, steps // splits, step0=i * (steps // splits), **par)
        if plain and dp:
            chs.chs_integrate_persistent(S.h, prm, abi, work)
        else:
            chs.chs_integrate_batch(S.h, prm, abi)
    torch.cuda.synchronize()
    return {f: getattr(ens, f).cpu().numpy() for f in ("x", "w", "ld", "h0", "dh_max", "n_exec", "status")}


def _same(a, b):
    for f in a:
        np.testing.assert_array_equal(a[f], b[f], err_msg=f)


CASES = [(chs.RK4, 240), (chs.DOP853, 30)]


@pytest.mark.parametrize("integrator,steps", CASES)
@pytest.mark.parametrize("kind", ["all", "scattered", "blocks", "last", "none"])
@pytest.mark.parametrize("n", [14593, 70001, 131072, 131073])
def test_dense_groups_equal_plain_launch(integrator, steps, kind, n):
    kw = dict(ld_p=0.5, escape_r2=4.0, sample_every=20)
    a, b = (_run(n, 2, plain, steps, kind, integrator, **kw) for plain in (False, True))
    _same(a, b)
    if kind == "scattered":
        runs = _statuses(n, kind)[n // 2] == chs.ORBIT_OK  # the cell whose start is not finite
        assert {chs.ORBIT_OK, chs.ORBIT_ESCAPED} <= set(a["status"].tolist())
        assert (a["status"][n // 2] == chs.ORBIT_NONFINITE) == runs


@pytest.mark.parametrize("integrator,steps", CASES)
@pytest.mark.parametrize("k,kw", [(4, dict(ld_p=0.5, dh_limit=2e-11)), (3, dict(early_exit=True, sali_threshold=0.5)),
                                  (4, dict(clock_budget=1)), (2, dict(renorm=False)), (3, dict(ld_p=1.3))])
def test_dense_groups_health_checks_and_resume(integrator, steps, k, kw):
    kw = dict(dict(escape_r2=4.0, sample_every=10), **kw)
    a, b = (_run(30011, k, plain, steps, "scattered", integrator, **kw) for plain in (False, True))
    _same(a, b)
    if "clock_budget" not in kw:
        _same(a, _run(30011, k, False, steps, "scattered", integrator, splits=2, **kw))


@pytest.mark.parametrize("integrator,steps", [(chs.RK4, 100), (chs.DOP853, 10)])
@pytest.mark.parametrize("n,k", [(300001, 2), (1 << 20, 2), ((1 << 20) + 1, 2), (1 << 20, 4)])
def test_dense_groups_of_large_ensembles(integrator, steps, n, k):
    kw = dict(ld_p=0.5, escape_r2=4.0, sample_every=10)
    a, b = (_run(n, k, plain, steps, "scattered", integrator, **kw) for plain in (False, True))
    _same(a, b)

"""Small Henon-Heiles ensembles take fixed DOP853 steps as a pipeline of warps; larger ones one thread
per orbit.  Both compute every quantity by the same operations, so states, vectors, LD, counters and
statuses are the same bit for bit whether an ensemble runs alone or at the head of a larger one: for
every vector count, with and without the LD, ragged orbit counts, uneven end steps, every way an orbit
freezes, resumed runs and compacted lists."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2507_00622_gb300 import chs  # noqa: E402

PAD = 15000  # more orbits than the pipeline takes


def _ics(n, seed):
    """Bound orbits, some that escape (energies up to 0.4) and one that is not finite."""
    rng = np.random.default_rng(seed)
    ics = rng.uniform(-0.35, 0.35, (4, n))
    ics[2:, ::5] *= 2.2
    if n > 8:
        ics[0, 7] = np.nan
    return ics


def _run(n, k, steps, pad, launch="batch", splits=1, t_end=None, **kw):
    m = max(n, PAD) if pad else n
    ics = np.full((4, m), 0.1)
    ics[:, :n] = _ics(n, n + k)
    S = chs.System(chs.HENON_HEILES, 2)
    dt = kw.pop("dt", 0.1)
    ens = chs.DeviceEnsemble.empty(m, 4, k)
    ens.ld.zero_()
    te = None
    if t_end is not None:
        te = torch.full((m,), 10 ** 6, dtype=torch.int64)
        te[:n] = torch.from_numpy(t_end)
        te = te.cuda()
    abi = ens.abi(with_ld=kw.get("ld_p", 0.0) > 0, t_end=te)
    par = dict(n_dev=k, seed=3, integrator=chs.DOP853, **kw)
    chs.chs_ensemble_init(S.h, chs.params(dt, 1, **par), abi, torch.from_numpy(ics).cuda())
    if k:  # a padded ensemble draws the vectors of its own size: both start from the same ones
        w = np.random.default_rng(9).normal(size=(k, 4, PAD))[:, :, :m]
        w /= np.sqrt((w * w).sum(1, keepdims=True))
        ens.w.copy_(torch.from_numpy(np.ascontiguousarray(w)).reshape(ens.w.shape))
    work = chs.compact_work(m)
    for i in range(splits):
        prm = chs.params(dt, steps // splits, step0=i * (steps // splits), **par)
        if launch == "compacted":
            chs.chs_integrate_compacted(S.h, prm, abi, 23, work)
        elif launch == "persistent":
            chs.chs_integrate_persistent(S.h, prm, abi, work)
        else:
            chs.chs_integrate_batch(S.h, prm, abi)
    torch.cuda.synchronize()
    return {f: getattr(ens, f).cpu().numpy()[..., :n] for f in ("x", "w", "ld", "h0", "dh_max", "n_exec", "status")}


def _same(a, b):
    for f in a:
        np.testing.assert_array_equal(a[f], b[f], err_msg=f)


@pytest.mark.parametrize("k", [1, 2, 3, 4])
@pytest.mark.parametrize("ld_p", [0.0, 0.5, 1.3])
@pytest.mark.parametrize("n", [1, 33, 782])
def test_pipeline_equals_one_thread_form(k, ld_p, n):
    kw = dict(ld_p=ld_p, escape_r2=4.0, sample_every=25)
    a, b = (_run(n, k, 230, pad, **kw) for pad in (False, True))
    _same(a, b)
    if n > 100:
        assert {chs.ORBIT_OK, chs.ORBIT_ESCAPED, chs.ORBIT_NONFINITE} <= set(a["status"].tolist())


def test_pipeline_uneven_ends_resume_and_lists():
    n, k = 1500, 2
    t_end = np.random.default_rng(1).integers(-3, 300, n)
    kw = dict(t_end=t_end, ld_p=0.5, escape_r2=4.0, sample_every=30)
    a = _run(n, k, 240, True, **kw)
    _same(a, _run(n, k, 240, False, **kw))
    _same(a, _run(n, k, 240, False, splits=5, **kw))
    _same(a, _run(n, k, 240, False, launch="compacted", **kw))
    _same(a, _run(n, k, 240, False, launch="persistent", **kw))


@pytest.mark.parametrize("kw", [dict(sample_every=0), dict(sample_every=8, dh_limit=1e-9),
                                dict(sample_every=40, early_exit=True, sali_threshold=0.5),
                                dict(sample_every=20, clock_budget=1), dict(sample_every=20, renorm=False),
                                dict(sample_every=20, escape_r2=0.0), dict(sample_every=20, dt=-0.1)])
def test_pipeline_health_checks(kw):
    kw = dict(dict(ld_p=0.5, escape_r2=4.0), **kw)
    a, b = (_run(900, 3, 120, pad, **kw) for pad in (False, True))
    _same(a, b)


@pytest.mark.parametrize("k,ld", [(2, True), (4, True), (4, False)])
def test_pipeline_at_its_largest_size(k, ld):
    n = 152 * 32 * (2 if ld and k > 2 else 3)
    kw = dict(ld_p=0.5 if ld else 0.0, escape_r2=4.0, sample_every=10)
    a, b = (_run(n, k, 40, pad, **kw) for pad in (False, True))
    _same(a, b)

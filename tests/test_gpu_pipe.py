"""Small Henon-Heiles ensembles run as a pipeline of warps (one orbit's step spread over a block);
an explicit block size runs the one-thread-per-orbit form.  Both compute every quantity by the same
operations, so states, vectors, LD, counters and statuses are the same bit for bit: for every vector
count, with and without the LD, ragged orbit counts, uneven end steps, every way an orbit freezes,
resumed runs and compacted lists."""
import numpy as np
import pytest

from paper_2507_00622_gb300.inputs import uniform_vectors

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2507_00622_gb300 import chs  # noqa: E402


def _ics(n, seed):
    """Bound orbits, some that escape (energies up to 0.4) and one that is not finite."""
    rng = np.random.default_rng(seed)
    ics = rng.uniform(-0.35, 0.35, (4, n))
    ics[2:, ::5] *= 2.2
    if n > 8:
        ics[0, 7] = np.nan
    return torch.from_numpy(ics).cuda()


def _run(n, k, block, steps, launch="batch", splits=1, t_end=None, w_in=None, **kw):
    S = chs.System(chs.HENON_HEILES, 2)
    dt = kw.pop("dt", 0.01)
    ld = kw.get("ld_p", 0.0) > 0
    ens = chs.DeviceEnsemble.empty(n, 4, k)
    ens.ld.zero_()
    abi = ens.abi(with_ld=ld, t_end=t_end)
    par = dict(n_dev=k, seed=3, block_threads=block, **kw)
    chs.chs_ensemble_init(S.h, chs.params(dt, 1, **par), abi, _ics(n, n + k), None, w_in)
    work = chs.compact_work(n)
    for i in range(splits):
        prm = chs.params(dt, steps // splits, step0=i * (steps // splits), **par)
        if launch == "compacted":
            chs.chs_integrate_compacted(S.h, prm, abi, 23, work)
        elif launch == "persistent":
            chs.chs_integrate_persistent(S.h, prm, abi, work)
        else:
            chs.chs_integrate_batch(S.h, prm, abi)
    torch.cuda.synchronize()
    return {f: getattr(ens, f).cpu().numpy() for f in ("x", "w", "ld", "h0", "dh_max", "n_exec", "status")}


def _same(a, b):
    for f in a:
        np.testing.assert_array_equal(a[f], b[f], err_msg=f)


@pytest.mark.parametrize("k", [2, 3, 4])
@pytest.mark.parametrize("ld_p", [0.0, 0.5, 1.3])
@pytest.mark.parametrize("n", [1, 33, 782])
def test_pipeline_equals_one_thread_form(k, ld_p, n):
    kw = dict(ld_p=ld_p, escape_r2=4.0, sample_every=25)
    a, b = (_run(n, k, blk, 460, **kw) for blk in (0, 32))
    _same(a, b)
    if n > 100:
        assert {chs.ORBIT_OK, chs.ORBIT_ESCAPED, chs.ORBIT_NONFINITE} <= set(a["status"].tolist())


def test_pipeline_uneven_ends_resume_and_lists():
    n, k = 1500, 2
    t_end = torch.from_numpy(np.random.default_rng(1).integers(-3, 300, n)).cuda()
    kw = dict(ld_p=0.5, escape_r2=4.0, sample_every=30)
    a = _run(n, k, 64, 240, t_end=t_end, **kw)
    _same(a, _run(n, k, 0, 240, t_end=t_end, **kw))
    _same(a, _run(n, k, 0, 240, splits=5, t_end=t_end, **kw))
    _same(a, _run(n, k, 0, 240, launch="compacted", t_end=t_end, **kw))
    _same(a, _run(n, k, 0, 240, launch="persistent", t_end=t_end, **kw))


@pytest.mark.parametrize("kw", [dict(sample_every=0), dict(sample_every=16, dh_limit=2e-11),
                                dict(sample_every=40, early_exit=True, sali_threshold=0.5),
                                dict(sample_every=20, clock_budget=1), dict(sample_every=20, renorm=False),
                                dict(sample_every=20, escape_r2=0.0), dict(sample_every=20, dt=-0.01)])
def test_pipeline_health_checks(kw):
    base = dict(escape_r2=4.0, ld_p=0.5)
    base.update(kw)
    a, b = (_run(300, 3, blk, 330, **dict(base)) for blk in (0, 128))
    _same(a, b)


def test_pipeline_given_vectors():
    n, k = 97, 4
    w = torch.from_numpy(uniform_vectors(4, n, k, 4)).cuda()
    _same(_run(n, k, 0, 200, w_in=w, escape_r2=4.0), _run(n, k, 32, 200, w_in=w, escape_r2=4.0))


@pytest.mark.parametrize("n", [1, 33, 4864, 4865, 7001, 14593, 18432, 18433])
@pytest.mark.parametrize("status", ["none", "some", "few", "no orbit", "in place"])
def test_lyapunov_pipeline_equals_one_thread_form(n, status):
    ics = _ics(n, 3 * n)
    rng = np.random.default_rng(n)
    st = rng.choice([chs.ORBIT_OK, chs.ORBIT_FORBIDDEN, chs.ORBIT_ESCAPED], n, p=[0.75, 0.2, 0.05]).astype(np.int32)
    if status == "few":
        st[n // 50:] = chs.ORBIT_FORBIDDEN
    elif status == "no orbit":
        st[:] = chs.ORBIT_FORBIDDEN
    S = chs.System(chs.HENON_HEILES, 2)
    out = []
    for block in (0, 32):
        ic = None if status == "none" else torch.from_numpy(st.copy()).cuda()
        lam = torch.full((4, n), 7.0, dtype=torch.float64, device="cuda")
        so = ic if status == "in place" else torch.full((n,), 77, dtype=torch.int32, device="cuda")
        chs.chs_lyapunov_spectrum(S.h, chs.params(0.01, 47, qr_every=7, sample_every=20, block_threads=block), n, ics, ic,
                                  lam, so)
        torch.cuda.synchronize()
        out.append((lam.cpu().numpy(), so.cpu().numpy()))
    np.testing.assert_array_equal(out[0][0], out[1][0])
    np.testing.assert_array_equal(out[0][1], out[1][1])

"""The surrogate's forward pass sums every output as the FP32 chain acc = fma(w_k, a_k, acc),
k ascending, plus the bias, whatever unit computes it: activations and outputs equal the chain's
bit for bit, for the tile sizes of the kernel (16- and 32-sample tiles, one warp to many blocks),
for freshly drawn and for trained weights, and for inputs that are huge or not finite."""
import numpy as np
import pytest

from paper_2507_00622_gb300.inputs import mlp_init

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2507_00622_gb300 import chs  # noqa: E402
from paper_2507_00622_gb300.surrogate import Surrogate  # noqa: E402


def _bf16(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to(torch.bfloat16).float().numpy()


def _chain(W, b, a):
    """[u][n] FP32: one rounding per multiply-add (the product of two BF16 values, or of a BF16 and an
    FP32 one, is exact in FP64)."""
    acc = np.zeros((W.shape[0], a.shape[1]), dtype=np.float32)
    for k in range(W.shape[1]):
        acc = (acc.astype(np.float64) + W[:, k:k + 1].astype(np.float64) * a[k].astype(np.float64)).astype(np.float32)
    return (acc + b[:, None]).astype(np.float32)


def _forward(p, X):
    acts, a, o = [], X, 0
    for u, k in ((128, 12), (128, 128), (128, 128), (2, 128)):
        v = _chain(p[o:o + u * k].reshape(u, k), p[o + u * k:o + u * k + u], a)
        o += u * k + u
        if u == 2:
            return v, np.stack(acts)
        a = _bf16(np.fmax(v, np.float32(0)))
        acts.append(a)


def _params(which):
    if which == "trained":
        pb = Surrogate.load().params
        return pb.float().cpu().numpy(), pb
    p = _bf16(mlp_init(5) + 0.05 * np.random.default_rng(6).standard_normal(34946))
    return p, torch.from_numpy(p).to(torch.bfloat16).cuda()


@pytest.mark.parametrize("which", ["drawn", "trained"])
@pytest.mark.parametrize("n", [1, 15, 16, 33, 6100])
def test_forward_equals_the_fp32_chain(which, n):
    p, pb = _params(which)
    rng = np.random.default_rng(n)
    X = rng.standard_normal((12, n)).astype(np.float32)
    if n > 100:
        X[3, 5], X[4, 6], X[7, 7] = np.inf, -np.inf, np.nan
        X[:, 8] *= np.float32(3e18)  # squares beyond FP32
        X[:, 9] = 0
    Y = torch.empty((2, n), dtype=torch.float32, device="cuda")
    act = torch.empty((3, 128, n), dtype=torch.bfloat16, device="cuda")
    chs.chs_mlp_forward(pb, torch.from_numpy(X).cuda(), n, Y, act)
    Y2 = torch.empty_like(Y)
    chs.chs_mlp_forward(pb, torch.from_numpy(X).cuda(), n, Y2)
    torch.cuda.synchronize()
    with np.errstate(all="ignore"):
        Yr, acts = _forward(p, X)
    np.testing.assert_array_equal(act.float().cpu().numpy(), acts)
    np.testing.assert_array_equal(Y.cpu().numpy(), Yr)
    np.testing.assert_array_equal(Y2.cpu().numpy(), Yr)

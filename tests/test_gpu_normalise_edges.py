"""The normaliser bit for bit against NumPy in FP64: block lengths around its
register tiles (1 .. 4096 bins, short last blocks, few and many blocks), powers
that tie in FP32, powers beyond FP32, zeros, infinities and values that are not
numbers, in place and out of place."""
import numpy as np
import pytest

from parity import lib_ready

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return lib_ready()


def want(F, B):
    out = np.empty_like(F)
    re, im = F.real.astype(np.float64), F.imag.astype(np.float64)
    p = re * re + im * im
    for s in range(0, F.size, B):
        q = np.sort(p[s:s + B])                          # NaN last
        med = q[(q.size - 1) // 2]
        scale = 1.0 / np.sqrt(med / 0.69314718055994530942) if med > 0.0 else 1.0
        out.real[s:s + B] = (re[s:s + B] * scale).astype(np.float32)
        out.imag[s:s + B] = (im[s:s + B] * scale).astype(np.float32)
    return out


def make(kind, n, rng):
    F = ((rng.standard_normal(n) + 1j * rng.standard_normal(n)) * 37.0).astype(np.complex64)
    if kind == "ties":
        # moduli a few FP64 units apart that round to one FP32 power
        F.real[:] = np.float32(3.0)
        F.imag[:] = (2.0 ** -rng.integers(8, 20, n)).astype(np.float32)
    elif kind == "equal":
        F[:] = np.complex64(1.5 - 0.25j)
    elif kind == "zeros":
        F[rng.random(n) < 0.7] = 0
    elif kind == "large":
        F *= np.float32(1e17)
    elif kind == "tiny":
        F *= np.float32(1e-22)
    elif kind == "mixed":
        F *= (10.0 ** rng.uniform(-18, 18, n)).astype(np.float32)
    elif kind == "odd":
        F[rng.random(n) < 0.2] = np.complex64(complex(np.inf, 1.0))
        F[rng.random(n) < 0.1] = np.complex64(complex(np.nan, 1.0))
    return F


@pytest.mark.parametrize("B,n", [(1, 70), (7, 100), (64, 1000), (256, 1025), (257, 2000), (1000, 2500), (1024, 3000),
                                 (1024, 1024 * 1300 + 5), (1025, 5000), (4096, 9000)])
def test_block_lengths(pkg, B, n):
    rng = np.random.default_rng(B + n)
    F = make("noise", n, rng)
    check(pkg, F, B)


@pytest.mark.parametrize("kind", ["ties", "equal", "zeros", "large", "tiny", "mixed", "odd"])
@pytest.mark.parametrize("B", [100, 1024, 2000])
def test_values(pkg, kind, B):
    check(pkg, make(kind, 6001, np.random.default_rng(len(kind) + B)), B)


def check(pkg, F, B):
    p = pkg.make_params(2, 2, 0, 20, max_bins=64, norm_block=B)
    with np.errstate(all="ignore"):
        ref = want(F, B)
    with pkg.Plan(p, build_templates=False) as plan:
        x = torch.from_numpy(F).cuda()
        y = torch.empty_like(x)
        plan.normalise(x, y)
        plan.normalise(x, x)                             # in place
        torch.cuda.synchronize()
    for got in (x, y):
        g = got.cpu().numpy()
        for a, b in ((g.real, ref.real), (g.imag, ref.imag)):
            assert np.array_equal(a, b, equal_nan=True)

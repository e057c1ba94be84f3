"""The test that leaves a line out of a velocity sample (k_solve_impl.cuh,
line_is_far), restated in NumPy float32: when it says so, every bin of the warp
gets fma(chi0, g, chi) = chi and fma(eta0, g, eta) = eta bit for bit, for any
chi >= chi_c and eta >= eta_c that the other lines left, with g at the upper end
of ex2.approx's error.  With the threshold 10 % lower it leaves out lines that
change the sum.  CPU only."""
import numpy as np

f32 = np.float32
ARG_SCALE = 1.2011224087864498
KC = 299792.458
E_EX2 = 2.0 ** -20


def fma(a, b, c):
    return (np.float64(a) * np.float64(b) + np.float64(c)).astype(f32)


def bins(rng, n_freq, lines, ratio_step):
    """A and B of line 0 at the bins of every line (profile constants, prescaled)."""
    x = np.linspace(-4.0, 4.0, n_freq) if n_freq > 1 else np.zeros(1)
    ub = x * rng.uniform(0.2, 3.0)
    A, B = [], []
    for l in range(lines):
        r = 1.0 + ratio_step * l
        A.append((KC * (r - 1.0) + r * ub) * ARG_SCALE)
        B.append(r * (1.0 + ub / KC) * ARG_SCALE)
    return np.concatenate(A).astype(f32), np.concatenate(B).astype(f32)


def is_far(dl, rdv, cc, ec, c0, e0, A, B, scale=1.0):
    if c0 == 0 and e0 == 0:
        return True
    lo = f32(fma(B.min() if dl >= 0 else B.max(), dl, A.min()) * rdv)
    hi = f32(fma(B.max() if dl >= 0 else B.min(), dl, A.max()) * rdv)
    with np.errstate(divide="ignore"):
        re = f32(e0 / ec) if e0 > 0 else f32(0)
    x = max(f32(c0 / cc), re, f32(1e-30))
    t = min(f32(f32(np.sqrt(max(f32(25.05) + np.log2(x), f32(0)))) * f32(1.0001)), f32(12.1)) * f32(scale)
    return lo >= t or hi <= -t


def unchanged(dl, rdv, cc, ec, c0, e0, A, B, rng):
    a = (fma(B, dl, A) * rdv).astype(f32)
    q = (a * a).astype(f32).astype(np.float64)
    g = np.where(q >= 128.0, 0.0, np.exp2(-q) * (1.0 + E_EX2)).astype(f32)  # ftz flushes the subnormals
    for base in (0.0, rng.uniform(0, 3) * float(cc)):
        chi, eta = f32(float(cc) + base), f32(float(ec) * (1.0 + base / float(cc)))
        if not (np.all(fma(c0, g, chi) == chi) and np.all(fma(e0, g, eta) == eta)):
            return False
    return True


def cases(rng, n):
    for _ in range(n):
        lines = int(rng.integers(1, 4))
        A, B = bins(rng, int(rng.integers(1, 40)), lines, rng.choice([1e-3, 1e-5]))
        rdv = f32(1.0 / rng.uniform(0.1, 3.0))
        cc = f32(10.0 ** rng.uniform(-12, 0))
        c0 = f32(0.0 if rng.uniform() < 0.05 else 10.0 ** rng.uniform(-6, 3))
        S = 10.0 ** rng.uniform(-2, 2)
        ec = f32(0.0 if rng.uniform() < 0.1 else float(cc) * S)
        e0 = f32(0.0 if rng.uniform() < 0.1 else float(c0) * 10.0 ** rng.uniform(-2, 2))
        with np.errstate(divide="ignore", invalid="ignore"):
            need = 25.05 + np.log2(max(float(c0) / float(cc), float(e0) / float(ec) if ec > 0 else 1e30, 1e-30))
        t = min(np.sqrt(max(need, 0.0)), 12.1)
        end = A.argmax() if rng.uniform() < 0.5 else A.argmin()  # the nearest bin close to the threshold
        sign = 1.0 if end == A.argmin() else -1.0
        dl = f32((sign * t * (1.0 + rng.uniform(-3e-2, 3e-2)) / float(rdv) - float(A[end])) / float(B[end]))
        yield dl, rdv, cc, ec, c0, e0, A, B


def test_a_line_left_out_changes_no_bin():
    rng = np.random.default_rng(5)
    out = 0
    for c in cases(rng, 6000):
        if is_far(*c):
            out += 1
            assert unchanged(*c, rng)
    assert out > 1500


def test_a_lower_threshold_goes_wrong():
    rng = np.random.default_rng(6)
    bad = sum(1 for c in cases(rng, 3000) if is_far(*c, scale=0.9) and not unchanged(*c, rng))
    assert bad > 10

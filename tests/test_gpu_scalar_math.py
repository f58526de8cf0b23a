"""The scalar FP64 arithmetic of the solvers' serial chains against exact values.

Every input is chosen so that the quantity is reached exactly up to the one
operation under test, and every bound counts the roundings of that operation
(u = 2^-53 relative each).
"""
from decimal import Decimal, getcontext
from fractions import Fraction as F

import numpy as np
import pytest

import workloads as W
from tests._gpu import ensure_built, torch_cuda

pytestmark = pytest.mark.gpu

getcontext().prec = 60


@pytest.fixture(scope="module")
def env():
    torch = torch_cuda()
    ed = ensure_built()
    ctx = ed.ed_ctx_create(0)
    yield ed, ctx, torch
    ed.ed_ctx_destroy(ctx)


@pytest.mark.parametrize("power", [-36, 0, 70])   # 70: the sum of squares leaves a float's range
@pytest.mark.parametrize("reorth", [True, False])
def test_first_beta_is_rounded_once(env, reorth, power):
    """One step from a basis state of a star of one electron: H v - alpha v is the
    row of hops, whose squares add up exactly, so beta_1 (the residual after one
    step) is the square root rounded once: u."""
    ed, ctx, torch = env
    r = np.random.default_rng(11)
    n, worst = 24, 0.0
    for _ in range(20):
        T = np.zeros((n, n))
        h = r.integers(1, 2000, n - 1) / 64.0 * 2.0 ** power
        T[0, 1:] = T[1:, 0] = h
        T[0, 0] = 0.5 * 2.0 ** power
        sec = ed.ed_sector_create(ctx, W.Model(n, T, np.zeros(n)), 1, 0, "fp64")
        try:
            v0 = torch.zeros(n, dtype=torch.float64, device="cuda")
            v0[0] = 1.0
            _, info, _ = ed.ed_lanczos(sec, k=1, tol=1e-300, max_iter=1, check_every=1, v0=v0, reorth=reorth,
                                       allow_not_converged=True)
        finally:
            ed.ed_sector_destroy(sec)
        v = sum(F(float(x)) ** 2 for x in h)
        root = (Decimal(v.numerator) / Decimal(v.denominator)).sqrt()
        worst = max(worst, float(abs(Decimal(info.residual[0]) / root - 1) * 2 ** 53))
    assert worst <= 1.0 + 1e-9, worst


@pytest.mark.parametrize("scale", [1.0, 1e-25, 1e25, 1e160])   # inside and outside the squares' float range
def test_one_level_fraction(env, scale):
    """G of one empty site of energy zero is 1 / z, one reciprocal c - i d over q =
    c^2 + d^2: u/2 of q from the smaller square, u from the sum, u from the
    quotient; and over many z no less accurate than Smith's division."""
    ed, ctx, torch = env
    r = np.random.default_rng(12)
    n = 4096
    z = (r.standard_normal(n) + 1j * np.abs(r.standard_normal(n)) * 10.0 ** r.uniform(-2, 2, n)) * scale
    psi = torch.ones(1, dtype=torch.float64, device="cuda")
    G = ed.ed_greens_cf_z(ctx, W.Model(1, np.zeros((1, 1)), np.zeros(1)), "fp64", [(0, 0, 0.0, psi)], z, 1.0, depth=1)
    c, d = z.real, z.imag
    big = np.abs(c) >= d
    with np.errstate(over="ignore"):
        t = np.where(big, d / c, c / d)
        den = np.where(big, c + d * t, c * t + d)
        smith = np.where(big, 1 / den, t / den) - 1j * np.where(big, t / den, 1 / den)
    err = {"G": [], "smith": []}
    for i in range(n):
        cf, df = F(float(c[i])), F(float(d[i]))
        q = cf * cf + df * df
        for name, g in (("G", G[i]), ("smith", smith[i])):
            err[name] += [float(abs(F(float(g.real)) * q / cf - 1) * 2 ** 53), float(abs(F(float(g.imag)) * q / -df - 1) * 2 ** 53)]
    rms = {k: float(np.sqrt(np.mean(np.square(v)))) for k, v in err.items()}
    if scale == 1.0:
        assert max(err["G"]) <= 2.5 + 1e-9, max(err["G"])
    assert rms["G"] <= 1.02 * rms["smith"], rms   # 2%: four times the spread of a mean over 8,192 roundings


HARNESS = r"""
#include "lanczos_kernels.h"
using namespace ed;
namespace ed { void set_error(const char*, ...) {}
int dev_alloc(Ctx*, void**, size_t) { return 1; }
void dev_free(Ctx*, void*, size_t) {}
int apply_fast(const Sector*, const void*, void*, cudaStream_t, double*, int*) { return 1; }
int apply_h(const Sector*, const void*, void*, cudaStream_t) { return 1; } }
template <class V>
__global__ void k_macs(const V* x, const V* y, int n, int terms, float2* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float2 d = make_float2(0.f, 0.f), h = d;
  for (int k = 0; k < terms; ++k) {
    const V a = x[(size_t)k * n + i], b = y[(size_t)k * n + i];
    dmac(d, a, b);
    hmac(h, acc_of(a), b);
  }
  out[i] = d;
  out[n + i] = h;
}
__global__ void k_vecs(const double* a, const double* b, int m, double* theta, double* S, double* work) {
  extern __shared__ __align__(16) double sh[];
  const size_t j = blockIdx.x;
  tri_pair_one(a + j * m, b + j * m, m, 0, theta + j, S + j * m, m, work, sh);
}
extern "C" int run_macs(int floats, const void* x, const void* y, int n, int terms, void* out) {
  if (floats) k_macs<float><<<(n + 255) / 256, 256>>>((const float*)x, (const float*)y, n, terms, (float2*)out);
  else k_macs<float2><<<(n + 255) / 256, 256>>>((const float2*)x, (const float2*)y, n, terms, (float2*)out);
  return (int)cudaDeviceSynchronize();
}
extern "C" int run_vecs(const double* a, const double* b, int n, int m, double* theta, double* S) {
  k_vecs<<<n, 32, tri_smem(m)>>>(a, b, m, theta, S, nullptr);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def harness(env, tmp_path_factory):
    """The internal headers' device functions behind kernels of their own."""
    import ctypes
    import subprocess
    from paper_1004_3354_gb300 import _build
    d = tmp_path_factory.mktemp("harness")
    (d / "h.cu").write_text(HARNESS)
    subprocess.run([_build._nvcc(), *_build.ARCH, *_build.FLAGS, "-I", _build.CSRC, "-shared", "-o", str(d / "h.so"),
                    str(d / "h.cu")], check=True)
    return ctypes.CDLL(str(d / "h.so"))


def _two_sum(a, b):
    s = a + b
    bb = s - a
    return s, (a - (s - bb)) + (b - bb)


def _fma32(a, b, c):
    return (a.astype(np.longdouble) * b.astype(np.longdouble) + c.astype(np.longdouble)).astype(np.float32)


@pytest.mark.parametrize("vectors", ["df64", "fp32"])
@pytest.mark.parametrize("what", ["dot", "norm"])
def test_double_float_sums_carry_both_errors(env, harness, what, vectors):
    """Dot products and projections add the error of the product (fused
    multiply-add), the cross terms and the error of the sum (TwoSum), each formed on
    its own: over 200,000 sums of ten products the error against extended
    precision is that of those steps, to 1% (three times the spread of the ratio)."""
    import ctypes as C
    ed, ctx, torch = env
    n, terms = 200000, 10
    r = np.random.default_rng(13)
    X = r.standard_normal((terms, n))
    Y = X if what == "norm" else r.standard_normal((terms, n))

    def split(v):
        hi = v.astype(np.float32)
        lo = (v - hi).astype(np.float32) if vectors == "df64" else np.zeros_like(hi)
        return hi, lo
    (xh, xl), (yh, yl) = split(X), split(Y)
    hi, lo = np.zeros(n, np.float32), np.zeros(n, np.float32)
    for k in range(terms):
        p = xh[k] * yh[k]
        e = _fma32(xh[k], yh[k], -p)
        e = _fma32(xh[k], yl[k], e)
        e = _fma32(xl[k], yh[k], e)
        hi, t = _two_sum(hi, p)
        lo = lo + (t + e)
    L = np.longdouble
    exact = sum((xh[k].astype(L) + xl[k]) * (yh[k].astype(L) + yl[k]) for k in range(terms))
    rms = lambda h, l: float(np.sqrt(np.mean(((h.astype(L) + l - exact) ** 2).astype(np.float64))))
    dev = lambda h, l: torch.from_numpy(np.ascontiguousarray(h if vectors == "fp32" else np.stack([h, l], -1))).cuda()
    xd, yd, out = dev(xh, xl), dev(yh, yl), torch.empty(2 * n, 2, device="cuda")
    assert harness.run_macs(C.c_int(vectors == "fp32"), C.c_void_p(xd.data_ptr()), C.c_void_p(yd.data_ptr()), n, terms,
                            C.c_void_p(out.data_ptr())) == 0
    o = out.cpu().numpy().reshape(2, n, 2)
    want = rms(hi, lo)
    for got in o:
        assert rms(got[:, 0], got[:, 1]) <= 1.01 * want, (rms(got[:, 0], got[:, 1]), want)


def test_tridiagonal_vectors_divide_like_a_division(env, harness):
    """Vectors of 20,000 tridiagonal matrices of 50 rows by inverse iteration: the
    residual (against the vector's own Rayleigh quotient, in extended precision)
    is that of the same elimination and substitution with plain divisions, to
    1.5% in the median (more than twice the spread of the ratio)."""
    import ctypes as C
    ed, ctx, torch = env
    N, m = 20000, 50
    r = np.random.default_rng(14)
    a = r.uniform(-6, 6, (N, m))
    b = np.abs(r.normal(4, 1.5, (N, m)))
    b[:, 0] = 0.0
    ad, bd = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
    th, S = torch.empty(N, dtype=torch.float64, device="cuda"), torch.empty(N, m, dtype=torch.float64, device="cuda")
    assert harness.run_vecs(C.c_void_p(ad.data_ptr()), C.c_void_p(bd.data_ptr()), N, m, C.c_void_p(th.data_ptr()),
                            C.c_void_p(S.data_ptr())) == 0
    L = np.longdouble
    fma = lambda x, y, z: (x.astype(L) * y.astype(L) + z.astype(L)).astype(np.float64)
    A, B, t0 = a.T, b.T, th.cpu().numpy()
    # elimination with row interchanges, then three solves
    R, DL, DU, DU2, P = [], [], [], [], []
    d, u = A[0] - t0, B[1]
    for i in range(m - 1):
        sub, nd, nu = B[i + 1], A[i + 1] - t0, B[i + 2] if i + 2 < m else np.zeros(N)
        keep = np.abs(d) >= np.abs(sub)
        f = np.where(keep, sub, d) / np.where(keep, d, sub)
        R.append(np.where(keep, d, sub)), DL.append(f), DU.append(np.where(keep, u, nd)), DU2.append(np.where(keep, 0, nu))
        P.append(~keep)
        d, u = np.where(keep, fma(-f, u, nd), fma(-f, nd, u)), np.where(keep, nu, -f * nu)
    R.append(d)
    tiny = 2.2e-16 * np.max(np.abs(A) + np.abs(B) + np.vstack([B[1:], np.zeros((1, N))]), axis=0)
    R = [np.where(np.abs(x) < tiny, np.where(x < 0, -tiny, tiny), x) for x in R]
    x = [np.full(N, 1.0 + 0.01 * ((i * 7919) % 97) / 97.0) for i in range(m)]
    for _ in range(3):
        t = x[0]
        for i in range(m - 1):
            x[i], t = np.where(P[i], x[i + 1], t), fma(-DL[i], np.where(P[i], x[i + 1], t), np.where(P[i], t, x[i + 1]))
        x1, x2 = t / R[m - 1], np.zeros(N)
        x[m - 1] = x1
        for i in range(m - 2, -1, -1):
            x[i] = fma(-DU[i], x1, fma(-DU2[i], x2, x[i])) / R[i]
            x1, x2 = x[i], x1
        X = np.array(x)
        X = X / np.max(np.abs(X), axis=0)
        x = list(X / np.sqrt((X * X).sum(0)))

    def residual(X):
        X = X.astype(L)
        TX = A * X
        TX[1:] += B[1:] * X[:-1]
        TX[:-1] += B[1:] * X[1:]
        rho = (X * TX).sum(0) / (X * X).sum(0)
        return float(np.median(np.sqrt(((TX - rho * X) ** 2).sum(0)).astype(np.float64)))
    got, want = residual(S.cpu().numpy().T), residual(np.array(x))
    assert got <= 1.015 * want, (got, want)

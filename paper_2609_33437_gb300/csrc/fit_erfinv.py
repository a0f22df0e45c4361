"""Fit the polynomial coefficients of the device erfinv used by the Gaussian
Perturb transform (smat_device.cuh: coef_p, coef_q, used by erfinv_ratio and
erfinv_central2).

Method (structure of M. Giles, "Approximating the erfinv function", GPU
Computing Gems Jade Edition, 2011; coefficients fitted here): for
x in (-1, 1) let a = |x|, t = 1 - a^2 and L = log2(t) <= 0.
  central  (L >= L0):  erfinv(x) = x * P(L)        P a polynomial in L
  tail     (L <  L0):  erfinv(x) = x * Q(s - S_MID),  s = sqrt(-L)
The device evaluates t with one fused multiply-add, L with the hardware's
approximate log2 and P, Q by Horner's rule in fp32.

P is fitted to the hardware's own log2 of every input sym(u) can produce, so
that the approximation's bias does not add to the polynomial's error: relative
least squares, 60% of the weight uniform over the inputs and 40% uniform over L,
the coefficients rounded to fp32 one at a time from the highest power, the rest
fitted again after each. Q is fitted at Chebyshev nodes of s in [sqrt(-L0),
sqrt(23)] (the smallest t of an input is 2^-23) with high-precision targets
(mpmath). Both in a variable scaled to magnitude 1 (unscaled, the high powers
spoil the conditioning).

Run: python fit_erfinv.py --dump FILE   (on the GPU: writes the hardware's log2)
     python fit_erfinv.py FILE          (prints the coefficients and the errors of
                                         the fp32 evaluation over every input)
"""

import os
import subprocess
import sys
import tempfile

import mpmath as mp
import numpy as np

mp.mp.dps = 40
L0 = -10.0         # central / tail boundary in log2(1 - x^2)
DEG_P = 10
DEG_Q = 7
S_MAX = float(mp.sqrt(23.0)) + 1e-3
S_MID = 4.0        # tail Horner variable s - S_MID (exact in fp32), |s - S_MID| <= 1
OVER_L = 0.4       # share of the weight that is uniform over L

DUMP = r"""
#include <cstdint>
#include <cstdio>
#include <vector>
__global__ void log2_of(float* out) {  // input k = 2^23 + i, as the forward evaluates it
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  const float x = __fmaf_rn(__uint2float_rn((1u << 23) + i), 1.1920928955078125e-07f, -0.999999940395355224609375f);
  const float t = -__fmaf_rn(x, x, -1.0f);
  float L;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(L) : "f"(t));
  out[i] = L;
}
int main(int, char** argv) {
  const int n = 1 << 23;
  float* d = nullptr;
  if (cudaMalloc(&d, n * sizeof(float)) != cudaSuccess) return 1;
  log2_of<<<n / 256, 256>>>(d);
  std::vector<float> h(n);
  if (cudaMemcpy(h.data(), d, n * sizeof(float), cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
  FILE* f = fopen(argv[1], "wb");
  return f && fwrite(h.data(), sizeof(float), n, f) == (size_t)n && fclose(f) == 0 ? 0 : 1;
}
"""


def dump(path):
    with tempfile.TemporaryDirectory() as d:
        src, exe = os.path.join(d, "log2.cu"), os.path.join(d, "log2")
        with open(src, "w") as f:
            f.write(DUMP)
        subprocess.run(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-o", exe, src], check=True)
        subprocess.run([exe, path], check=True)


def f_tail(s):
    L = -mp.mpf(s) ** 2
    x = mp.sqrt(1 - mp.power(2, L))
    return mp.erfinv(x) / x


def fit_tail(lo, hi, deg, shift, n=400):
    """Relative-error fit at Chebyshev nodes (increasing powers)."""
    k = np.arange(n)
    nodes = 0.5 * (lo + hi) + 0.5 * (hi - lo) * np.cos(np.pi * (k + 0.5) / n)
    y = np.array([float(f_tail(v)) for v in nodes])
    scale = max(abs(lo - shift), abs(hi - shift))
    V = np.vander((nodes - shift) / scale, deg + 1, increasing=True) / y[:, None]
    c, *_ = np.linalg.lstsq(V, np.ones_like(y), rcond=None)
    w = np.ones_like(y)  # a few Lawson-style reweightings toward minimax
    for _ in range(40):
        r = V @ c - 1.0
        w = w * (np.abs(r) + 1e-30) ** 0.5
        w /= w.max()
        c, *_ = np.linalg.lstsq(V * w[:, None], w, rcond=None)
    return c / scale ** np.arange(deg + 1)


def fit_central(L, ratio):
    """fp32 coefficients of P (increasing powers) for the inputs' (L, erfinv(x) / x)."""
    at = np.arange(0, len(L), 16)
    at = np.concatenate([at, np.arange(max(0, len(L) - 60000), len(L))])
    v, y = L[at].astype(np.float64), ratio[at]
    count, edge = np.histogram(v, 64)
    share = len(v) / 64 / np.maximum(count[np.clip(np.searchsorted(edge, v) - 1, 0, 63)], 1)
    w = np.sqrt((1 - OVER_L) + OVER_L * share)
    fixed = {}
    for d in range(DEG_P, -1, -1):
        free = [k for k in range(DEG_P + 1) if k not in fixed]
        base = sum((c * v**k for k, c in fixed.items()), np.zeros(len(v)))
        V = np.stack([(v / -L0) ** k for k in free], 1) / y[:, None] * w[:, None]
        c, *_ = np.linalg.lstsq(V, (1 - base / y) * w, rcond=None)
        fixed[d] = float(np.float32(c[free.index(d)] / (-L0) ** d))
    return np.array([fixed[d] for d in range(DEG_P + 1)], np.float32)


def horner_f32(c, v):
    """fp32 Horner with fused multiply-adds (each step one rounding)."""
    v = np.asarray(v, np.float64)
    cc = np.asarray(c, np.float32).astype(np.float64)
    acc = np.full_like(v, cc[-1])
    for coef in cc[-2::-1]:
        acc = (acc * v + coef).astype(np.float32).astype(np.float64)
    return acc


def main(path):
    from scipy.special import erfinv

    L = np.fromfile(path, dtype=np.float32)  # of inputs sym(k), k = 2^23 .. 2^24 - 1 (x > 0)
    k = np.arange(1 << 23, 1 << 24, dtype=np.int64)
    x = (2 * k + 1 - (1 << 24)) * 2.0**-24
    ratio = erfinv(x) / x
    central = L >= np.float32(L0)
    cP = fit_central(L[central], ratio[central])
    cQ = np.float32(fit_tail(float(mp.sqrt(-L0)), S_MAX, DEG_Q, S_MID))
    print("// P(L), L in [%g, 0], increasing powers" % L0)
    print("{" + ", ".join("%.9ef" % v for v in cP) + "}")
    print("// Q(s - %g), s = sqrt(-L) in [%g, %g], increasing powers" % (S_MID, float(mp.sqrt(-L0)), S_MAX))
    print("{" + ", ".join("%.9ef" % v for v in cQ) + "}")
    p = np.empty(len(L))
    p[central] = horner_f32(cP, L[central])
    s = np.sqrt(-L[~central].astype(np.float64)).astype(np.float32)
    p[~central] = horner_f32(cQ, (s - np.float32(S_MID)).astype(np.float32))
    unit = (p * x).astype(np.float32).astype(np.float64)
    scale = float(np.float32(np.sqrt(2.0)))  # the forward's (scale p) x at sigma 1
    eps = ((scale * p).astype(np.float32).astype(np.float64) * x).astype(np.float32).astype(np.float64)
    for name, got, want in (("ratio", p, ratio), ("erfinv", unit, ratio * x), ("eps at sigma 1", eps, np.sqrt(2.0) * ratio * x)):
        r = np.abs(got / want - 1)
        print("%s: relative error at most %.4g, root mean square %.4g" % (name, r.max(), np.sqrt(np.mean(r**2))))
    print("tail fraction %.4g, monotone %s" % ((~central).mean(), bool(np.all(np.diff(unit) >= 0))))


if __name__ == "__main__":
    if sys.argv[1] == "--dump":
        dump(sys.argv[2])
    else:
        main(sys.argv[1])

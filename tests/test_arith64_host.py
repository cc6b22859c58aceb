"""The FP64 kernels' arithmetic on the integer pipes (arith64.cuh), compiled
as host C++, against plain FP64 operations, bit for bit:
  - soft_mul over the exponents its callers admit, with dense significands,
    significands of a few bits and products exactly halfway between two
    doubles;
  - the sums with a small correction and the exact r - 2;
  - whole Cash-Karp and Dormand-Prince attempts, Kerr and the q-metric, with
    ArithFast against the same attempt with ArithPlain: equal wherever
    ArithFast does not give the attempt back, which it does not for ordinary
    rays (the spin, L, p_theta or the whole right-hand side of p_theta' zero
    among them) and does for values outside its window, zeros, infinities and
    NaN where a product would meet them."""
import subprocess

import numpy as np
import pytest

from _df_host import build

HARNESS = r"""
#include "trace_device.cuh"
using namespace osiris_impl;
template <class Met, bool kSums>
static void attempt(const double* in, double* out) {
  RayK K;
  K.a = in[2];
  K.a2 = K.a * K.a;
  K.q = in[3];
  K.kap = K.q * (2.0 + K.q);
  K.E = in[4];
  K.L = in[5];
  K.aE = K.a * K.E;
  K.aL = K.a * K.L;
  K.E2 = K.E + K.E;
  State y;
  y.r = in[6];
  y.th = in[7];
  y.ph = 0.25;
  y.pr = in[8];
  y.pth = in[9];
  const double h = in[10];
  State o[2], d[2];
  Deriv k1[2] = {}, k7[2] = {};
  double twoH[2];
  ArithFast<kSums> fast(1.0, -0.0);
  if (in[1] == 0.0) {
    ck_step64<Met>(K, y, h, o[0], d[0], twoH[0], fast);
    ck_step64<Met>(K, y, h, o[1], d[1], twoH[1]);
  } else {
    dp_step64<Met>(K, y, h, false, k1[0], o[0], d[0], k7[0], fast);
    dp_step64<Met>(K, y, h, false, k1[1], o[1], d[1], k7[1]);
    twoH[0] = k1[0].twoH + k7[0].twoH;
    twoH[1] = k1[1].twoH + k7[1].twoH;
  }
  for (int i = 0; i < 2; ++i) {
    const double v[11] = {o[i].r, o[i].th, o[i].ph, o[i].pr, o[i].pth, d[i].r,
                          d[i].th, d[i].ph, d[i].pr, d[i].pth, twoH[i]};
    std::memcpy(out + 11 * i, v, sizeof v);
  }
  out[22] = fast.bad() ? 1.0 : 0.0;
}
int main(int, char** argv) {
  trig_table_init();
  explog_table_init();
  double in[11], out[23];
  if (argv[1][0] == 'm') {
    while (std::fread(in, sizeof(double), 2, stdin) == 2) {
      out[0] = soft_mul(in[0], in[1]);
      std::fwrite(out, sizeof(double), 1, stdout);
    }
    return 0;
  }
  if (argv[1][0] == 'a') {  // s, f: s + f, and f - 2 as a double
    while (std::fread(in, sizeof(double), 2, stdin) == 2) {
      ArithFast<true> fast(1.0, -0.0);
      out[0] = fast.add_small(in[0], (float)in[1]);
      out[1] = fast.minus_two(std::fabs(in[0]));
      std::fwrite(out, sizeof(double), 2, stdout);
    }
    return 0;
  }
  while (std::fread(in, sizeof(double), 11, stdin) == 11) {
    if (argv[1][0] == 's')
      in[0] == 0.0 ? attempt<KerrMetric, true>(in, out) : attempt<QMetric, true>(in, out);
    else
      in[0] == 0.0 ? attempt<KerrMetric, false>(in, out) : attempt<QMetric, false>(in, out);
    std::fwrite(out, sizeof(double), 23, stdout);
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def dev(tmp_path_factory):
    exe = build(tmp_path_factory, "arith64", HARNESS, device_shims=True)

    def run(op, x, width):
        inp = np.ascontiguousarray(x, dtype=np.float64)
        p = subprocess.run([str(exe), op], input=inp.tobytes(), capture_output=True, check=True)
        return np.frombuffer(p.stdout, dtype=np.float64).reshape(-1, width)
    return run


def _numbers(rng, n, span, bits=53):
    """n doubles with random signs, exponents in [-span, span) and significands
    of at most `bits` bits."""
    m = rng.integers(2 ** (bits - 1), 2 ** bits, n).astype(np.float64)  # exact: bits <= 53
    return np.ldexp(m, rng.integers(-span, span, n) - (bits - 1)) * rng.choice([-1.0, 1.0], n)


def test_products(dev):
    rng = np.random.default_rng(7)
    pairs = []
    for bits_a, bits_b in ((53, 53), (53, 3), (53, 2), (27, 27), (30, 24), (1, 53), (26, 26)):
        pairs.append(np.stack([_numbers(rng, 40000, 480, bits_a),
                               _numbers(rng, 40000, 480, bits_b)], 1))
    one = 1.0 + 2.0 ** -52
    edge = [1.0, one, 2.0 - 2.0 ** -52, 1.5, 1.5 + 2.0 ** -52, 2.0 ** -500, 2.0 ** 500]
    pairs.append(np.array([[a, b] for a in edge for b in edge]))
    x = np.concatenate(pairs)
    want = x[:, 0] * x[:, 1]
    got = dev("m", x, 1)[:, 0]
    assert np.array_equal(got.view(np.uint64), want.view(np.uint64))


def _rays(rng, n):
    """Ordinary rays of both space-times: rows (metric, integrator, a, q, E, L,
    r, theta, p_r, p_theta, h); the first ones with zeros where rays have them."""
    r = np.exp(rng.uniform(np.log(2.05), np.log(1100.0), n))
    x = np.stack([rng.integers(0, 2, n), rng.integers(0, 2, n), rng.uniform(0, 0.998, n),
                  rng.uniform(-0.5, 0.5, n), rng.uniform(0.9, 1.1, n), rng.uniform(-8, 8, n), r,
                  rng.uniform(0.02, np.pi - 0.02, n), rng.uniform(-2, 2, n),
                  rng.uniform(-8, 8, n), r * np.exp(rng.uniform(np.log(1e-6), np.log(0.1), n))],
                 1)
    x[:, 2] *= x[:, 0] == 0
    x[:, 3] *= x[:, 0] == 1
    k = n // 8
    x[:k, 2] = 0.0                 # Schwarzschild
    x[k:2 * k, 5] = 0.0            # the middle column
    x[2 * k:3 * k, 9] = 0.0        # the middle row, edge on
    x[2 * k:3 * k, 7] = np.pi / 2
    x[:k // 2, 5] = 0.0            # a = L = 0: p_theta' = 0
    x[3 * k:4 * k, 6] = 1000.0     # the observer's radius, first step length
    x[3 * k:4 * k, 10] = 10.0
    return x


def test_sums(dev):
    """s + f for floats of every size below and around the line to native
    sums, and r - 2 around 1, 2, 4, 2^52 and the ends of its range."""
    rng = np.random.default_rng(17)
    s = np.concatenate([_numbers(rng, 60000, 60), _numbers(rng, 30000, 60, 4),
                        2.0 ** rng.integers(-2, 56, 30000) *
                        (1.0 + rng.integers(-3, 4, 30000) * 2.0 ** -52)])
    ratio = 2.0 ** -rng.integers(0, 75, s.size).astype(np.float64)
    f = (s * ratio * rng.uniform(0.5, 2.0, s.size) * rng.choice([-1.0, 1.0], s.size))
    f = f.astype(np.float32)
    f[::11] = 0.0
    f[1::11] = np.ldexp(1.0, np.frexp(f[1::11])[1]).astype(np.float32)  # powers of two
    got = dev("a", np.stack([s, f.astype(np.float64)], 1), 2)
    want = np.stack([s + f.astype(np.float64), np.abs(s) - 2.0], 1)
    assert np.array_equal(got.copy().view(np.uint64), want.view(np.uint64))


@pytest.mark.parametrize("sums", ["s", "n"])
def test_attempts_bit_identical(dev, sums):
    rng = np.random.default_rng(11)
    x = _rays(rng, 16000)
    out = dev(sums, x, 23)
    kept = out[:, 22] == 0
    # a random step next to the horizon may throw a stage far out: 1 of these 16,000
    assert (~kept).sum() <= 4
    fast, plain = out[kept, :11], out[kept, 11:22]
    assert np.array_equal(fast.copy().view(np.uint64), plain.copy().view(np.uint64))


@pytest.mark.parametrize("column,value", [
    (8, 0.0), (8, 1e-25), (8, 1e25), (8, np.nan), (8, np.inf), (6, np.nan), (6, np.inf),
    (6, 1e-30), (6, 1e30), (4, np.nan), (7, np.nan), (9, np.inf), (9, 1e200), (10, 1e-30),
    (10, np.nan), (2, 1e-170), (5, 1e-310), (5, np.nan), (6, 2.0)])
def test_outside_the_window(dev, column, value):
    """An attempt that is not given back is right whatever its inputs."""
    rng = np.random.default_rng(13)
    x = _rays(rng, 800)
    x[:, column] = value
    out = dev("s", x, 23)
    fast, plain = out[:, :11].copy(), out[:, 11:22].copy()
    same = (fast.view(np.uint64) == plain.view(np.uint64)) | (np.isnan(fast) & np.isnan(plain))
    kept = out[:, 22] == 0
    assert same[kept].all()
    if column == 8 and value != value:
        assert not kept.any()

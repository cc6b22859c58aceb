"""What an attempt with products on the integer pipes (arith64.cuh) spends
before it is given back to plain FP64 instructions, on host builds of the FP64
stepper: none is given back for spins down to 2^-63, no evaluation is spent
where the ray's constants or the step length leave the window, and one at most
where its state does. Attempts with a kept first stage (Dormand-Prince) give
the bits of the plain ones."""
import numpy as np
import pytest

from _df_host import build
from test_arith64_host import _rays

HARNESS = r"""
#include "trace_device.cuh"
using namespace osiris_impl;
static long evaluations;
template <class Met>
struct Counted : Met {
  template <class A>
  static void rhs(const RayK& K, double r, double th, double pr, double pth, double& dr,
                  double& dth, double& dph, double& dpr, double& dpth, double& twoH,
                  double& scale, A& ar) {
    ++evaluations;
    Met::rhs(K, r, th, pr, pth, dr, dth, dph, dpr, dpth, twoH, scale, ar);
  }
};
// a kept first stage for Dormand-Prince (it comes from the plain evaluation)
template <class Met>
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
  State o[2] = {}, d[2] = {};
  Deriv k1 = {}, k7[2] = {};
  double twoH[2] = {};
  ArithFast<true> fast(1.0, -0.0);
  if (in[1] == 0.0) {
    evaluations = 0;
    ck_step64<Met>(K, y, h, o[0], d[0], twoH[0], fast);
    out[23] = (double)evaluations;
    ck_step64<Met>(K, y, h, o[1], d[1], twoH[1]);
  } else {
    rhs64_at<Met>(K, y, k1);
    evaluations = 0;
    dp_step64<Met>(K, y, h, true, k1, o[0], d[0], k7[0], fast);
    out[23] = (double)evaluations;
    dp_step64<Met>(K, y, h, true, k1, o[1], d[1], k7[1]);
    twoH[0] = k7[0].twoH;
    twoH[1] = k7[1].twoH;
  }
  for (int i = 0; i < 2; ++i) {
    const double v[11] = {o[i].r, o[i].th, o[i].ph, o[i].pr, o[i].pth, d[i].r,
                          d[i].th, d[i].ph, d[i].pr, d[i].pth, twoH[i]};
    std::memcpy(out + 11 * i, v, sizeof v);
  }
  out[22] = fast.bad() ? 1.0 : 0.0;
}
int main() {
  trig_table_init();
  explog_table_init();
  double in[11], out[24];
  while (std::fread(in, sizeof(double), 11, stdin) == 11) {
    in[0] == 0.0 ? attempt<Counted<KerrMetric>>(in, out) : attempt<Counted<QMetric>>(in, out);
    std::fwrite(out, sizeof(double), 24, stdout);
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def attempts(tmp_path_factory):
    import subprocess
    exe = build(tmp_path_factory, "arith64_window", HARNESS, device_shims=True)

    def run(x):
        p = subprocess.run([str(exe)], input=np.ascontiguousarray(x).tobytes(),
                           capture_output=True, check=True)
        return np.frombuffer(p.stdout, dtype=np.float64).reshape(-1, 24)
    return run


def _same(out):
    fast, plain = out[:, :11].copy(), out[:, 11:22].copy()
    return (fast.view(np.uint64) == plain.view(np.uint64)) | (np.isnan(fast) & np.isnan(plain))


@pytest.mark.parametrize("a", [0.0, 2.0 ** -63, 1e-12, 1e-10, 3e-10, 1e-3])
def test_small_spins_are_not_given_back(attempts, a):
    x = _rays(np.random.default_rng(19), 4000)
    x[:, 2] = np.where(x[:, 0] == 0, a, 0.0)
    out = attempts(x)
    kept = out[:, 22] == 0
    assert (~kept).sum() <= 4  # steps next to the horizon
    assert _same(out)[kept].all()
    assert (out[kept, 23] == 6).all()


@pytest.mark.parametrize("column,value,most", [
    (2, 1e-25, 0), (2, 1e-170, 0), (5, 1e-25, 0), (5, 1e25, 0), (10, 1e-30, 0), (10, np.nan, 0),
    (8, 0.0, 1), (8, 1e25, 1), (4, 1e25, 1), (6, np.inf, 1), (7, np.nan, 1)])
def test_attempts_outside_the_window_stop(attempts, column, value, most):
    """Kerr rays (the q-metric takes L and p_theta to no product on the integer pipes)."""
    x = _rays(np.random.default_rng(23), 800)
    x = x[x[:, 0] == 0]
    if value == 0.0:
        x = x[x[:, 1] == 0]  # Dormand-Prince has that stage, and goes on
    x[:, column] = value
    out = attempts(x)
    given_back = out[:, 22] != 0
    assert given_back.all()
    assert (out[given_back, 23] <= most).all()


def test_kept_first_stage_bit_identical(attempts):
    x = _rays(np.random.default_rng(29), 8000)
    x[:, 1] = 1.0
    out = attempts(x)
    kept = out[:, 22] == 0
    assert (~kept).sum() <= 4
    assert _same(out)[kept].all()

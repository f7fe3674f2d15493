"""Device code run on the host with the threads of a CTA one after another, in both orders: a result
that depends on the order shows threads that exchange data without a barrier."""
import numpy as np
import pytest

from tests.simt import cut, run

TREE = r"""
#include "simt.h"
inline double rcp_approx(double q) {           // 20 bits, subnormal results and arguments as zero
  if (std::fabs(q) < 2.2250738585072014e-308) return q < 0 ? -INFINITY : INFINITY;
  double r = 1.0 / q;
  if (std::fabs(r) < 2.2250738585072014e-308) return r < 0 ? -0.0 : 0.0;
  long long b = __double_as_longlong(r) & ~0xffffffffll;
  return __longlong_as_double(b);
}
namespace bse {
%s
}
"""


def tree_source():
    text = cut("tree_solve.cuh", "struct TV", "__host__ __device__ __forceinline__ uint64_t mix64")
    asm = 'asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(q));'
    assert asm in text
    text = text.replace(asm, "r = rcp_approx(q);")
    # the multisection (FP32 intrinsics) is not needed here
    i, j = text.index("// ---- the same count in double-FP32"), text.index("// ------", text.index("return 0.5 * (lo + hi)"))
    return TREE % (text[:i] + text[j:])


@pytest.mark.parametrize("h,nq", [(0, 2), (0, 40), (5, 1), (5, 2), (33, 29), (7, 64)])
def test_solve_tree_does_not_depend_on_the_order_of_lanes(tmp_path, h, nq):
    """(T - lambda I) x = r by a warp, both orders of its lanes, against a dense solve."""
    rng = np.random.default_rng(100 * h + nq)
    n = h + nq
    d, b = rng.uniform(1, 9, h), rng.uniform(0.1, 1, h)
    a, e = rng.uniform(1, 9, nq), rng.uniform(0.1, 3, nq - 1)      # |e| > |pivot| at times: rows exchange
    lam, r = 4.3, rng.standard_normal(n)
    arr = lambda v: "{" + ",".join([*map(repr, map(float, v)), "0"]) + "}"      # noqa: E731
    src = tree_source() + f"""
using namespace bse;
double d[] = {arr(d)}, b[] = {arr(b)}, a[] = {arr(a)}, e[] = {arr(e)}, r[] = {arr(r)};
int main() {{
  for (int desc = 0; desc < 2; ++desc) {{
    static double w[4][{n + 1}], x[{n + 1}];
    static unsigned char piv[{n + 1}];
    std::copy(r, r + {n}, x);
    TV T{{d, b, {h}, a, e, {n}}};
    Fact F{{w[0], w[1], w[2], w[3], piv}};
    if (!simt::run_block(32, desc, [&] {{
          factor_tree(T, {lam}, 1e-15, F, threadIdx.x);
          solve_tree(T, F, x, threadIdx.x);
        }})) return 1;
    for (int i = 0; i < {n}; ++i) printf("%.17g ", x[i]);
    printf("\\n");
  }}
}}
"""
    up, down = run(tmp_path, src)
    m = np.diag(np.concatenate([d, a]) - lam)
    m[:h, h] = m[h, :h] = b
    for t in range(nq - 1):
        m[h + t, h + t + 1] = m[h + t + 1, h + t] = e[t]
    assert up == down
    # backward stable: ||T x - r|| <= c n u ||T|| ||x||
    assert np.linalg.norm(m @ up - r) <= 64 * n * 2.0 ** -53 * np.linalg.norm(m, 2) * np.linalg.norm(up)


PANEL = r"""
#include "simt.h"
#define __restrict__
namespace bse {
constexpr int DNB = 32;
%s
}
using namespace bse;
int main(int, char** argv) {
  const int n = atoi(argv[1]), ld = (n + 31) / 32 * 32, kb = std::min(n, DNB), nt = std::max(1, (n - kb + 31) / 32);
  for (int desc = 0; desc < 2; ++desc) {
    std::vector<double> M(ld * n), D(DNB * DNB);
    int notpd = 0;
    for (int j = 0; j < n; ++j)
      for (int i = 0; i < n; ++i) M[j * ld + i] = (i == j ? n + 1.0 : 0.0) + std::cos(0.7 * (i - j) * (i - j));
    for (int b = 0; b < nt; ++b) {
      blockIdx.x = b;
      if (!simt::run_block(256, desc, [&] { k_dn_panel(M.data(), ld, n, 0, kb, D.data(), &notpd); })) return 1;
    }
    for (int c = 0; c < kb; ++c)
      for (int r = c; r < kb; ++r) M[c * ld + r] = D[c * DNB + r];
    for (int c = 0; c < kb; ++c)
      for (int r = 0; r < n; ++r) printf("%%.17g ", r < c ? 0.0 : M[c * ld + r]);
    printf("%%d\n", notpd);
  }
}
"""


@pytest.mark.parametrize("n", [1, 17, 32, 33, 75])
def test_cholesky_panel_does_not_depend_on_the_order_of_threads(tmp_path, n):
    """The first panel of the dense method's Cholesky factorisation, both orders of a CTA's threads."""
    src = PANEL % cut("k_dense.cu", "__global__ void __launch_bounds__(256) k_dn_panel", "// trailing update")
    up, down = run(tmp_path, src, n)
    assert up == down
    k = min(n, 32)
    i = np.arange(n)
    m = np.cos(0.7 * (i[:, None] - i[None, :]) ** 2) + (n + 1.0) * np.eye(n)
    ref = np.linalg.cholesky(m)[:, :k]
    assert up[-1] == 0
    np.testing.assert_allclose(np.reshape(up[:-1], (k, n)).T, ref, rtol=0, atol=64 * n * 2.0 ** -53 * np.sqrt(n + 2))

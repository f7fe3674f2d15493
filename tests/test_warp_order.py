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

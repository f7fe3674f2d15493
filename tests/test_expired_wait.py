"""An expired wait of a product kernel fails the call that ran into it, not the handle's later calls: the
host's part of the error path, compiled for the host with stand-ins for the runtime's copies."""
from tests.simt import cut, run

SRC = r"""
#include <cstdio>
#include <cstring>
enum { BSE_OK = 0, BSE_ETIMEOUT = 5, BSE_ECUDA = 6, cudaSuccess = 0, cudaMemcpyDeviceToHost = 2 };
typedef int cudaError_t;
typedef void* cudaStream_t;
#define CK(x) do { if ((x) != cudaSuccess) return BSE_ECUDA; } while (0)
static int cudaMemcpyAsync(void* d, const void* s, size_t n, int, cudaStream_t) { memcpy(d, s, n); return 0; }
static int cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { memset(d, v, n); return 0; }
static int cudaStreamSynchronize(cudaStream_t) { return 0; }
struct bse_handle { int* prod_err; cudaStream_t stream; };
%s
int main() {
  int flag = 0;
  bse_handle h{&flag, nullptr}, none{nullptr, nullptr};
  const int a = sync_product(&h);
  flag = 1;                                // as a kernel's expired wait leaves it
  const int b = sync_product(&h), c = sync_product(&h);
  printf("%%d %%d %%d %%d %%d\n", a, b, c, sync_product(&none), flag);
}
"""


def test_only_one_call_fails(tmp_path):
    assert run(tmp_path, SRC % cut("bse_api.cu", "// BSE_ETIMEOUT when perr", "int map_status")) == [[0, 5, 0, 0, 0]]

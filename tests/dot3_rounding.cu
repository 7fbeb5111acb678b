// The three-term complex products of the stencils, contractions and transports
// against separately formed products, one thread per product; called by
// test_gpu_dot3_rounding.py.
#include "contract.cuh"

using namespace tsm;

template <class R>
__global__ void dots(const cx<R>* a, const cx<R>* b, cx<R>* dot, cx<R>* chain, cx<R>* spin, cx<R>* sums, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const cx<R>*x = a + 3 * i, *y = b + 3 * i;
  dot[i] = cdot3(x[0], y[0], x[1], y[1], x[2], y[2]);
  chain[i] = cdot3_chain(x[0], y[0], x[1], y[1], x[2], y[2]);
  spin[i] = spin_product<R>(x, y);
  sums[i] = x[0] * y[0] + x[1] * y[1] + x[2] * y[2];
}

extern "C" int dot3_rounding(const void* a, const void* b, void* dot, void* chain, void* spin, void* sums, int n) {
  using C = cx<float>;
  dots<float><<<(n + 127) / 128, 128>>>(static_cast<const C*>(a), static_cast<const C*>(b), static_cast<C*>(dot),
                                       static_cast<C*>(chain), static_cast<C*>(spin), static_cast<C*>(sums), n);
  return (int)cudaDeviceSynchronize();
}

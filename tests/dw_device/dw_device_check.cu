// Device check of the double-word arithmetic (csrc/dw.cuh, csrc/dw2.cuh): the
// reciprocal and division, whose device code differs from what the host check
// compiles, against float64, and the packed fiber product against the scalar
// operations, bit for bit.  Prints "name value" per check.
#include <cstdint>
#include <cstdio>
#include <cstring>

#include "dw2.cuh"

using namespace ax;

// counter-based random bits
__host__ __device__ inline uint64_t mix(uint64_t z) {
  z += 0x9e3779b97f4a7c15ull;
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}
// a double-word value +-[1, 2) 2^e (positive: plus)
__device__ dw::dw value(uint64_t key, int e, bool positive) {
  const uint64_t a = mix(key), b = mix(a);
  double v = 1.0 + (double)(a >> 11) * 0x1p-53;
  if (!positive && (b & 1)) v = -v;
  return dw::from_double(ldexp(v, e));
}

// err[0]: largest |y rcp(y) - 1| in units of 2^-24, y over [2^-100, 2^101);
// err[1]: largest relative error of x / y in units of 2^-47, y over the
// determinants (L / 2)^3 of elements of the accepted extents L in [2^-20, 2^24]
// with room for their shape, x over the products of three weights.
__global__ void quotients(int n, unsigned *err) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= n) return;
  const float w = value(7 * (uint64_t)q, (int)(mix(3 * (uint64_t)q + 2) % 201) - 100, true).hi;
  const double r = fabs(fma((double)dw::rcp(w), (double)w, -1.0)) * 0x1p24;
  const int ey = (int)(mix(3 * (uint64_t)q) % 147) - 75, ex = (int)(mix(3 * (uint64_t)q + 1) % 22) - 21;
  const dw::dw y = value(5 * (uint64_t)q, ey, true), x = value(5 * (uint64_t)q + 1, ex, false);
  const dw::dw d = dw::div(x, y);
  const double ref = dw::to_double(x) / dw::to_double(y);
  const double e = fabs((double)d.hi - ref + (double)d.lo) / fabs(ref) * 0x1p47;
  atomicMax(&err[0], __float_as_uint((float)r));
  atomicMax(&err[1], __float_as_uint((float)e));
}

// the scalar fiber product, operation by operation
template <int N1>
__device__ __noinline__ void scalar_product(const float4 *eo2, const dw::dw *in, dw::dw *out) {
  constexpr int c = N1 / 2;
  for (int i = 0; i < c; ++i) {
    dw::acc p{0.f, 0.f}, q{0.f, 0.f};
    for (int m = 0; m < c; ++m) {
      const float4 k = eo2[i * c + m];
      const dw::dw e = dw::add_lazy(in[m], in[N1 - 1 - m]), o = dw::sub_lazy(in[m], in[N1 - 1 - m]);
      const dw::dw A{k.x, k.z}, B{k.y, k.w};
      if (m == 0) {
        p = dw::mul_acc(A, e);
        q = dw::mul_acc(B, o);
      } else {
        dw::mac(p, A, e);
        dw::mac(q, B, o);
      }
    }
    if (N1 < 16) {
      out[i] = dw::acc_sum(p, q);
      out[N1 - 1 - i] = dw::acc_dif(q, p);
    } else {
      const dw::dw P = dw::fin(p), Q = dw::fin(q);
      out[i] = dw::add(P, Q);
      out[N1 - 1 - i] = dw::sub(Q, P);
    }
  }
}
template <int N1>
__global__ void products(int n, unsigned *bad) {
  constexpr int c = N1 / 2;
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= n) return;
  float4 eo2[c * c];
  dw::dw in[N1], got[N1], ref[N1];
  uint64_t key = 1000003ull * N1 + (uint64_t)q * 4096;
  for (int m = 0; m < c * c; ++m) {
    const dw::dw a = value(key++, (int)(mix(key) % 13) - 6, false), b = value(key++, (int)(mix(key) % 13) - 6, false);
    eo2[m] = make_float4(a.hi, b.hi, a.lo, b.lo);
  }
  for (int m = 0; m < N1; ++m) in[m] = value(key++, (int)(mix(key) % 41) - 20, false);
  dw2::contract<N1>(eo2, in, got);
  scalar_product<N1>(eo2, in, ref);
  unsigned b = 0;
  for (int m = 0; m < N1; ++m)
    b += __float_as_uint(got[m].hi) != __float_as_uint(ref[m].hi) || __float_as_uint(got[m].lo) != __float_as_uint(ref[m].lo);
  if (b) atomicAdd(bad, b);
}

int main() {
  unsigned *d = nullptr, h[10] = {};
  if (cudaMalloc(&d, sizeof h) != cudaSuccess || cudaMemset(d, 0, sizeof h) != cudaSuccess) return 1;
  const int n = 1 << 20, m = 1 << 14;
  quotients<<<n / 256, 256>>>(n, d);
  products<2><<<m / 64, 64>>>(m, d + 2);
  products<4><<<m / 64, 64>>>(m, d + 3);
  products<6><<<m / 64, 64>>>(m, d + 4);
  products<8><<<m / 64, 64>>>(m, d + 5);
  products<10><<<m / 64, 64>>>(m, d + 6);
  products<12><<<m / 64, 64>>>(m, d + 7);
  products<14><<<m / 64, 64>>>(m, d + 8);
  products<16><<<m / 64, 64>>>(m, d + 9);
  if (cudaMemcpy(h, d, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
  float e[2];
  std::memcpy(e, h, sizeof e);
  std::printf("rcp %.6f\ndiv %.6f\n", e[0], e[1]);
  for (int q = 0; q < 8; ++q) std::printf("product%d %u\n", 2 * (q + 1), h[2 + q]);
  return 0;
}

// lb_step_f64.cu -- double-precision dispatch of the fused step kernels: the launch, persistent
// launch and set-up entry points, which reach the kernels through the kernel families compiled
// in lb_step_f64_gen.cu, lb_step_f64_b64.cu and lb_step_f64_b128.cu (one translation unit each
// keeps the build parallel).
#include <mutex>

#include "lb_step_impl.cuh"

namespace lbk {

#define LB_STEP_INST(real)                                                                                         \
  template size_t step_smem_bytes<real>(int);                                                                      \
  template cudaError_t prepare_step<real>(int);                                                                    \
  template cudaError_t launch_step<real>(const StepArgs<real>&, int, bool, int, bool, cudaStream_t);               \
  template int persistent_grid<real>(int, int, bool);                                                              \
  template cudaError_t launch_step_persistent<real>(const StepArgs<real>&, int, int, int, bool, const PersistArgs&, \
                                                    int, cudaStream_t);                                         \
  template cudaError_t launch_debug_normals<real>(const uint32_t*, int64_t, double*, const NormalTables*, cudaStream_t);
LB_STEP_INST(double)

// ---- the tables of the double-precision normals (lb_normals64.cuh) -------------------------------
namespace {

__device__ NormalTables g_normals;
__device__ int g_normals_filled;  // zero until the tables are: in the module, like them

// ln 2 in two parts, the first with 24 bits, so that its product with an exponent is exact
constexpr double kLn2Hi = 0.693147182464599609375, kLn2Lo = -1.904654299957768e-09;

// sqrt(-2 ln(x)) (side 0) or sqrt(-2 ln(1 - x)) (side 1) as a sum: the root of the rounded argument, and
// the first-order correction for what the roundings of the argument and the root left out
__device__ void radius_sum(int side, double x, double& r, double& corr) {
  double hi, lo = 0.0;
  if (side == 0) {
    int e;
    double f = frexp(x, &e);  // [1/2, 1)
    if (f < 0.70710678118654752) {
      f *= 2.0;
      e -= 1;
    }
    const double big = -2.0 * e * kLn2Hi, small = -2.0 * (log(f) + e * kLn2Lo);
    hi = big + small;
    lo = fabs(big) >= fabs(small) ? (big - hi) + small : (small - hi) + big;
  } else {
    hi = -2.0 * log1p(-x);
  }
  r = sqrt(hi);
  corr = (fma(-r, r, hi) + lo) / (2.0 * r);
}

__global__ void fill_normals_kernel() {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const double two60 = 1152921504606846976.0, two24 = 16777216.0;
  if (i < 2 * 4096) {
    const int side = i >> 12, idx = i & 4095, sh = idx < 512 ? 0 : (idx >> 8) - 1;
    if (idx == 0) return;
    const double w = (double)(1 << sh) / two24, q0 = (double)(idx - sh * 256) * w;  // [q0, q0 + w)
    NormalTables::Segment sg = {};
    double r, corr;
    if (sh == 0) {  // one value of q per segment: T = 0
      radius_sum(side, q0, r, corr);
      sg.c0 = llrint(r * two60) + llrint(corr * two60);
    } else {
      // y(z) = -2 ln u at u = middle + z w: y0 + sum_k a_k z^k; the root's series b_k from
      // sum_{i+j=k} b_i b_j = a_k; then moved from z = T - 1/2 to T/2
      const double x0 = q0 + 0.5 * w, t = side == 0 ? w / x0 : -w / (1.0 - x0);
      radius_sum(side, x0, r, corr);
      double b[6], tk = 1.0;
      b[0] = r;
      for (int k = 1; k < 6; ++k) {
        tk *= t;
        double acc = ((k & 1) ? -2.0 : 2.0) * tk / k;
        for (int j = 1; j < k; ++j) acc -= b[j] * b[k - j];
        b[k] = acc / (2.0 * r);
      }
      const double binom[6][6] = {{1}, {1, 1}, {1, 2, 1}, {1, 3, 3, 1}, {1, 4, 6, 4, 1}, {1, 5, 10, 10, 5, 1}};
      double c[6];
      for (int j = 5; j >= 0; --j) {
        double v = 0.0, h = 1.0;  // h = (-1/2)^(k - j)
        for (int k = j; k < 6; ++k, h *= -0.5)
          if (k > 0) v += b[k] * binom[k][j] * h;
        c[j] = v * (double)(1 << j);
      }
      sg.c0 = llrint(r * two60) + llrint((c[0] + corr) * two60);
      sg.c1 = llrint(c[1] * two60);
      sg.c2 = llrint(c[2] * two60);
      sg.c3 = llrint(c[3] * two60);
      sg.c4 = (int)llrint(c[4] * two60);
      sg.c5 = (int)llrint(c[5] * two60);
    }
    g_normals.radius[i] = sg;
  } else if (i < 2 * 4096 + 1024) {
    const int j = i - 2 * 4096;
    double s, c;
    sincospi((double)j / 2048.0, &s, &c);
    const double two63 = 8.0 * two60;
    g_normals.turn[j] = make_ulonglong2((unsigned long long)(c * two63), (unsigned long long)(s * two63));
  } else if (i < 2 * 4096 + 1024 + 2048) {
    const int j = i - 2 * 4096 - 1024;
    double s, c, hs, hc;
    sincospi((double)(2 * j + 1) / (0.5 * two24), &s, &c);
    sincospi((double)(2 * j + 1) / two24, &hs, &hc);
    const double two73 = 8192.0 * two60;
    g_normals.rest[j] = make_ulonglong2((unsigned long long)(s * two73), (unsigned long long)(2.0 * hs * hs * two73));
  }
}

}  // namespace

// The note that the tables are filled lies beside them on the device, so that it holds for the current
// context's tables and for no others: after a device reset, or in a second context of the device, both are
// new.  Fill and note are on the legacy stream, as is what the caller does next (lb_create_batch waits for
// that stream before it returns).
cudaError_t normal_tables(const NormalTables** tab) {
  static std::mutex mu;
  std::lock_guard<std::mutex> g(mu);
  void* p = nullptr;
  cudaError_t e = cudaGetSymbolAddress(&p, g_normals);
  int filled = 0;
  if (e == cudaSuccess) e = cudaMemcpyFromSymbol(&filled, g_normals_filled, sizeof(filled));
  if (e == cudaSuccess && !filled) {
    fill_normals_kernel<<<(2 * 4096 + 1024 + 2048 + 127) / 128, 128>>>();
    e = cudaGetLastError();
    filled = 1;
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_normals_filled, &filled, sizeof(filled));
  }
  if (e != cudaSuccess) return e;
  *tab = static_cast<const NormalTables*>(p);
  return cudaSuccess;
}

}  // namespace lbk

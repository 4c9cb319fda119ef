// lb_diag.cu -- diagnostics of the fluctuating LB method: structure factors (Appendix A,
// Eqs. SF1 and integral, on the lattice: S(q) = |delta phi(q)|^2 with the unitary 2D
// transform), mean mechanical pressure and per-species mass (Sec. II.A, III.C), plus the
// utility kernels that convert between stored and absolute populations.
//
// Structure factors: the step kernel writes the four fields of every site on a sample step;
// here one block per group of rows transforms them along x (two real rows per complex
// transform) and one block per strip of adjacent q_x transforms the columns along z, squares,
// scales by 1 / (Lx Lz) and adds the result to double-precision Kahan (compensated)
// accumulators.
#include <algorithm>
#include <type_traits>

#include "lb_internal.cuh"

namespace lbk {

template <class real>
struct Cplx {
  real re, im;
};

// One stored (A, B) pair.
template <class real>
struct PairType {
  using type = typename std::conditional<sizeof(real) == 4, float2, double2>::type;
};

namespace {

// Twiddle tables of the transforms, exp(-2 pi i k / n) for k < n/2, every power of two n = 2 .. 8192 at
// offset n/2 - 1.  Single precision: filled by prepare_sf, which only contexts call.  Double precision: part
// of the module, since lb_power_spectrum reads it without a context, from its first call on, in a stream
// capture or not; a fill by a kernel (then a wait for the device) would break a capture, and a note that it
// was done would outlive the table when the device is reset.
constexpr int TW_TABLE = 8192;

// The unevaluated sum of two doubles, and the product of two of them to about 2^-104 (Dekker 1971), for the
// compiler's evaluation of the table.
struct TwoDoubles {
  double hi, lo;
};
constexpr TwoDoubles two_sum(double a, double b) {
  const double s = a + b, t = s - a;
  return {s, (a - (s - t)) + (b - t)};
}
constexpr TwoDoubles two_product(double a, double b) {
  const double ca = 134217729.0 * a, cb = 134217729.0 * b;  // 2^27 + 1
  const double ah = ca - (ca - a), bh = cb - (cb - b), al = a - ah, bl = b - bh;
  const double p = a * b;
  return {p, ((ah * bh - p) + ah * bl + al * bh) + al * bl};
}
constexpr TwoDoubles add(TwoDoubles a, TwoDoubles b) {
  const TwoDoubles s = two_sum(a.hi, b.hi);
  return two_sum(s.hi, s.lo + (a.lo + b.lo));
}
constexpr TwoDoubles multiply(TwoDoubles a, TwoDoubles b) {
  const TwoDoubles p = two_product(a.hi, b.hi);
  return two_sum(p.hi, p.lo + (a.hi * b.lo + a.lo * b.hi));
}

struct TwiddleTable {
  Cplx<double> v[TW_TABLE];
};
constexpr TwiddleTable make_twiddles() {
  // cos and sin of 2 pi j / 8192 in the first octant: the powers of exp(2 pi i / 8192), each the product of
  // the last and the first; the rest by symmetry
  const TwoDoubles c1{0x1.fffff62161a34p-1, -0x1.136dcb1f9b9c4p-57}, s1{0x1.921fb2aecb360p-11, 0x1.876157e566b4cp-65};
  double co[1025] = {}, si[1025] = {};
  TwoDoubles c{1.0, 0.0}, s{0.0, 0.0};
  for (int j = 0; j <= 1024; ++j) {
    co[j] = c.hi;
    si[j] = s.hi;
    const TwoDoubles ss = multiply(s, s1), cn = add(multiply(c, c1), TwoDoubles{-ss.hi, -ss.lo});
    s = add(multiply(s, c1), multiply(c, s1));
    c = cn;
  }
  TwiddleTable t{};
  for (int n = 2; n <= TW_TABLE; n *= 2)
    for (int k = 0; k < n / 2; ++k) {
      const int j = k * (TW_TABLE / n), m = j <= 2048 ? j : 4096 - j;  // angle, and its mirror image below pi/2
      const double cm = m <= 1024 ? co[m] : si[2048 - m], sm = m <= 1024 ? si[m] : co[2048 - m];
      t.v[n / 2 - 1 + k] = Cplx<double>{j <= 2048 ? cm : -cm, -sm};
    }
  return t;
}

__device__ Cplx<float> g_tw_f[TW_TABLE];
__device__ const TwiddleTable g_tw_d = make_twiddles();
template <class real>
__device__ __forceinline__ const Cplx<real>* tw_table();
template <>
__device__ __forceinline__ const Cplx<float>* tw_table<float>() { return g_tw_f; }
template <>
__device__ __forceinline__ const Cplx<double>* tw_table<double>() { return g_tw_d.v; }

__global__ void fill_tw_table_kernel() {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < TW_TABLE - 1; i += gridDim.x * blockDim.x) {
    const int n = 2 << (31 - __clz(i + 1));  // the table holding entry i: n/2 - 1 <= i < n - 1
    const int k = i - (n / 2 - 1);
    float c, sn;
    sincospif(-2.0f * (float)k / (float)n, &sn, &c);  // k / n is exact in binary
    g_tw_f[i] = Cplx<float>{c, sn};
  }
}

// The twiddles of an n-point transform into shared memory, from the table.
template <class real>
__device__ void load_twiddles(Cplx<real>* tw, int n) {
  const Cplx<real>* t = tw_table<real>() + (n / 2 - 1);
  for (int k = threadIdx.x; k < (n >> 1); k += blockDim.x) tw[k] = t[k];
}

__device__ __forceinline__ void neumaier_add(double& sum, double& comp, double v) {
  const double t = sum + v;
  if (fabs(sum) >= fabs(v)) comp += (sum - t) + v;
  else comp += (v - t) + sum;
  sum = t;
}

// ---- sample-step transforms: self-sorting (Stockham) radix-16/8/4/2 passes --------------------
// A pass of radix R over sequences of n points that have already been combined in spans of Ns
// (Ns = product of the earlier radices): butterfly j (k = j mod Ns) takes the points j + r n/R,
// r = 0 .. R-1, turns point r by exp(-2 pi i r k / (Ns R)), forms their R-point DFT in registers
// and stores output q at (j - k) R + k + q Ns.  After the last pass the sequence holds its DFT
// X_k = sum_j x_j exp(-2 pi i j k / n) in natural order (the autosort formulation of Stockham's
// FFT, e.g. Govindaraju et al., SC 2008).  Each thread holds PTS points per pass; a barrier
// separates its loads from its stores, so one buffer serves every pass.

template <class real>
__device__ __forceinline__ Cplx<real> cmul(Cplx<real> a, Cplx<real> b) {
  return Cplx<real>{a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re};
}

// cos and sin of 2 pi k / 16, k = 0 .. 7
__host__ __device__ constexpr double cos16(int k) {
  return k == 0 ? 1.0
       : k == 1 ? 0.92387953251128675613
       : k == 2 ? 0.70710678118654752440
       : k == 3 ? 0.38268343236508977173
       : k == 4 ? 0.0
       : k == 5 ? -0.38268343236508977173
       : k == 6 ? -0.70710678118654752440
                : -0.92387953251128675613;
}
__host__ __device__ constexpr double sin16(int k) { return k <= 4 ? cos16(4 - k) : cos16(k - 4); }

// x exp(-2 pi i k / 16) for a compile-time k in 0 .. 7 (after unrolling), without products where
// the factor is 1 or -i.
template <class real>
__device__ __forceinline__ Cplx<real> turn16(Cplx<real> x, int k) {
  if (k == 0) return x;
  if (k == 4) return Cplx<real>{x.im, -x.re};
  const real c = (real)cos16(k), s = (real)sin16(k);
  return Cplx<real>{x.re * c + x.im * s, x.im * c - x.re * s};
}

// i (0 .. 2^bits - 1, bits <= 4) with its bits reversed
__host__ __device__ constexpr int bitrev_small(int i, int bits) {
  return (((i & 1) << 3) | ((i & 2) << 1) | ((i & 4) >> 1) | ((i & 8) >> 3)) >> (4 - bits);
}

// In-order R-point DFT of v[0 .. R-1] in registers (R = 2, 4, 8, 16): radix-2 butterflies on the
// bit-reversed inputs.
template <class real, int R>
__device__ __forceinline__ void dft_regs(Cplx<real>* v) {
  constexpr int bits = R == 16 ? 4 : R == 8 ? 3 : R == 4 ? 2 : 1;
  Cplx<real> t[R];
#pragma unroll
  for (int i = 0; i < R; ++i) t[i] = v[bitrev_small(i, bits)];
#pragma unroll
  for (int h = 1; h < R; h <<= 1) {
#pragma unroll
    for (int g = 0; g < R; g += 2 * h) {
#pragma unroll
      for (int p = 0; p < h; ++p) {
        const Cplx<real> a = t[g + p], b = turn16(t[g + p + h], p * (8 / h));
        t[g + p] = Cplx<real>{a.re + b.re, a.im + b.im};
        t[g + p + h] = Cplx<real>{a.re - b.re, a.im - b.im};
      }
    }
  }
#pragma unroll
  for (int i = 0; i < R; ++i) v[i] = t[i];
}

// One pass over `seqs` sequences of n points at s + seq * sf_seq_stride(n) (point p at p + p/16);
// tw: exp(-2 pi i e / n) for e < n/2.
template <class real, int R, int PTS>
__device__ __forceinline__ void stockham_pass(Cplx<real>* s, const Cplx<real>* tw, int n, int Ns, int seqs) {
  constexpr int BPT = PTS / R;  // butterflies per thread
  const int nb = n / R, lnb = 31 - __clz(nb);
  const int total = seqs * nb, SS = sf_seq_stride(n);
  const int unit = n / (Ns * R), h = n >> 1;
  Cplx<real> v[PTS];
#pragma unroll
  for (int i = 0; i < BPT; ++i) {
    const int b = threadIdx.x + i * blockDim.x;
    if (b < total) {
      const int seq = b >> lnb, j = b & (nb - 1), k = j & (Ns - 1);
      const Cplx<real>* src = s + seq * SS;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int p = j + r * nb;
        v[i * R + r] = src[p + (p >> 4)];
      }
      if (k != 0) {
        const int st = k * unit;
#pragma unroll
        for (int r = 1; r < R; ++r) {
          const int e = r * st;  // < n
          const Cplx<real> w = tw[e < h ? e : e - h];
          const Cplx<real> ws = e < h ? w : Cplx<real>{-w.re, -w.im};
          v[i * R + r] = cmul(v[i * R + r], ws);
        }
      }
      dft_regs<real, R>(v + i * R);
    }
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < BPT; ++i) {
    const int b = threadIdx.x + i * blockDim.x;
    if (b < total) {
      const int seq = b >> lnb, j = b & (nb - 1), k = j & (Ns - 1);
      Cplx<real>* dst = s + seq * SS;
      const int d = (j - k) * R + k;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int p = d + r * Ns;
        dst[p + (p >> 4)] = v[i * R + r];
      }
    }
  }
  __syncthreads();
}

// DFT of `seqs` sequences of n = 2^m points in place (seqs n <= PTS blockDim.x): passes of radix PTS
// (4, 8 or 16), then one pass of the remaining radix.
template <class real, int PTS>
__device__ void stockham_fft(Cplx<real>* s, const Cplx<real>* tw, int n, int seqs) {
  constexpr int bits = PTS == 16 ? 4 : PTS == 8 ? 3 : 2;
  int left = 31 - __clz(n), Ns = 1;
  for (; left >= bits; left -= bits, Ns <<= bits) stockham_pass<real, PTS, PTS>(s, tw, n, Ns, seqs);
  if (PTS > 8 && left == 3) stockham_pass<real, PTS < 8 ? PTS : 8, PTS>(s, tw, n, Ns, seqs);
  else if (PTS > 4 && left == 2) stockham_pass<real, 4, PTS>(s, tw, n, Ns, seqs);
  else if (left == 1) stockham_pass<real, 2, PTS>(s, tw, n, Ns, seqs);
}

// Global loads per thread that the transforms issue before they wait for the first (row pass,
// column pass; fewer in double precision, whose registers hold the 16 points of a pass).
template <class real>
struct SfBatch {
  static constexpr int rows = sizeof(real) == 4 ? 8 : 4, cols = sizeof(real) == 4 ? 4 : 2;
};

// R real rows of n points at src (contiguous) to the q_x = 0 .. n/2 bins of their transforms at out
// (n/2 + 1 per row).  Rows 2c and 2c + 1 enter as the real and imaginary parts of sequence c, so one
// complex transform gives both: with Z = DFT(a + i b), A_q = (Z_q + conj Z_{n-q}) / 2 and
// B_q = (Z_q - conj Z_{n-q}) / (2 i).  The sequences stay in s.
template <class real, int PTS>
__device__ __forceinline__ void transform_rows(const real* __restrict__ src, int n, int R, Cplx<real>* out,
                                               Cplx<real>* tw, Cplx<real>* s) {
  const int logn = 31 - __clz(n), H = sf_half(n), SS = sf_seq_stride(n), seqs = (R + 1) >> 1;
  load_twiddles<real>(tw, n);
  const int total = seqs * n, T = blockDim.x;
  // loads in batches of SfBatch<real>::rows per thread, all issued before their shared-memory stores
  for (int base = threadIdx.x; base < total; base += SfBatch<real>::rows * T) {
    real a[SfBatch<real>::rows], b[SfBatch<real>::rows];
#pragma unroll
    for (int i = 0; i < SfBatch<real>::rows; ++i) {
      const int idx = base + i * T;
      if (idx < total) {
        const int c = idx >> logn, j = idx & (n - 1);
        a[i] = src[(int64_t)(2 * c) * n + j];
        b[i] = 2 * c + 1 < R ? src[(int64_t)(2 * c + 1) * n + j] : real(0);
      }
    }
#pragma unroll
    for (int i = 0; i < SfBatch<real>::rows; ++i) {
      const int idx = base + i * T;
      if (idx < total) {
        const int c = idx >> logn, j = idx & (n - 1);
        s[c * SS + j + (j >> 4)] = Cplx<real>{a[i], b[i]};
      }
    }
  }
  __syncthreads();
  stockham_fft<real, PTS>(s, tw, n, seqs);
  const int dc = T / H, dq = T - dc * H;
  int c = threadIdx.x / H, q = threadIdx.x - c * H;
  for (int idx = threadIdx.x; idx < seqs * H; idx += T) {
    const int qm = (n - q) & (n - 1);
    const Cplx<real> Z = s[c * SS + q + (q >> 4)], M = s[c * SS + qm + (qm >> 4)];
    const real hf = real(0.5);
    out[(int64_t)(2 * c) * H + q] = Cplx<real>{hf * (Z.re + M.re), hf * (Z.im - M.im)};
    if (2 * c + 1 < R) out[(int64_t)(2 * c + 1) * H + q] = Cplx<real>{hf * (Z.im + M.im), hf * (M.re - Z.re)};
    c += dc;
    q += dq;
    if (q >= H) {
      q -= H;
      ++c;
    }
  }
}

// Row pass: one block per (lattice, field * Lz + z0), rows z0 .. z0 + R - 1 with
// R = sf_row_group(Lx, Lz, cap).  q_x = 0 .. Lx/2 of every row goes to tmp; the q_x = 0 bin is the row
// sum, whose mean goes to the profile.
template <class real>
__global__ void __launch_bounds__(512) sf_rows_kernel(const DiagLattice* lat, const int2* tasks, const real* fields, Cplx<real>* tmp,
                               double* prof_sum, double* prof_comp, int n_rows, int cap) {
  extern __shared__ __align__(16) unsigned char smem[];
  wait_for_previous_grid();
  const int2 task = tasks[blockIdx.x];
  const DiagLattice L = lat[task.x];
  const int n = L.Lx, SS = sf_seq_stride(n), R = sf_row_group(n, L.Lz, cap);
  Cplx<real>* tw = reinterpret_cast<Cplx<real>*>(smem);
  Cplx<real>* s = tw + ((n >> 1) + 1);
  transform_rows<real, 16>(fields + 4 * L.site_off + (int64_t)task.y * n, n, R,
                       tmp + 4 * L.site_off + (int64_t)task.y * sf_half(n), tw, s);
  const int fld = task.y / L.Lz, z0 = task.y - fld * L.Lz;
  for (int r = threadIdx.x; r < R; r += blockDim.x) {
    const Cplx<real> Z0 = s[(r >> 1) * SS];
    const int64_t k = (int64_t)fld * n_rows + L.row_off + z0 + r;
    neumaier_add(prof_sum[k], prof_comp[k], (double)((r & 1) ? Z0.im : Z0.re) / (double)n);
  }
}

// Kahan summation of non-negative terms: the estimate of the total is sum - comp.
__device__ __forceinline__ void kahan_add(double& sum, double& comp, double v) {
  const double y = v - comp;
  const double t = sum + y;
  comp = (t - sum) - y;
  sum = t;
}

// Walk of a block's threads over the points idx = j w + c of a strip (row j, column c) in steps of T.
struct StripWalk {
  int j, c, dj, dc, w;
  __device__ __forceinline__ StripWalk(int w_, int T) : w(w_) {
    dj = T / w;
    dc = T - dj * w;
    j = threadIdx.x / w;
    c = threadIdx.x - j * w;
  }
  __device__ __forceinline__ void advance() {
    j += dj;
    c += dc;
    if (c >= w) {
      c -= w;
      ++j;
    }
  }
};

// The DFTs along z of w adjacent columns (n points, row stride H) of `in`, left in s (sequence c:
// column c).
template <class real, int PTS>
__device__ __forceinline__ void transform_columns(const Cplx<real>* __restrict__ in, int H, int n, int w,
                                                  Cplx<real>* tw, Cplx<real>* s) {
  load_twiddles<real>(tw, n);
  const int T = blockDim.x, total = w * n, SS = sf_seq_stride(n);
  StripWalk k(w, T);
  for (int b0 = threadIdx.x; b0 < total; b0 += SfBatch<real>::cols * T) {
    Cplx<real> x[SfBatch<real>::cols];
    int at[SfBatch<real>::cols];
#pragma unroll
    for (int i = 0; i < SfBatch<real>::cols; ++i) {
      if (b0 + i * T < total) x[i] = in[(int64_t)k.j * H + k.c];
      at[i] = k.c * SS + k.j + (k.j >> 4);
      k.advance();
    }
#pragma unroll
    for (int i = 0; i < SfBatch<real>::cols; ++i)
      if (b0 + i * T < total) s[at[i]] = x[i];
  }
  __syncthreads();
  stockham_fft<real, PTS>(s, tw, n, w);
}

// Column pass: one block per (lattice, field * Lx + q_x0), the strip of cq = sf_col_strip(Lx, Lz,
// cap) adjacent q_x from q_x0 (fewer at the end of q_x = 0 .. Lx/2; the fields are real, so
// S(-q) = S(q) and the rest is filled by symmetry when the spectrum is read out).  Rows of the
// strip are read and accumulated with contiguous accesses; the power is formed in the working
// precision and added to a double-precision Kahan sum.
template <class real>
__global__ void __launch_bounds__(512) sf_cols_kernel(const DiagLattice* lat, const int2* tasks, const Cplx<real>* tmp, double* acc_sum,
                               double* acc_comp, int cap) {
  extern __shared__ __align__(16) unsigned char smem[];
  wait_for_previous_grid();
  const int2 task = tasks[blockIdx.x];
  const DiagLattice L = lat[task.x];
  const int n = L.Lz, Lx = L.Lx, H = sf_half(Lx), SS = sf_seq_stride(n);
  const int fld = task.y / Lx, qx0 = task.y - fld * Lx;
  const int cq = sf_col_strip(Lx, n, cap), w = min(cq, H - qx0);
  Cplx<real>* tw = reinterpret_cast<Cplx<real>*>(smem);
  Cplx<real>* s = tw + ((n >> 1) + 1);
  transform_columns<real, 16>(tmp + 4 * L.site_off + (int64_t)fld * H * n + qx0, H, n, w, tw, s);
  const int64_t base = 4 * L.site_off + (int64_t)fld * Lx * n + qx0;  // accumulators
  const int T = blockDim.x, total = w * n;
  const real scale = real(1) / ((real)Lx * (real)n);
  StripWalk k(w, T);
  for (int b0 = threadIdx.x; b0 < total; b0 += SfBatch<real>::cols * T) {
    double sm[SfBatch<real>::cols], cp[SfBatch<real>::cols];
    real pw[SfBatch<real>::cols];
    int64_t o[SfBatch<real>::cols];
#pragma unroll
    for (int i = 0; i < SfBatch<real>::cols; ++i) {
      if (b0 + i * T < total) {
        const Cplx<real> v = s[k.c * SS + k.j + (k.j >> 4)];
        pw[i] = (v.re * v.re + v.im * v.im) * scale;
        o[i] = base + (int64_t)k.j * Lx + k.c;
        sm[i] = acc_sum[o[i]];
        cp[i] = acc_comp[o[i]];
      }
      k.advance();
    }
#pragma unroll
    for (int i = 0; i < SfBatch<real>::cols; ++i) {
      if (b0 + i * T < total) {
        kahan_add(sm[i], cp[i], (double)pw[i]);
        acc_sum[o[i]] = sm[i];
        acc_comp[o[i]] = cp[i];
      }
    }
  }
}

// ---- power spectrum of one real field (one snapshot, written out, nothing accumulated) -----
// The sample step's transforms on one double-precision field, bound by the FP64 pipe (about 40
// instructions per point and dimension): two real rows per complex transform, so that only
// q_x = 0 .. Lx/2 goes through tmp and the column pass, which writes S(-q) = S(q) beside S(q).
// 2048 x 1024: 158 us (448 us with radix-2 passes over all Lx complex columns), 64 x 64: 6.8 us (8.2).
// The most threads ps_pass launches with PTS points each: a sequence of 4096 points (PTS 4) or 8192.
template <int PTS>
struct PsThreads {
  static constexpr int most = (PTS == 4 ? 4096 : 8192) / PTS;
  static_assert(most <= 1024, "a block cannot have more, and the compiler divides the registers by the bound");
};
template <int PTS>
__global__ void __launch_bounds__(PsThreads<PTS>::most) ps_rows_kernel(const double* __restrict__ phi, int Lx, int R,
                                                      Cplx<double>* __restrict__ tmp) {
  extern __shared__ __align__(16) unsigned char smem[];
  Cplx<double>* tw = reinterpret_cast<Cplx<double>*>(smem);
  const int64_t z0 = (int64_t)blockIdx.x * R;
  transform_rows<double, PTS>(phi + z0 * Lx, Lx, R, tmp + z0 * sf_half(Lx), tw, tw + ((Lx >> 1) + 1));
}

template <int PTS>
__global__ void __launch_bounds__(PsThreads<PTS>::most) ps_cols_kernel(const Cplx<double>* __restrict__ tmp, int Lx, int Lz, int cq,
                                                      double* __restrict__ out) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int n = Lz, H = sf_half(Lx), SS = sf_seq_stride(n), q0 = blockIdx.x * cq, w = min(cq, H - q0);
  Cplx<double>* tw = reinterpret_cast<Cplx<double>*>(smem);
  Cplx<double>* s = tw + ((n >> 1) + 1);
  transform_columns<double, PTS>(tmp + q0, H, n, w, tw, s);
  const int T = blockDim.x, total = w * n;
  const double scale = 1.0 / ((double)Lx * (double)n);
  StripWalk k(w, T);
  for (int b = threadIdx.x; b < total; b += T, k.advance()) {
    const Cplx<double> v = s[k.c * SS + k.j + (k.j >> 4)];
    const double p = (v.re * v.re + v.im * v.im) * scale;
    const int q = q0 + k.c;
    out[(int64_t)k.j * Lx + q] = p;
    if (q > 0 && 2 * q < Lx) out[(int64_t)((n - k.j) & (n - 1)) * Lx + Lx - q] = p;
  }
}

// One warp per lattice: lanes strided over the lattice's items, then a fixed butterfly, so the
// order of the sums is fixed (deterministic) and a lattice of many items costs a few loads per
// lane rather than one long chain.
__device__ __forceinline__ double warp_total(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ void finalize_lattices(int block, const DiagLattice* lat, int n_lat, const double* partials,
                                                  DiagStats* stats) {
  const int i = (int)((block * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (i >= n_lat) return;  // the whole warp
  const DiagLattice L = lat[i];
  double p = 0, ma = 0, mb = 0;
  for (int k = L.item_begin + lane; k < L.item_end; k += 32) {
    p += partials[3 * k];
    ma += partials[3 * k + 1];
    mb += partials[3 * k + 2];
  }
  p = warp_total(p);
  ma = warp_total(ma);
  mb = warp_total(mb);
  if (lane != 0) return;
  DiagStats st = stats[i];
  const double P = L.P_bg_mean + p / L.n_sites;
  st.P_last = P;
  neumaier_add(st.P_sum, st.P_comp, P);
  st.massA_last = L.mass_bg[0] + ma;
  st.massB_last = L.mass_bg[1] + mb;
  if (!isfinite(P) || !isfinite(st.massA_last) || !isfinite(st.massB_last)) st.nonfinite = 1;
  stats[i] = st;
}
__global__ void finalize_kernel(const DiagLattice* lat, int n_lat, const double* partials, DiagStats* stats) {
  finalize_lattices((int)blockIdx.x, lat, n_lat, partials, stats);
}

// Mass of the stored state of one lattice, both species at once.  Bound by memory in FP64 and by the
// FP64 pipe in FP32 (a conversion and an addition per value).  The blocks stride over the 16-byte
// groups of pairs, MASS_UNROLL loads in flight per thread, and the block that finishes last adds the
// block sums in order, so the result does not depend on which blocks ran when.  8192 x 2048 in FP32 (1.2 GB): 1.15 ms, 84.5 ms with one block per
// species; in FP64 (2.4 GB) 0.62 ms.
constexpr int MASS_THREADS = 256, MASS_UNROLL = 8;

// Block-wide sums of (a, b) in a fixed order, valid in thread 0.
__device__ __forceinline__ double2 block_total(double a, double b) {
  __shared__ double red[2][MASS_THREADS / 32];
  a = warp_total(a);
  b = warp_total(b);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();  // red may still be read for the previous sums
  if (lane == 0) {
    red[0][wid] = a;
    red[1][wid] = b;
  }
  __syncthreads();
  double2 t = make_double2(0.0, 0.0);
  if (threadIdx.x == 0)
    for (int w = 0; w < MASS_THREADS / 32; ++w) {
      t.x += red[0][w];
      t.y += red[1][w];
    }
  return t;
}

// The sums over species A and B of a 16-byte group of stored pairs.
__device__ __forceinline__ void add_group(const float4 v, double& a, double& b) {
  a += widen(v.x) + widen(v.z);
  b += widen(v.y) + widen(v.w);
}
__device__ __forceinline__ void add_group(const double2 v, double& a, double& b) {
  a += v.x;
  b += v.y;
}

// out: the two masses, then the block counter (zero before the call and left zero), then the block
// sums (MassBuf).
template <class real, class group>
__global__ void __launch_bounds__(MASS_THREADS) mass_kernel(const real* __restrict__ f, BgParams bp, double* out) {
  const int64_t n = 18 * (int64_t)bp.Lx * bp.Lz;
  constexpr int per = 16 / sizeof(real);  // values per group (an even number: whole pairs)
  const int64_t groups = n / per;
  const group* g = reinterpret_cast<const group*>(f);  // a lattice's block is 16-byte aligned
  double a = 0.0, b = 0.0;
  const int64_t stride = (int64_t)gridDim.x * MASS_THREADS;
  int64_t k = blockIdx.x * (int64_t)MASS_THREADS + threadIdx.x;
  for (; k + (MASS_UNROLL - 1) * stride < groups; k += MASS_UNROLL * stride) {
    group v[MASS_UNROLL];
#pragma unroll
    for (int i = 0; i < MASS_UNROLL; ++i) v[i] = __ldg(g + k + i * stride);
#pragma unroll
    for (int i = 0; i < MASS_UNROLL; ++i) add_group(v[i], a, b);
  }
  for (; k < groups; k += stride) add_group(__ldg(g + k), a, b);
  if (groups * per < n && blockIdx.x == 0 && threadIdx.x == 0) {  // an odd number of FP32 pairs
    a += (double)f[n - 2];
    b += (double)f[n - 1];
  }
  double2 t = block_total(a, b);
  unsigned* counter = reinterpret_cast<unsigned*>(out + 2);
  double2* sums = reinterpret_cast<double2*>(out + 4);
  __shared__ bool last;
  if (threadIdx.x == 0) {
    sums[blockIdx.x] = t;
    __threadfence();
    last = atomicAdd(counter, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  a = b = 0.0;
  for (int i = threadIdx.x; i < (int)gridDim.x; i += MASS_THREADS) {
    const double2 v = __ldcg(sums + i);
    a += v.x;
    b += v.y;
  }
  t = block_total(a, b);
  a = b = 0.0;
  if (bp.dev)
    for (int z = threadIdx.x; z < bp.Lz; z += MASS_THREADS) {
      const double c0 = 0.5 + (z + 0.5 - 0.5 * bp.Lz) * bp.grad_c0;
      a += bp.rho_bar * c0;
      b += bp.rho_bar * (1.0 - c0);
    }
  const double2 bg = block_total(a, b);
  if (threadIdx.x == 0) {
    out[0] = bg.x * bp.Lx + t.x;
    out[1] = bg.y * bp.Lx + t.y;
    *counter = 0;
  }
}

__device__ __forceinline__ double weight_of(int l) { return l == 0 ? 4.0 / 9.0 : (l <= 4 ? 1.0 / 9.0 : 1.0 / 36.0); }

__device__ __forceinline__ double background(const BgParams& bp, int s, int l, int z) {
  if (!bp.dev) return 0.0;
  const double c0 = 0.5 + (z + 0.5 - 0.5 * bp.Lz) * bp.grad_c0;
  return weight_of(l) * bp.rho_bar * (s == 0 ? c0 : 1.0 - c0);
}

// The API layout [species][link][z][x] (index k) against the stored pairs (state_index).
template <class real>
__global__ void to_absolute_kernel(const real* f, BgParams bp, double* out) {
  const int64_t LzLx = (int64_t)bp.Lx * bp.Lz, n = 18 * LzLx;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    const int sl = (int)(k / LzLx), s = sl / 9, l = sl - 9 * s;
    const int64_t r = k - sl * LzLx;
    const int z = (int)(r / bp.Lx);
    out[k] = (double)f[state_index(s, l, 0, 0, bp.Lx, LzLx) + 2 * r] + background(bp, s, l, z);
  }
}

template <class real>
__global__ void from_absolute_kernel(const double* in, BgParams bp, real* f) {
  const int64_t LzLx = (int64_t)bp.Lx * bp.Lz, n = 18 * LzLx;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    const int sl = (int)(k / LzLx), s = sl / 9, l = sl - 9 * s;
    const int64_t r = k - sl * LzLx;
    const int z = (int)(r / bp.Lx);
    f[state_index(s, l, 0, 0, bp.Lx, LzLx) + 2 * r] = (real)(in[k] - background(bp, s, l, z));
  }
}

// Rest state f^S_l = w_l rho_bar c^S_0(z) (stored as zero deviations in deviation mode).
template <class real>
__global__ void init_rest_kernel(real* f, BgParams bp) {
  const int64_t LzLx = (int64_t)bp.Lx * bp.Lz, n = 18 * LzLx;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    if (bp.dev) {
      f[k] = real(0);
    } else {  // element k of the stored pairs: species k mod 2 of pair k / 2
      const int64_t q = k >> 1;
      const int s = (int)(k & 1), l = (int)(q / LzLx);
      const int z = (int)((q - l * LzLx) / bp.Lx);
      const double c0 = 0.5 + (z + 0.5 - 0.5 * bp.Lz) * bp.grad_c0;
      f[k] = (real)(weight_of(l) * bp.rho_bar * (s == 0 ? c0 : 1.0 - c0));
    }
  }
}

// Columns x_first .. x_first + n - 1 of every (species, link) plane, to (TO_BUF) or from a packed
// buffer [9 * species + link][Lz][n] (the API layout).  A thread moves whole (A, B) pairs: one
// access of the state, one of each species' plane.  Wide ranges (WIDE): a block takes COL_TILE
// columns of one row (link, z), so the row is found once per block and every access of a warp is
// contiguous, four pairs in flight per thread; narrow ones (a halo of a few columns) run over the
// pairs in a row with the row found per pair.  All 8192 columns of 8192 x 2048 in FP32 (2.4 GB
// moved): 0.43 ms (5.6 TB/s), 1.63 ms with one value per thread and 64-bit divisions.
constexpr int COL_THREADS = 256, COL_TILE = 1024;

template <class real, bool TO_BUF>
__device__ __forceinline__ void move_pair(typename PairType<real>::type* g, real* pa, real* pb) {
  if (TO_BUF) {
    const typename PairType<real>::type v = *g;
    *pa = v.x;
    *pb = v.y;
  } else {
    typename PairType<real>::type v;
    v.x = *pa;
    v.y = *pb;
    *g = v;
  }
}

template <class real, bool TO_BUF, bool WIDE>
__global__ void __launch_bounds__(COL_THREADS)
    columns_kernel(typename PairType<real>::type* f, int Lx, int Lz, int x_first, int n, real* buf) {
  const int64_t plane = (int64_t)9 * Lz * n;  // species B's planes follow species A's
  if (WIDE) {
    const int tiles = (n + COL_TILE - 1) / COL_TILE;
    const int row = blockIdx.x / tiles, j0 = (blockIdx.x - row * tiles) * COL_TILE;  // row = link * Lz + z
    typename PairType<real>::type* g = f + (int64_t)row * Lx + x_first;
    real* b = buf + (int64_t)row * n;
#pragma unroll
    for (int i = 0; i < COL_TILE / COL_THREADS; ++i) {
      const int j = j0 + i * COL_THREADS + threadIdx.x;
      if (j < n) move_pair<real, TO_BUF>(g + j, b + j, b + plane + j);
    }
  } else {
    const unsigned k = blockIdx.x * COL_THREADS + threadIdx.x, row = k / (unsigned)n, j = k - row * n;
    if (row >= 9u * (unsigned)Lz) return;
    move_pair<real, TO_BUF>(f + (int64_t)row * Lx + x_first + j, buf + k, buf + plane + k);
  }
}

// ---- results on their way to the host ----------------------------------------------------------------
// A result, scaled (and mirrored, for spectra) on the device, and behind it the context's error flag, so
// that a read is one launch and one copy.  Separate copies of the sums, their compensations and the flag
// cost 10 us each: 32 lattices of 128 x 32, their
// spectra, correlations, profiles and pressures (256 reads): about 9 -> 6 ms.
__global__ void read_spectrum_kernel(const double* __restrict__ sum, const double* __restrict__ comp, int Lx, int Lz, int n,
                                     double inv, const int* __restrict__ err, double* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) out[n] = (double)*err;
  if (i >= n) return;
  // accumulated: q_x = 0 .. Lx/2 (Kahan sums: total = sum - comp); the rest by S(q) = S(-q)
  const int r = i / Lx, q = i - r * Lx;
  const bool own = q <= Lx / 2;
  const int64_t src = (int64_t)(own || r == 0 ? r : Lz - r) * Lx + (own ? q : Lx - q);
  out[i] = (sum[src] - comp[src]) * inv;
}

// out[i] = (a[i] + b[i]) inv, or a[i] inv without b.
__global__ void read_scaled_kernel(const double* __restrict__ a, const double* __restrict__ b, int n, double inv,
                                   const int* __restrict__ err, double* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) out[n] = (double)*err;
  if (i < n) out[i] = (b ? a[i] + b[i] : a[i]) * inv;
}

// Fused multiply-add throughput: eight independent chains per thread x <- x a + b (|a| < 1, so the
// values stay bounded), enough resident warps to fill every pipe; the sum keeps the chains live.
template <class T>
__global__ void fma_rate_kernel(T* out, int iters, T a, T b) {
  T x[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) x[k] = (T)(threadIdx.x + k) * (T)1e-6;
  for (int i = 0; i < iters; ++i) {
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = fma(x[k], a, b);
  }
  T sum = 0;
#pragma unroll
  for (int k = 0; k < 8; ++k) sum += x[k];
  out[blockIdx.x * blockDim.x + threadIdx.x] = sum;
}

}  // namespace

cudaError_t measure_fma_rate(bool fp64, double* flops_per_s) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const int threads = 256, blocks = 8 * sms, iters = fp64 ? 2048 : 16384;
  void* out = nullptr;
  e = cudaMalloc(&out, (size_t)threads * blocks * sizeof(double));
  if (e != cudaSuccess) return e;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  auto run = [&]() {
    if (fp64) fma_rate_kernel<double><<<blocks, threads>>>((double*)out, iters, 0.9999999, 1e-9);
    else fma_rate_kernel<float><<<blocks, threads>>>((float*)out, iters, 0.9999f, 1e-6f);
  };
  float best = 1e30f;
  if ((e = cudaEventCreate(&e0)) == cudaSuccess && (e = cudaEventCreate(&e1)) == cudaSuccess) {
    run();  // warm-up
    for (int r = 0; r < 5 && e == cudaSuccess; ++r) {
      cudaEventRecord(e0);
      run();
      cudaEventRecord(e1);
      e = cudaEventSynchronize(e1);
      float ms = 0;
      if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
      if (e == cudaSuccess) best = std::min(best, ms);
    }
  }
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  cudaFree(out);
  if (e == cudaSuccess) *flops_per_s = 2.0 * 8 * iters * (double)threads * blocks / (best * 1e-3);
  return e;
}

cudaError_t launch_read_spectrum(const double* sum, const double* comp, int Lx, int Lz, int n, double inv, const int* err,
                                 double* out, cudaStream_t s) {
  read_spectrum_kernel<<<n / 256 + 1, 256, 0, s>>>(sum, comp, Lx, Lz, n, inv, err, out);
  return cudaGetLastError();
}

cudaError_t launch_read_scaled(const double* a, const double* b, int n, double inv, const int* err, double* out,
                               cudaStream_t s) {
  read_scaled_kernel<<<n / 256 + 1, 256, 0, s>>>(a, b, n, inv, err, out);
  return cudaGetLastError();
}

template <class real>
cudaError_t launch_columns(real* f, int Lx, int Lz, int x_first, int n, real* buf, bool to_buf, cudaStream_t s) {
  auto* g = reinterpret_cast<typename PairType<real>::type*>(f);
  const int64_t rows = 9 * (int64_t)Lz, pairs = rows * n;  // fewer than 2^30 (lattice size limit)
  // the row split pays from half a block of columns on
  if (n >= COL_THREADS / 2) {
    const unsigned blocks = (unsigned)(rows * ((n + COL_TILE - 1) / COL_TILE));
    if (to_buf) columns_kernel<real, true, true><<<blocks, COL_THREADS, 0, s>>>(g, Lx, Lz, x_first, n, buf);
    else columns_kernel<real, false, true><<<blocks, COL_THREADS, 0, s>>>(g, Lx, Lz, x_first, n, buf);
  } else {
    const unsigned blocks = (unsigned)((pairs + COL_THREADS - 1) / COL_THREADS);
    if (to_buf) columns_kernel<real, true, false><<<blocks, COL_THREADS, 0, s>>>(g, Lx, Lz, x_first, n, buf);
    else columns_kernel<real, false, false><<<blocks, COL_THREADS, 0, s>>>(g, Lx, Lz, x_first, n, buf);
  }
  return cudaGetLastError();
}

template <class real>
cudaError_t prepare_sf(size_t smem_rows, size_t smem_cols) {
  cudaError_t e = cudaSuccess;
  if (sizeof(real) == 4) {
    fill_tw_table_kernel<<<(TW_TABLE + 255) / 256, 256>>>();
    e = cudaDeviceSynchronize();
  }
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(sf_rows_kernel<real>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_rows);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(sf_cols_kernel<real>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_cols);
}

template <class real>
cudaError_t launch_sf(const SfPlan& p, const real* fields, void* tmp, double* acc_sum, double* acc_comp,
                      cudaStream_t s) {
  launch_overlapped(p.overlap, sf_rows_kernel<real>, dim3(p.n_row_tasks), p.threads, p.smem_rows, s, p.lat, p.row_tasks,
                    fields, (Cplx<real>*)tmp, p.prof_sum, p.prof_comp, p.n_rows, p.cap);
  launch_overlapped(p.overlap, sf_cols_kernel<real>, dim3(p.n_col_tasks), p.threads, p.smem_cols, s, p.lat, p.col_tasks,
                    (const Cplx<real>*)tmp, acc_sum, acc_comp, p.cap);
  return cudaGetLastError();
}

cudaError_t launch_finalize(const DiagLattice* d_lat, int n_lat, const double* partials, DiagStats* stats,
                            cudaStream_t s) {
  finalize_kernel<<<(n_lat + 3) / 4, 128, 0, s>>>(d_lat, n_lat, partials, stats);  // 4 lattices per block
  return cudaGetLastError();
}

template <class real>
cudaError_t launch_mass(const real* f, const BgParams& bp, double* out, cudaStream_t s) {
  using group = typename std::conditional<sizeof(real) == 4, float4, double2>::type;
  const int64_t groups = 18 * (int64_t)bp.Lx * bp.Lz * (int64_t)sizeof(real) / 16;
  // four unrolled rounds per thread, up to MASS_BLOCKS blocks (eight per SM of a full chip)
  const int64_t want = groups / (4 * MASS_UNROLL * MASS_THREADS);
  const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>(want, MASS_BLOCKS));
  mass_kernel<real, group><<<blocks, MASS_THREADS, 0, s>>>(f, bp, out);
  return cudaGetLastError();
}

template <class real>
cudaError_t launch_to_absolute(const real* f, const BgParams& bp, double* out, cudaStream_t s) {
  to_absolute_kernel<real><<<1024, 256, 0, s>>>(f, bp, out);
  return cudaGetLastError();
}

template <class real>
cudaError_t launch_from_absolute(const double* in, const BgParams& bp, real* f, cudaStream_t s) {
  from_absolute_kernel<real><<<1024, 256, 0, s>>>(in, bp, f);
  return cudaGetLastError();
}

template <class real>
cudaError_t launch_init_rest(real* f, const BgParams& bp, cudaStream_t s) {
  init_rest_kernel<real><<<1024, 256, 0, s>>>(f, bp);
  return cudaGetLastError();
}

// One pass of the snapshot transforms over `seqs` sequences of n points.  A warp's FP64 instruction
// holds the SM's pipe for 16 clocks however few of its lanes work, so a small pass wants many threads
// of few points each (radix 4), a large one few passes through shared memory (radix 16).  Both passes,
// in us with 4 / 8 / 16 points per thread: 64 x 64 16.6 / 24.7 / 38.9, 512 x 256 24.7 / 32.9 / 51.4, 1024 x 256
// 35 / 35 / 53, 1024 x 512 61 / 55 / 62, 2048 x 1024 215 / 210 / 206, 2048 x 4096 918 / 788 / 757; the lines lie at
// 2^17 and 2^19 complex points of a pass.  Blocks are of 64 or 128 threads (the best at each size), a
// sequence that needs more takes a block of its own.
struct PsPass {
  int pts, threads, seqs;
  size_t smem;
};
static PsPass ps_pass(int n, int seqs) {
  PsPass p;
  const int64_t points = (int64_t)n * seqs;
  p.pts = points < (1 << 17) && n <= 4096 ? 4 : points < (1 << 19) ? 8 : 16;
  p.threads = std::max(p.pts == 8 ? 128 : 64, n / p.pts);
  p.seqs = std::min(seqs, p.pts * p.threads / n);
  p.smem = ((size_t)(n / 2 + 1) + (size_t)p.seqs * sf_seq_stride(n)) * sizeof(Cplx<double>);
  return p;
}
// The largest of them: one sequence of 8192 points and its twiddles (204,832 bytes of the 227 KB a
// block may opt in to).
constexpr size_t kPsSmemMax = (8192 / 2 + 1 + 8192 + 8192 / 16 + 1) * sizeof(Cplx<double>);

template <int PTS>
static cudaError_t prepare_ps() {
  cudaError_t e = cudaFuncSetAttribute(ps_rows_kernel<PTS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPsSmemMax);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(ps_cols_kernel<PTS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPsSmemMax);
}

cudaError_t prepare_power_spectrum() {  // attributes only: legal while a stream is captured
  cudaError_t e = prepare_ps<4>();
  if (e == cudaSuccess) e = prepare_ps<8>();
  if (e == cudaSuccess) e = prepare_ps<16>();
  return e;
}

template <int PTS>
static void launch_ps_rows(const PsPass& r, const double* field, int Lx, int Lz, void* tmp, cudaStream_t s) {
  // Lz/2 and r.seqs are powers of two: every block is full
  ps_rows_kernel<PTS><<<Lz / 2 / r.seqs, r.threads, r.smem, s>>>(field, Lx, 2 * r.seqs, (Cplx<double>*)tmp);
}
template <int PTS>
static void launch_ps_cols(const PsPass& c, const void* tmp, int Lx, int Lz, double* out, cudaStream_t s) {
  ps_cols_kernel<PTS><<<(sf_half(Lx) + c.seqs - 1) / c.seqs, c.threads, c.smem, s>>>((const Cplx<double>*)tmp, Lx, Lz, c.seqs, out);
}

cudaError_t launch_power_spectrum(const double* field, int Lx, int Lz, double* out, void* tmp, cudaStream_t s) {
  const PsPass r = ps_pass(Lx, Lz / 2), c = ps_pass(Lz, sf_half(Lx));
  if (r.pts == 4) launch_ps_rows<4>(r, field, Lx, Lz, tmp, s);
  else if (r.pts == 8) launch_ps_rows<8>(r, field, Lx, Lz, tmp, s);
  else launch_ps_rows<16>(r, field, Lx, Lz, tmp, s);
  if (c.pts == 4) launch_ps_cols<4>(c, tmp, Lx, Lz, out, s);
  else if (c.pts == 8) launch_ps_cols<8>(c, tmp, Lx, Lz, out, s);
  else launch_ps_cols<16>(c, tmp, Lx, Lz, out, s);
  return cudaGetLastError();
}

// z-profile of the pressure (Sec. III.C): warp r of the grid sums global row r of the sampled
// pressure over x in a fixed order (lane-strided partial sums in the working precision, four
// values at a time, then in double and a butterfly) and adds the row mean to the compensated sum.
template <class real>
__device__ __forceinline__ void profile_rows(int block, const DiagLattice* __restrict__ lat,
                                             const int* __restrict__ row_lat, int n_rows,
                                             const real* __restrict__ pfield, double* __restrict__ prof_sum,
                                             double* __restrict__ prof_comp) {
  const int r = (int)(((int64_t)block * blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (r >= n_rows) return;  // whole warps
  const DiagLattice& L = lat[row_lat[r]];
  const int Lx = L.Lx, z = r - L.row_off;
  const real* p0 = pfield + L.site_off + (int64_t)z * Lx;
  double acc = 0.0;
  if ((Lx & 3) == 0) {
    for (int x = lane * 4; x < Lx; x += 128) acc += (double)((p0[x] + p0[x + 1]) + (p0[x + 2] + p0[x + 3]));
  } else {
    for (int x = lane; x < Lx; x += 32) acc += (double)p0[x];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) neumaier_add(prof_sum[4 * (int64_t)n_rows + r], prof_comp[4 * (int64_t)n_rows + r], acc / (double)Lx);
}

// Real-space correlation of one sample: block (CORR_TILE^2 threads) per (lattice, field, z tile,
// z' tile); x runs in chunks of 32 staged in shared memory, each chunk's products summed in the
// working precision and the chunk sums in double.
template <class real>
__device__ __forceinline__ void corr_real_tile(int4 t, const DiagLattice* __restrict__ lat,
                                               const real* __restrict__ fields, double* __restrict__ R) {
  constexpr int T = CORR_TILE;
  __shared__ real a[32][T + 1], b[32][T + 1];
  const DiagLattice& L = lat[t.x];
  const int Lx = L.Lx, Lz = L.Lz, fld = t.y, z0 = t.z * T, zp0 = t.w * T;
  const int tz = threadIdx.x % T, tzp = threadIdx.x / T;
  const real* f = fields + 4 * L.site_off + (int64_t)fld * Lx * Lz;
  double acc = 0.0;
  for (int x0 = 0; x0 < Lx; x0 += 32) {
    for (int i = threadIdx.x; i < 32 * T; i += T * T) {
      const int xx = i & 31, zz = i >> 5, x = x0 + xx, z = z0 + zz, zp = zp0 + zz;
      a[xx][zz] = (x < Lx && z < Lz) ? f[(int64_t)z * Lx + x] : real(0);
      b[xx][zz] = (x < Lx && zp < Lz) ? f[(int64_t)zp * Lx + x] : real(0);
    }
    __syncthreads();
    real sum = 0;
#pragma unroll 8
    for (int xx = 0; xx < 32; ++xx) sum += a[xx][tz] * b[xx][tzp];
    acc += (double)sum;
    __syncthreads();
  }
  const int z = z0 + tz, zp = zp0 + tzp;
  if (z < Lz && zp < Lz) R[L.r_off + ((int64_t)fld * Lz + z) * Lz + zp] += acc / (double)Lx;
}

// Mode correlation of one sample: thread per (z, z') of a tile, from the row transforms
// X(q, z) = sum_x dphi(x, z) exp(-i q x) (unnormalised): C += conj(X(q, z)) X(q, z') / Lx.
template <class real>
__device__ __forceinline__ void corr_mode_tile(int4 t, const DiagLattice* __restrict__ lat,
                                               const int* __restrict__ modes, int n_modes,
                                               const Cplx<real>* __restrict__ tmp, double* __restrict__ C) {
  constexpr int T = CORR_TILE;
  const DiagLattice& L = lat[t.x];
  const int Lx = L.Lx, Lz = L.Lz, fld = t.y / n_modes, m = t.y - fld * n_modes, k = modes[m];
  const int z = t.z * T + (int)threadIdx.x % T, zp = t.w * T + (int)threadIdx.x / T;
  if (z >= Lz || zp >= Lz) return;
  const int H = sf_half(Lx);
  const Cplx<real>* X = tmp + 4 * L.site_off + (int64_t)fld * Lz * H;
  // q_x > Lx/2 from the conjugate symmetry of a real field's transform
  const int kk = k < H ? k : Lx - k;
  const double sg = k < H ? 1.0 : -1.0;
  const Cplx<real> u = X[(int64_t)z * H + kk], v = X[(int64_t)zp * H + kk];
  const double ur = u.re, ui = sg * (double)u.im, vr = v.re, vi = sg * (double)v.im, inv = 1.0 / (double)Lx;
  double* c = C + L.c_off + ((((int64_t)fld * n_modes + m) * Lz + z) * Lz + zp) * 2;
  c[0] += (ur * vr + ui * vi) * inv;
  c[1] += (ur * vi - ui * vr) * inv;
}

// What is left of a sample after the transforms, one launch: blocks of correlation tiles, of pressure
// rows and of lattices' statistics, which do not depend on one another (a launch each, they ran one after
// another).  The three launches of a sample overlap at their ends where the steps do.  400 steps of 32
// lattices of 128 x 32 in FP32 with 40 samples and their readouts: 11.9 -> 10.7 ms.
// What the launches before hand on comes without __restrict__, as everywhere where launches overlap: with const
// it would let the compiler read them as constant for the whole kernel, before the wait too.
constexpr int TAIL_THREADS = CORR_TILE * CORR_TILE;
template <class real>
__global__ void __launch_bounds__(TAIL_THREADS) sample_tail_kernel(SampleTail p, const real* fields, const real* pfield,
                                                                   const Cplx<real>* tmp) {
  wait_for_previous_grid();
  int b = (int)blockIdx.x;
  if (b < p.n_real_tasks) return corr_real_tile<real>(p.real_tasks[b], p.lat, fields, p.R);
  b -= p.n_real_tasks;
  if (b < p.n_mode_tasks) return corr_mode_tile<real>(p.mode_tasks[b], p.lat, p.modes, p.n_modes, tmp, p.C);
  b -= p.n_mode_tasks;
  if (b < p.row_blocks) return profile_rows<real>(b, p.lat, p.row_lat, p.n_rows, pfield, p.prof_sum, p.prof_comp);
  finalize_lattices(b - p.row_blocks, p.lat, p.n_lat, p.partials, p.stats);
}

template <class real>
cudaError_t launch_sample_tail(SampleTail p, const real* fields, const real* pfield, const void* tmp, cudaStream_t s) {
  constexpr int W = TAIL_THREADS / 32;  // rows and lattices per block
  p.row_blocks = (p.n_rows + W - 1) / W;
  const int blocks = p.n_real_tasks + p.n_mode_tasks + p.row_blocks + (p.n_lat + W - 1) / W;
  launch_overlapped(p.overlap, sample_tail_kernel<real>, dim3(blocks), TAIL_THREADS, 0, s, p, fields, pfield,
                    (const Cplx<real>*)tmp);
  return cudaGetLastError();
}

#define LB_INST(real)                                                                                        \
  template cudaError_t prepare_sf<real>(size_t, size_t);                                                     \
  template cudaError_t launch_sf<real>(const SfPlan&, const real*, void*, double*, double*, cudaStream_t);   \
  template cudaError_t launch_mass<real>(const real*, const BgParams&, double*, cudaStream_t);               \
  template cudaError_t launch_to_absolute<real>(const real*, const BgParams&, double*, cudaStream_t);        \
  template cudaError_t launch_from_absolute<real>(const double*, const BgParams&, real*, cudaStream_t);      \
  template cudaError_t launch_init_rest<real>(real*, const BgParams&, cudaStream_t);                         \
  template cudaError_t launch_columns<real>(real*, int, int, int, int, real*, bool, cudaStream_t);           \
  template cudaError_t launch_sample_tail<real>(SampleTail, const real*, const real*, const void*, cudaStream_t);
LB_INST(float)
LB_INST(double)

}  // namespace lbk

// FP64 transforms of rows in shared memory, computed in 64-bit fixed point.
//
// This part issues two FP64 operations per clock and SM against 128 integer ones, so a 243-point FP64 pass over the half
// spectrum of 243^3 took 438 us for a memory floor of 34 us, at 91% of the FP64 issue rate.  A row is scaled by a power of
// two and transformed with integer additions and 32 x 32 -> 64-bit multiply-adds; the conversions are integer operations
// on the bits of the doubles.
//
// Range: the scale brings the sum of the moduli of a row's components to at most 2^61 (1.06 times that with the parts the
// estimate drops), which bounds every intermediate and final value of the transform, whatever the passes.  The first pass
// is bounded by its own 2 p components, so its input has up to log2(N / p) more bits, dropped before the second (on long rows
// pass by pass): rounding the input to 2^-53 of the largest component would be the largest error.  Errors of a row are then a few units of 2^-61 of that
// sum, below FP64's rounding of the same transform: relative 2-norm errors against extended precision, random rows of 243,
// 729 and 2187 entries: FP64 3.6e-16, 4.3e-16, 4.9e-16, this 7.7e-17, 8.7e-17, 1.3e-16.  Rows are scaled one by one, so
// a small row keeps its own accuracy.
// Measured: 243-point passes over 243^3 438 -> 175 us, fused row pass 1078 -> 412 us, FP64 application 9.55 -> 3.83 ms,
// 105 x 147 x 75 anisotropic 0.93 -> 0.60 ms, Ga at 63^3 0.86 -> 0.50 ms.  The integer pipes bound it now (60% of their
// rate, about 580 instructions a point, 24 warps an SM); with the conversions unrolled into the butterflies instead of in
// loops of their own a pass took 30 us more, waiting for instructions.
// A row with an entry that is not finite becomes NaN as a whole.  Rows of up to 9 points stay in FP64 (fp64_rows).
#pragma once

namespace lrfg {

struct __align__(16) Fix2 {
  long long x, y;
};

constexpr int kFixMaxRows = 64;  // rows of a tile at most

// what the transforms of a kernel keep beside its tiles: 192 bytes, which leave a row of 3627 points, the longest of prime
// factors up to 31, its 64 bytes a point (static arrays of ints in each instantiation took up to 1.2 KB)
struct FixShared {
  unsigned short scale[kFixMaxRows];  // 16 top + room, see fix_rows
  int2 part[8];
};
__device__ __forceinline__ FixShared& fix_shared() {
  __shared__ FixShared s;
  return s;
}

// a * w with a = ah 2^31 + al, 0 <= al < 2^31, and w = wh 2^31 + wl, |wl| <= 2^30 (fixed_root), a factor times 2^62:
// a w / 2^62 = ah wh + (al wh + ah wl) / 2^31, with the product of the lower parts left out, at most half a unit and on average
// half of wl / 2^31; `mid` starts with the half that rounds its shift.
constexpr unsigned kFixHalf = 1u << 30;
__device__ __forceinline__ int fix_hi(long long a) {
  return (int)__funnelshift_r((unsigned)a, (unsigned)((unsigned long long)a >> 32), 31);
}
__device__ __forceinline__ int fix_lo(long long a) { return (int)((unsigned)a & 0x7fffffffu); }
// a b + c as one instruction (the compiler takes (long long)a * b for a 64 x 64 product where a comes from a shift: three)
__device__ __forceinline__ long long fix_mad(int a, int b, long long c) {
  long long d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
}
__device__ __forceinline__ long long fix_mul(int a, int b) {
  long long d;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(d) : "r"(a), "r"(b));
  return d;
}

__device__ __forceinline__ Fix2 operator+(Fix2 a, Fix2 b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ Fix2 operator-(Fix2 a, Fix2 b) { return {a.x - b.x, a.y - b.y}; }

// w = (x upper, x lower, y upper, y lower) of exp(-2 pi i j / N); SIGN > 0 multiplies by its conjugate.  With |a| <= 1.06 2^61
// and |w| <= 2^62 the sums of `mid` stay below 2^63: the two products of al and bl, each below 2^31, with w's upper parts are
// together at most sqrt 2 2^31 2^31, those of ah and bh with its lower parts at most 1.06 2^30 sqrt 2 2^30, 1.79 2^62 in all
// (2.16 2^62 with lower parts up to 2^31: one of some 10^4 rows with a single entry overflowed).
template <int SIGN>
__device__ __forceinline__ Fix2 fix_cmul(Fix2 a, int4 w) {
  const int ah = fix_hi(a.x), al = fix_lo(a.x), bh = fix_hi(a.y), bl = fix_lo(a.y);
  // re = a w_x - b w_y, im = b w_x + a w_y, or with the conjugate re = a w_x + b w_y, im = b w_x - a w_y
  const int ch = SIGN < 0 ? -bh : bh, cl = SIGN < 0 ? -bl : bl, dh = SIGN < 0 ? ah : -ah, dl = SIGN < 0 ? al : -al;
  const long long mr = fix_mad(cl, w.z, fix_mad(ch, w.w, fix_mad(al, w.x, fix_mad(ah, w.y, kFixHalf))));
  const long long mi = fix_mad(dl, w.z, fix_mad(dh, w.w, fix_mad(bl, w.x, fix_mad(bh, w.y, kFixHalf))));
  return {fix_mad(ch, w.z, fix_mad(ah, w.x, mr >> 31)), fix_mad(dh, w.z, fix_mad(bh, w.x, mi >> 31))};
}

// one component times a real factor (h, l)
__device__ __forceinline__ long long fix_rmul(long long a, int h, int l) {
  const int ah = fix_hi(a);
  return fix_mad(ah, h, fix_mad(fix_lo(a), h, fix_mad(ah, l, kFixHalf)) >> 31);
}

// a / 2^s rounded to nearest, 0 <= s < 32, half = 2^s / 2
__device__ __forceinline__ long long fix_shift(long long a, int s, unsigned half) {
  a += half;
  const int hi = (int)(a >> 32);
  return ((long long)(hi >> s) << 32) | __funnelshift_r((unsigned)a, (unsigned)hi, s);
}

// ---- conversions ------------------------------------------------------------------------------------------------
// bits of a double to fixed point in a row's scale c: times 2^(1101 - c), rounded to nearest
__device__ __forceinline__ long long fix_from_bits(unsigned long long u, int c) {
  const int e = (int)((unsigned)(u >> 52) & 0x7ffu);
  unsigned long long m = u & 0xfffffffffffffULL;
  m |= (unsigned long long)(e ? 1u : 0u) << 52;
  const int sh = c - 17 - (e > 1 ? e : 1);  // of the mantissa at bit 62, less the rounding bit: 1 <= sh
  m = (m << 10) >> (sh < 63 ? sh : 63);
  const long long v = (long long)((m + 1) >> 1);
  return (long long)u < 0 ? -v : v;
}

// v * 2^p as a double, rounded to nearest (ties away); no FP64 operation on the common path, not even a sign change
__device__ __forceinline__ double fix_to_double(long long v, int p) {
  const long long neg = v >> 63;
  unsigned long long a = (unsigned long long)((v ^ neg) - neg);
  const unsigned hi = (unsigned)(a >> 32);
  const int lz = __clz(hi ? hi : (unsigned)a) + (hi ? 0 : 32);  // 64 for 0
  a <<= lz & 63;
  const unsigned long long m = (a >> 11) + ((a >> 10) & 1ULL);  // 2^52 <= m <= 2^53
  const int e = p + 11 - lz + 1075;                // exponent field of m 2^(p + 11 - lz)
  const unsigned long long sign = (unsigned long long)neg & 0x8000000000000000ULL;
  if (e > 0 && e < 2046) return __longlong_as_double((long long)(a ? sign | (((unsigned long long)(e - 1) << 52) + m) : 0ULL));
  return a ? scalbn(neg ? -(double)m : (double)m, p + 11 - lz) : 0.0;  // subnormal or overflowing
}

// ---- butterflies ------------------------------------------------------------------------------------------------
template <int P, int SIGN>
struct FixDFT {  // odd prime P (5, 7) by the symmetric halves of the inputs, see RegDFT<7>
  static __device__ __forceinline__ void run(Fix2* x) {
    constexpr int h = (P - 1) / 2;
    Fix2 s[h], d[h];
    const Fix2 x0 = x[0];
    Fix2 sum = x0;
#pragma unroll
    for (int r = 0; r < h; ++r) {
      s[r] = x[r + 1] + x[P - 1 - r];
      d[r] = x[r + 1] - x[P - 1 - r];
      sum = sum + s[r];
    }
    x[0] = sum;
#pragma unroll
    for (int q = 1; q <= h; ++q) {
      Fix2 re = x0, u = {0, 0};
#pragma unroll
      for (int r = 0; r < h; ++r) {
        const int4 w = c_roots_x[RootOff<P>::v + (q * (r + 1)) % P];
        re = re + Fix2{fix_rmul(s[r].x, w.x, w.y), fix_rmul(s[r].y, w.x, w.y)};
        u = u + Fix2{fix_rmul(d[r].x, w.z, w.w), fix_rmul(d[r].y, w.z, w.w)};
      }
      // the forward sum (w_y = -sin), its conjugate coefficients for the inverse
      const Fix2 iu = SIGN < 0 ? Fix2{-u.y, u.x} : Fix2{u.y, -u.x};
      x[q] = re + iu;
      x[P - q] = re - iu;
    }
  }
};

template <int SIGN>
struct FixDFT<3, SIGN> {
  static __device__ __forceinline__ void run(Fix2* x) {
    const int4 w = c_roots_x[kRootOff3 + 1];  // its sine is negative
    const Fix2 t1 = x[1] + x[2], t2 = x[1] - x[2];
    const long long ux = fix_rmul(t2.x, w.z, w.w), uy = fix_rmul(t2.y, w.z, w.w);
    const Fix2 iu = SIGN < 0 ? Fix2{-uy, ux} : Fix2{uy, -ux};
    const Fix2 m = {x[0].x - (t1.x >> 1), x[0].y - (t1.y >> 1)};
    x[0] = x[0] + t1;
    x[1] = m + iu;
    x[2] = m - iu;
  }
};

template <int SIGN>
struct FixDFT<9, SIGN> {  // 3 x 3, see reg_dft_split
  static __device__ __forceinline__ void run(Fix2* x) {
    Fix2 y[3][3];
#pragma unroll
    for (int n1 = 0; n1 < 3; ++n1) {
      Fix2 t[3] = {x[n1], x[n1 + 3], x[n1 + 6]};
      FixDFT<3, SIGN>::run(t);
#pragma unroll
      for (int k2 = 0; k2 < 3; ++k2)
        y[n1][k2] = (n1 && k2) ? fix_cmul<SIGN>(t[k2], c_roots_x[kRootOff9 + n1 * k2]) : t[k2];
    }
#pragma unroll
    for (int k2 = 0; k2 < 3; ++k2) {
      Fix2 t[3] = {y[0][k2], y[1][k2], y[2][k2]};
      FixDFT<3, SIGN>::run(t);
#pragma unroll
      for (int k1 = 0; k1 < 3; ++k1) x[3 * k1 + k2] = t[k1];
    }
  }
};

// A row's scale at a pass: the largest component's plus min(room, lg) bits, lg = log2 of the components a sum of the pass has,
// rounded up, room that of the row's own sum.  A pass drops the bits between its and the one before's after its twiddles, so
// that both round once (nothing to drop: scale is null).
struct FixDrop {
  const unsigned short* scale;
  int before, now;
  __device__ __forceinline__ int bits(int row) const {
    const int room = scale[row] & 15;
    return min(room, now) - min(room, before);
  }
};

// One pass of radix P over nf rows from a into b.
template <int P, int SIGN>
__device__ __forceinline__ void fix_pass(const Fix2* __restrict__ a, Fix2* __restrict__ b, int nf, int ld, int N, int L,
                                         const int4* W, const FixDrop drop) {
  const int mp = N / (L * P);
  const int nb = N / P;
  const int total = nb * nf;
  const float inv_nb = 1.0f / (float)nb, inv_L = 1.0f / (float)L;
  for (int t = threadIdx.x; t < total; t += blockDim.x) {
    const int row = small_div(t, nb, inv_nb);
    const int bt = t - row * nb;
    const int c = small_div(bt, L, inv_L);
    const int f = bt - c * L;
    const Fix2* in = a + row * ld + c * L + f;
    Fix2* out = b + row * ld + c * L * P + f;
    Fix2 x[P];
#pragma unroll
    for (int r = 0; r < P; ++r) x[r] = in[r * mp * L];
    if (f) {
#pragma unroll
      for (int r = 1; r < P; ++r) x[r] = fix_cmul<SIGN>(x[r], W[f * r * mp]);
    }
    if (drop.scale) {
      const int s = drop.bits(row);
      const unsigned half = (1u << s) >> 1;
#pragma unroll
      for (int r = 0; r < P; ++r) x[r] = {fix_shift(x[r].x, s, half), fix_shift(x[r].y, s, half)};
    }
    FixDFT<P, SIGN>::run(x);
#pragma unroll
    for (int q = 0; q < P; ++q) out[q * L] = x[q];
  }
}

// a pass of a prime radix p > 7, by the symmetric halves of the inputs
template <int SIGN>
__device__ __noinline__ void fix_pass_prime(int p, const Fix2* __restrict__ a, Fix2* __restrict__ b, int nf, int ld, int N,
                                            int L, const int4* W, const FixDrop drop) {
  const int mp = N / (L * p), nb = N / p, total = nb * nf, h = (p - 1) / 2, step = N / p;
  const float inv_nb = 1.0f / (float)nb, inv_L = 1.0f / (float)L;
  for (int t = threadIdx.x; t < total; t += blockDim.x) {
    const int row = small_div(t, nb, inv_nb);
    const int bt = t - row * nb;
    const int c = small_div(bt, L, inv_L);
    const int f = bt - c * L;
    const Fix2* in = a + row * ld + c * L + f;
    Fix2* out = b + row * ld + c * L * p + f;
    const int sh = drop.scale ? drop.bits(row) : 0;
    const unsigned half = (1u << sh) >> 1;
    auto load = [&](int r) {
      Fix2 v = in[r * mp * L];
      if (r && f) v = fix_cmul<SIGN>(v, W[f * r * mp]);
      return Fix2{fix_shift(v.x, sh, half), fix_shift(v.y, sh, half)};
    };
    Fix2 s[kMaxGenericRadix / 2 + 1], d[kMaxGenericRadix / 2 + 1];
    const Fix2 x0 = load(0);
    Fix2 sum = x0;
    for (int r = 1; r <= h; ++r) {
      const Fix2 u = load(r), v = load(p - r);
      s[r] = u + v;
      d[r] = u - v;
      sum = sum + s[r];
    }
    out[0] = sum;
    for (int q = 1; q <= h; ++q) {
      Fix2 re = x0, im = {0, 0};
      int j = 0;
      for (int r = 1; r <= h; ++r) {
        j += q;
        if (j >= p) j -= p;
        const int4 w = W[j * step];
        re = re + Fix2{fix_rmul(s[r].x, w.x, w.y), fix_rmul(s[r].y, w.x, w.y)};
        im = im + Fix2{fix_rmul(d[r].x, w.z, w.w), fix_rmul(d[r].y, w.z, w.w)};
      }
      const Fix2 iu = SIGN < 0 ? Fix2{-im.y, im.x} : Fix2{im.y, -im.x};
      out[q * L] = re + iu;
      out[(p - q) * L] = re - iu;
    }
  }
}

// largest exponent field and sum of components, in units of 2^-17 of its power of two, over entries part * 32 + lane, ... of a
// row (18-bit mantissas); the warp's together in every lane
__device__ __forceinline__ int2 fix_scan(const double2* row, int N, int first, int step) {
  int e = 1, sum = 0;
  for (int n = first; n < N; n += step) {
    const double2 v = row[n];
    const int hx = __double2hiint(v.x) & 0x7fffffff, hy = __double2hiint(v.y) & 0x7fffffff;
    const int ex = max(hx >> 20, 1), ey = max(hy >> 20, 1), en = max(e, max(ex, ey));
    const int mx = ((hx & 0xfffff) | (hx >> 20 ? 0x100000 : 0)) >> 3, my = ((hy & 0xfffff) | (hy >> 20 ? 0x100000 : 0)) >> 3;
    sum = (sum >> min(en - e, 31)) + (mx >> min(en - ex, 31)) + (my >> min(en - ey, 31));
    e = en;
  }
  const int et = __reduce_max_sync(0xffffffff, e);
  return make_int2(et, __reduce_add_sync(0xffffffff, sum >> min(et - e, 31)));
}

// log2 of a row's sum in the scan's units above 18 bits, rounded up (the sum holds the largest component's mantissa, unless
// the row is zero or subnormal)
__device__ __forceinline__ int fix_room(int2 m) { return max(0, 14 - __clz(m.y)); }

__device__ __forceinline__ void fix_row(double2* row, int N, int first, int step, int c) {
  for (int n = first; n < N; n += step) {
    const ulonglong2 u = *reinterpret_cast<const ulonglong2*>(row + n);
    *reinterpret_cast<Fix2*>(row + n) = {fix_from_bits(u.x, c), fix_from_bits(u.y, c)};
  }
}

// Rows of one butterfly in FP64, a row a thread: converting them would take longer than the transform (90,000 rows of 3 points
// transformed in 21 us and under a multiplier in 20, in fixed point 57 and 68; of 9 points 40 and 46, 62 and 80; from 11
// points on fixed point is the faster, but for 15 in launches as large, 68 us against 51).
template <int P, int SIGN>
__device__ __forceinline__ void fp64_butterflies(const double2* __restrict__ a, double2* __restrict__ b, int nf, int ld) {
  for (int row = threadIdx.x; row < nf; row += blockDim.x) {
    double2 x[P];
#pragma unroll
    for (int r = 0; r < P; ++r) x[r] = a[row * ld + r];
    RegDFT<P, SIGN, double2>::run(x);
#pragma unroll
    for (int r = 0; r < P; ++r) b[row * ld + r] = x[r];
  }
}
template <int SIGN>
__device__ __noinline__ void fp64_rows(int N, const double2* a, double2* b, int nf, int ld) {
  switch (N) {
    case 3: fp64_butterflies<3, SIGN>(a, b, nf, ld); break;
    case 5: fp64_butterflies<5, SIGN>(a, b, nf, ld); break;
    case 7: fp64_butterflies<7, SIGN>(a, b, nf, ld); break;
    default: fp64_butterflies<9, SIGN>(a, b, nf, ld);
  }
}

// The transform of nf rows (double2 in, double2 out): see stockham_rows.  The conversions are loops of their own: unrolled
// into the butterflies they made the kernels wait for instructions (the largest stall of a 243-point pass).
template <int SIGN>
__device__ double2* fix_rows(double2* a, double2* b, int nf, int ld, const FftPlan& pl, const int4* W) {
  FixShared& sh = fix_shared();
  const int N = pl.N;
  if (N == 1 || nf <= 0) {
    __syncthreads();
    return a;
  }
  if (N <= 9) {
    fp64_rows<SIGN>(N, a, b, nf, ld);
    __syncthreads();
    return b;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int all = 31;  // above every room
  int lg = pl.nst == 1 ? all : 32 - __clz(2 * pl.radix[0] - 1);
  // a warp takes a row, or a part of one where rows are few
  const int parts = nf >= nw ? 1 : nw / nf;  // parts * nf <= nw <= 8 where rows are few
  const int part = warp % parts;
  for (int row = warp / parts; row < nf; row += nw / parts) {
    double2* const p = a + row * ld;
    int2 m = fix_scan(p, N, part * 32 + lane, 32 * parts);
    if (parts > 1) {
      if (lane == 0) sh.part[warp] = m;
      asm volatile("bar.sync %0, %1;" ::"r"(1 + row), "r"(32 * parts) : "memory");
      const int q0 = warp - part;
      for (int q = q0; q < q0 + parts; ++q) m.x = max(m.x, sh.part[q].x);
      m.y = 0;
      for (int q = q0; q < q0 + parts; ++q) m.y += sh.part[q].y >> min(m.x - sh.part[q].x, 31);
    }
    const int room = fix_room(m);
    if (lane == 0 && part == 0) sh.scale[row] = (unsigned short)((m.x + 18) << 4 | room);  // room <= 14
    fix_row(p, N, part * 32 + lane, 32 * parts, m.x + 18 + min(room, lg));
  }
  __syncthreads();
  Fix2 *x = reinterpret_cast<Fix2*>(a), *y = reinterpret_cast<Fix2*>(b);
  int L = 1;
  for (int s = 0; s < pl.nst; ++s) {
    const int p = pl.radix[s];
    FixDrop drop{nullptr, lg, lg};
    if (s > 0 && lg < all) {
      // rows of up to 600 entries gain little from a third scale
      drop.scale = sh.scale;
      drop.now = (N <= 600 || s == pl.nst - 1) ? all : 32 - __clz(2 * L * p - 1);
      lg = drop.now;
    }
    switch (p) {
      case 3: fix_pass<3, SIGN>(x, y, nf, ld, N, L, W, drop); break;
      case 5: fix_pass<5, SIGN>(x, y, nf, ld, N, L, W, drop); break;
      case 7: fix_pass<7, SIGN>(x, y, nf, ld, N, L, W, drop); break;
      case 9: fix_pass<9, SIGN>(x, y, nf, ld, N, L, W, drop); break;
      default: fix_pass_prime<SIGN>(p, x, y, nf, ld, N, L, W, drop);
    }
    __syncthreads();
    Fix2* tmp = x;
    x = y;
    y = tmp;
    L *= p;
  }
  double2* res = reinterpret_cast<double2*>(x);
  for (int row = warp / parts; row < nf; row += nw / parts) {
    const int top = sh.scale[row] >> 4, c = top + (sh.scale[row] & 15) - 1101;
    for (int n = part * 32 + lane; n < N; n += 32 * parts) {
      const Fix2 v = x[row * ld + n];
      const double nan = __longlong_as_double(0x7ff8000000000000LL);
      res[row * ld + n] = top == 0x7ff + 18 ? make_double2(nan, nan) : make_double2(fix_to_double(v.x, c), fix_to_double(v.y, c));
    }
  }
  __syncthreads();
  return res;
}

}  // namespace lrfg

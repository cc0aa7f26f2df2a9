// Element kernel of Hbar psibar (Eqs. 15, 21) in fixed point with a float tail (fixed.cuh):
// the FP64 applications, single-system and batched.
//
// What bounds it.  The FP64 pipe of GB300 (2 operations per clock and SM) held the FP64
// contractions to 0.63 T FMA/s.  Here the nine contractions run on the integer and FP32
// pipes; the FP64 pipe only scales the gathered values (one multiplication each) and
// forms the results (two additions each).
//
// Operator.  With B' = W^1/2 B (rows scaled by the square roots of the Gauss weights) and
// K' = W^-1/2 Kq W^-1/2 the element form of elements.cu is
//   (B'^T)^(x)3 [ cx K' (x) I (x) I + cy I (x) K' (x) I + cz I (x) I (x) K' + J V ] B'^(x)3,
// without pointwise weights.  The row sums of |B'| are at most 1 for every degree, so the
// forward values keep the input's bound |V| < 2^kFxBits; the middle operator is scaled by a
// power of two per element, 2^er > max|J V| + (cx + cy + cz) max row sum |K'|, so that its
// values keep it too.  B' and B'^T are kernel parameters; the three scaled K' tables of an
// element are built in shared memory once per CTA.
//
// Layout: one P1 x P1 thread plane per element, real lines, the real and the imaginary
// part one after the other, the next orbital's columns copied to shared memory meanwhile.
// The largest value of an element's part (real or imaginary) sets its exponent: one integer
// maximum over the element's threads.  (With one exponent for both, the imaginary part of an
// orbital after a weak kick kept only the bits that the real part left.)  Measured per
// application of 16 orbitals on 16^3 elements, p = 6: 4.62 ms with FP64 contractions (95 % of the
// FP64 pipe), 1.43 ms here (8300 instructions per warp and orbital at 50 % issue activity, wide
// multiply-adds 42 % of their pipe, two CTAs of 128 registers per SM); 1.38 ms while the inputs'
// bits below the unit were dropped and the values not raised.  Three CTAs per SM (80 registers,
// spills) or smaller CTAs were slower (1.70, 1.53 ms).  A non-finite input or potential makes the
// results of its element NaN.  The scale s_j of a Krylov vector is left out here and applied by
// the assembly (and to alpha), so results are those of V_j.
#include "elements.cuh"
#include "fixed.cuh"

using namespace tdks;

namespace {

// Tables passed as a kernel parameter.
template <int P1>
struct FxTab {
  static constexpr int CS = FxOp<P1>::CS, KS = FxOp<P1>::KS;
  FxC c[2 * CS];        // folded B', then B'^T
  float k[2 * KS];      // their tail constants
  const double* dK;     // folded K' (device): leading parts, then the rest
  double kinf;          // largest row sum of |K'|
  double iw[P1];        // 1 / Gauss weight
};

// B' and B'^T in shared memory from p = 6 on (with constant-bank operands the compiler
// keeps them in registers and spills), the J V limbs in shared memory up to p = 6 and in
// registers above (shared memory for two CTAs per SM)
template <int P1>
constexpr bool kFxBs = P1 >= 7;
template <int P1>
constexpr bool kFxVs = P1 <= 7;

// Dynamic shared memory of E elements: the three scaled K' tables and their tail
// constants, the integer lines, the float tails (both in SplitLayout), the prefetch buffer
template <int P1>
struct FxSmem {
  static constexpr int CS = FxOp<P1>::CS, KS = FxOp<P1>::KS, P2 = P1 * P1;
  static constexpr int ES = SplitLayout<P1, double>::ES, EF = SplitLayout<P1, float>::ES;
  __host__ __device__ static size_t kc(int E) { return (size_t)E * 3 * CS * sizeof(FxC); }
  __host__ __device__ static size_t lines(int E) { return (kc(E) + (size_t)E * 3 * KS * sizeof(float) + 15) & ~size_t(15); }
  __host__ __device__ static size_t tails(int E) { return lines(E) + (size_t)E * ES * sizeof(long long); }
  __host__ __device__ static size_t pf(int E) { return pf_offset(tails(E) + (size_t)E * EF * sizeof(float)); }
  __host__ __device__ static size_t vx(int E) { return pf(E) + (size_t)E * P2 * P1 * sizeof(double2); }
  static size_t bytes(int E) { return vx(E) + (kFxVs<P1> ? (size_t)E * P2 * P1 * sizeof(FxL) : 0); }
};

constexpr int kAcc = 8;   // integer accumulators of u . r of an element's part (24-bit limbs)

__device__ __forceinline__ int exp_field(double x) { return (int)(((unsigned)__double2hiint(x) >> 20) & 0x7ffu); }

// Integer and tail of a line as 62-bit integers: shifted left by the line's free bits (at
// most 19; |f| < 8; returned), the tail rounded to the new unit by adding 1.5 2^(23 - s)
template <int P1>
__device__ __forceinline__ int fx_join(long long (&t)[P1], const float (&tf)[P1]) {
  unsigned big = 0;
#pragma unroll
  for (int q = 0; q < P1; ++q) {
    const int hw = (int)(t[q] >> 32);
    big |= (unsigned)(hw ^ (hw >> 31));
  }
  const int s = min(__clz((int)big + 2) - 2, 19);
  const int mg = 0x4b400000 - (s << 23);
#pragma unroll
  for (int q = 0; q < P1; ++q) t[q] = (t[q] << s) + (__float_as_int(tf[q] + __int_as_float(mg)) - mg);
  return s;
}

// Elements [eidx] of the calling rows for the orbitals o_begin <= o < o_end that orb(o, in, sc)
// accepts; element results (of V_j, not q_j) to ev, orbital stride ev_ostride entries,
// alpha partials (times sc^2) to part.  sV, sM[4], sR[2] and sA (a set per element and
// part) are zero and synchronized on entry.
// kPair: rows 2 e and 2 e + 1 of the block share element e, one takes the real parts, the
// other the imaginary parts (each with its own lines and tables); the results are the same.
template <int P1, bool kPair, class OrbFn>
__device__ __forceinline__ void hbar_elem_fx(const Geom& g, const FxTab<P1>& tab, FxC* sK, float* sKk, long long* S1,
                                             float* F1,
                                             int* sA, int* sE, unsigned* sV, unsigned* sM, unsigned* sR, int sm_stride,
                                             const double* __restrict__ vks, long long eidx, int o_begin, int o_end,
                                             OrbFn orb, double2* __restrict__ ev, long long ev_ostride, double* part,
                                             int64_t part_stride, long long pslot, double2* __restrict__ pfbuf) {
  constexpr bool kVs = kFxVs<P1>, kBs = kFxBs<P1>;
  FxL* const vs = reinterpret_cast<FxL*>(pfbuf + (size_t)blockDim.x * blockDim.y * P1);
  constexpr int P2 = P1 * P1, P3 = P2 * P1, CS = FxTab<P1>::CS, KS = FxTab<P1>::KS;
  constexpr int LS = SplitLayout<P1, double>::LS, PS = SplitLayout<P1, double>::PS;
  constexpr int LF = SplitLayout<P1, float>::LS, PF = SplitLayout<P1, float>::PS;
  long long* S2 = S1 + P1 * PS;
  float* F2 = F1 + P1 * PF;
  const int u = threadIdx.x % P1, v = threadIdx.x / P1, el = threadIdx.y;
  const int tid = threadIdx.x + blockDim.x * threadIdx.y;
  const int nthr = blockDim.x * blockDim.y;
  // lanes of this warp that work on the same element, and the lane that speaks for them
  const unsigned grp = __match_any_sync(__activemask(), el);
  const bool lead = (tid & 31) == __ffs(grp) - 1;
  int ex = 0, ey = 0, ez = 0;
  const bool valid = plain_elem(g, eidx, ex, ey, ez);
  double cd[3] = {0.0, 0.0, 0.0}, bound = 1.0, scale = 0.0;
  FxL vx[kVs ? 1 : P1];
  int er = 0;
  {
    double vj[P1];
    unsigned vm = 0;
#pragma unroll
    for (int q = 0; q < P1; ++q) vj[q] = 0.0;
    if (valid) {
      const double hx = g.brk[0][ex + 1] - g.brk[0][ex];
      const double hy = g.brk[1][ey + 1] - g.brk[1][ey];
      const double hz = g.brk[2][ez + 1] - g.brk[2][ez];
      const double J = 0.125 * hx * hy * hz;
      cd[0] = 0.25 * hy * hz * g.ih[0][ex];
      cd[1] = 0.25 * hx * hz * g.ih[1][ey];
      cd[2] = 0.25 * hx * hy * g.ih[2][ez];
      const double* vp = vks + eidx * P3 + v * P2 + u * P1;   // x-line (qy = u, qz = v)
#pragma unroll
      for (int q = 0; q < P1; ++q) {
        vj[q] = vp[q] * J;
        vm = max(vm, (unsigned)__double2hiint(vj[q]) & 0x7fffffffu);
      }
    }
    vm = __reduce_max_sync(grp, vm);
    if (lead) atomicMax(&sV[el], vm);
    __syncthreads();
    if (valid) {
      // the margin keeps every coefficient below 1 after rounding
      bound = (tab.kinf * (cd[0] + cd[1] + cd[2]) + __hiloint2double((int)sV[el], -1)) * 1.0000001;
      er = max(exp_field(bound) - 1022, -900);
      scale = pow2(63 - er);
      for (int i = threadIdx.x; i < 3 * CS; i += P2)
        sK[i] = fx_coef(fx_scaled(i < CS ? cd[0] : (i < 2 * CS ? cd[1] : cd[2]), tab.dK[i % CS], tab.dK[CS + i % CS], scale));
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 3 * KS; i += P2)
      sKk[i] = fx_tail_const<P1>([&](int j) { return sK[(i / KS) * CS + j]; }, i % KS);
#pragma unroll
    for (int q = 0; q < P1; ++q) {
      const FxC w = fx_coef(__double2ll_rn(vj[q] * scale));
      if constexpr (kVs) vs[q * nthr + tid] = FxL{w.h, w.l};
      else vx[q] = FxL{w.h, w.l};
    }
  }
  const bool bad = !(fabs(bound) < INFINITY);   // non-finite potential
  // gather: z-column (a = u, b = v) with its Loewdin scales
  const long long plane = (long long)g.nix * g.niy;
  const int Ig = ex * g.p + u, Jg = ey * g.p + v;
  const bool inG = valid && Ig >= 1 && Ig <= g.nix && Jg >= 1 && Jg <= g.niy;
  const long long baseG = inG ? (long long)(Ig - 1) + (long long)g.nix * (Jg - 1) : 0;
  const double sxy = inG ? g.s[0][Ig] * g.s[1][Jg] : 0.0;
  const double* const sz = g.s[2] + ez * g.p;
  auto issue = [&](const double2* src_base) {   // zero-filled outside the interior
#pragma unroll
    for (int c = 0; c < P1; ++c) {
      const int K = ez * g.p + c;
      const bool ok = inG && K >= 1 && K <= g.niz;
      const double2* src = ok ? src_base + baseG + plane * (K - 1) : src_base;
      const unsigned sa = (unsigned)__cvta_generic_to_shared(pfbuf + c * nthr + tid);
      asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;\n" ::"r"(sa), "l"(src), "r"(ok ? 16 : 0)
                   : "memory");
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  __shared__ FxC sB[kBs ? 2 * CS : 1];
  if (kBs) {
    for (int i = tid; i < 2 * CS; i += nthr) sB[i] = tab.c[i];
    __syncthreads();
  }
  int o = o_begin, it = 0, rb = 0;
  double sc = 1.0;
  {
    const double2* in0 = nullptr;
    while (o < o_end && !orb(o, in0, sc)) ++o;
    if (o < o_end) issue(in0);
  }
  const auto cB = [&](int i) { return kBs ? sB[i] : tab.c[i]; };
  const auto cBT = [&](int i) { return kBs ? sB[CS + i] : tab.c[CS + i]; };
  const auto kB = [&](int i) { return tab.k[i]; };
  const auto kBT = [&](int i) { return tab.k[KS + i]; };
  while (o < o_end) {
    int on = o_end;
    double sc_n = 1.0;
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    // scaled column, back into the thread's own buffer slots; maxima of the parts
    unsigned mx[2] = {0, 0};
#pragma unroll
    for (int c = 0; c < P1; ++c) {
      double2 w = pfbuf[c * nthr + tid];
      const double f = sxy * __ldg(sz + c);   // (the buffer holds 0 outside the interior)
      w.x *= f;
      w.y *= f;
      mx[0] = max(mx[0], (unsigned)__double2hiint(w.x) & 0x7fffffffu);
      mx[1] = max(mx[1], (unsigned)__double2hiint(w.y) & 0x7fffffffu);
      pfbuf[c * nthr + tid] = w;
    }
    // sM[2 (orbital parity) + part]: zeroed one orbital ahead, after the barrier that follows
    // the last read
    unsigned* const sm = sM + 2 * (it & 1) * sm_stride + el;
    unsigned* const sm_next = sM + 2 * ((it & 1) ^ 1) * sm_stride + el;
    if (kPair) {
      const unsigned r = __reduce_max_sync(grp, el & 1 ? mx[1] : mx[0]);
      if (lead) atomicMax(sm, r);
    } else {
      const unsigned r0 = __reduce_max_sync(grp, mx[0]), r1 = __reduce_max_sync(grp, mx[1]);
      if (lead) {
        atomicMax(sm, r0);
        atomicMax(sm + sm_stride, r1);
      }
    }
    __syncthreads();
    if (threadIdx.x == 0) sm_next[0] = sm_next[sm_stride] = 0;
    ++it;
    double2* evo = ev + (long long)o * ev_ostride + eidx * P3 + v * P2 + u * P1;
#pragma unroll 1
    for (int comp = kPair ? el & 1 : 0; comp < 2; comp += kPair ? 2 : 1) {   // real part, then imaginary part
      int eb = (int)(sm[kPair ? 0 : comp * sm_stride] >> 20);
      const bool poison = bad || eb == 2047;
      eb = eb < 64 ? 64 : (eb > 2046 ? 2046 : eb);
      // V = y 2^sh, sh = kFxBits - (eb - 1022); element results = V 2^(er - sh), less the raise
      const int e0 = er + 7 - kFxBits + eb - 1022;
      long long col[P1], t[P1];
      float cf[P1], tf[P1];
#pragma unroll
      for (int c = 0; c < P1; ++c) {
        const uint2 w = reinterpret_cast<const uint2*>(pfbuf + c * nthr + tid)[comp];
        col[c] = fx_from_bits(w.y, w.x, eb, cf[c]);
      }
      if (kPair || comp == 1) {   // the thread's slots are free: the next active orbital's column
        const double2* in_n = nullptr;
        on = o + 1;
        while (on < o_end && !orb(on, in_n, sc_n)) ++on;
        if (on < o_end) issue(in_n);
      }
      // stage outputs: to a line of the integer and the tail array, in place
      const auto to = [](long long* S, int stride, float* F, int fstride) {
        return [=](int q, long long x, float xf) {
          S[q * stride] = x;
          F[q * fstride] = xf;
        };
      };
      long long* const Sz = S1 + v * LS + u;
      float* const Fz = F1 + v * LF + u;
      long long *const Sy = S1 + v * PS + u, *const Ry = S2 + v * PS + u;
      float *const Fy = F1 + v * PF + u, *const Gy = F2 + v * PF + u;
      long long *const Sx = S1 + v * PS + u * LS, *const Rx = S2 + v * PS + u * LS;
      float *const Fx = F1 + v * PF + u * LF, *const Gx = F2 + v * PF + u * LF;
      fx_apply<P1>(cB, kB, col, cf, to(Sz, PS, Fz, PF));
      __syncthreads();
      load_line(col, Sy, LS);
      load_line(cf, Fy, LF);
      unsigned big = 0;
      fx_apply<P1>(cB, kB, col, cf, [&](int q, long long x, float xf) {
        Ry[q * LS] = x;
        Gy[q * LF] = xf;
        big |= fx_magnitude(x);
      });
      // the part raised by its free bits: a vector with one large entry loses three bits per
      // contraction, and the middle operator's bound takes up to ten more
      big = __reduce_or_sync(grp, big);
      if (lead) atomicOr(&sR[rb * sm_stride + el], big);
      __syncthreads();
      const int up = fx_free_bits(sR[rb * sm_stride + el]);
      rb ^= 1;
      if (threadIdx.x == 0) sR[rb * sm_stride + el] = 0;   // last read a part ago, several barriers back
      const int eo = e0 - up;
      const int ec = eo < -980 ? -980 : (eo > 900 ? 900 : eo);
      const int slot = kPair ? el : 2 * el + comp;         // of the alpha sums
      load_line(col, Rx, 1);
      load_line(cf, Gx, 1);
#pragma unroll
      for (int q = 0; q < P1; ++q) fx_raise(col[q], cf[q], up);
      fx_apply<P1>(cB, kB, col, cf, [&](int q, long long x, float xf) {   // U (Gauss-point values)
        t[q] = x;
        tf[q] = xf;
        Sx[q] = x;
        Fx[q] = xf;
      });
      fx_apply<P1>([&](int i) { return sK[i]; }, [&](int i) { return sKk[i]; }, t, tf,
                   [&](int q, long long x, float xf) {                    // R = J V U + cx K'_x U
                     FxL wl;
                     if constexpr (kVs) wl = vs[q * nthr + tid];
                     else wl = vx[q];
                     const FxC w{wl.h, wl.l, (float)wl.h * 0x1p-32f, (float)wl.l * 0x1p-32f};
                     const FxV y = fx_operand(t[q] + kFxHalf, tf[q]);
                     FxDot d;
                     d.term(w, y);
                     d.close(fmaf(w.cl, -1.5f, -1.5f));
                     d.top(w, y);
                     Rx[q] = x + d.hi;
                     Gx[q] = xf + d.f;
                   });
      __syncthreads();
      load_line(col, Sy, LS);
      load_line(cf, Fy, LF);
      fx_apply<P1>([&](int i) { return sK[CS + i]; }, [&](int i) { return sKk[KS + i]; }, col, cf,
                   [&](int q, long long x, float xf) {                    // R += cy K'_y U
                     Ry[q * LS] += x;
                     Gy[q * LF] += xf;
                   });
      __syncthreads();
      load_line(col, Sz, PS);
      load_line(cf, Fz, PF);
      {
        const long long* const Rz = S2 + v * LS + u;
        const float* const Gz = F2 + v * LF + u;
        FxInner ur;
        fx_apply<P1>([&](int i) { return sK[2 * CS + i]; }, [&](int i) { return sKk[2 * KS + i]; }, col, cf,
                     [&](int q, long long x, float xf) {                  // r = R + cz K'_z U, and u r
                       x += Rz[q * PS];
                       t[q] = x;
                       tf[q] = xf + Gz[q * PF];
                       ur.add(col[q], Fz[q * PF], x, tf[q]);
                     });
        if (part) {   // the element's sum: 24-bit limbs, added over its lanes and warps
          const long long dh = ur.dh, dm = ur.dm + __float2ll_rn(ur.da), dl = ur.dl;
          const int lim[kAcc] = {(int)(dl & 0xffffff), (int)((dl >> 24) & 0xffffff), (int)(dl >> 48),
                                 (int)(dm & 0xffffff), (int)((dm >> 24) & 0xffffff), (int)(dm >> 48),
                                 (int)(dh & 0xffffff), (int)(dh >> 24)};
#pragma unroll
          for (int i = 0; i < kAcc; ++i) {
            const int w = __reduce_add_sync(grp, lim[i]);
            if (lead) atomicAdd(&sA[kAcc * slot + i], w);
          }
          if (threadIdx.x == 0) sE[slot] = poison ? 1 << 30 : er + 2 * (7 - (kFxBits - eb + 1022)) - 7 - 2 * up;
        }
      }
      // backward z (on the thread's own z-line), y, x
      fx_apply<P1>(cBT, kBT, t, tf, to(Sz, PS, Fz, PF));
      __syncthreads();
      load_line(col, Sy, LS);
      load_line(cf, Fy, LF);
      fx_apply<P1>(cBT, kBT, col, cf, to(Ry, LS, Gy, LF));
      __syncthreads();
      load_line(col, Rx, 1);
      load_line(cf, Gx, 1);
      fx_apply<P1>(cBT, kBT, col, cf, [&](int q, long long x, float xf) {
        t[q] = x;
        tf[q] = xf;
      });
      const int es = (ec - fx_join<P1>(t, tf)) << 20;
      if (valid) {
        double* dst = reinterpret_cast<double*>(evo) + comp;
        if (poison || eo != ec) {   // rare: non-finite, or results near the ends of the FP64 range
          const double f = poison ? __hiloint2double(0x7ff80000, 0) : pow2(eo - ec);
#pragma unroll
          for (int a = 0; a < P1; ++a)
            dst[2 * a] = fx_to_double(t[a], es) * f;
        } else {
#pragma unroll
          for (int a = 0; a < P1; ++a) dst[2 * a] = fx_to_double(t[a], es);
        }
      }
    }
    // alpha partial: first warp, one element per lane; two barriers after the sums were
    // written, and at least three before the next orbital adds to them
    if (part && tid < 32) {
      double s = 0.0;
      const int ne = (int)blockDim.y >> (kPair ? 1 : 0);
      for (int e = tid; e < ne; e += 32)
        for (int c = 2 * e; c < 2 * e + 2; ++c) {   // real part, imaginary part
          int A[kAcc];
#pragma unroll
          for (int i = 0; i < kAcc; ++i) {
            A[i] = sA[kAcc * c + i];
            sA[kAcc * c + i] = 0;
          }
          const long long l = (unsigned)A[0] + ((long long)(unsigned)A[1] << 24) + ((long long)A[2] << 48);
          const long long m = (unsigned)A[3] + ((long long)(unsigned)A[4] << 24) + ((long long)A[5] << 48);
          const long long h = (unsigned)A[6] + ((long long)A[7] << 24);
          const int x = sE[c];
          const double d = fma((double)h, 0x1p64, fma((double)m, 0x1p32, (double)l * 0x1p10));
          s += x == 1 << 30 ? __hiloint2double(0x7ff80000, 0) : d * pow2(x / 2) * pow2(x - x / 2);
        }
      const int nl = nthr < 32 ? nthr : 32;
      const unsigned mask = nl == 32 ? 0xffffffffu : (1u << nl) - 1u;
      for (int off = 16; off > 0; off >>= 1) {
        const double w = __shfl_down_sync(mask, s, off);
        if (tid + off < nl) s += w;
      }
      if (tid == 0) part[(long long)o * part_stride + pslot] = s * sc * sc;
    }
    o = on;
    sc = sc_n;
  }
}

template <int P1, bool kPair>
__global__ void __launch_bounds__(256, 2) k_hbar_fx(Geom g, const __grid_constant__ FxTab<P1> tab,
                                                    const double* __restrict__ vks, ApplyArgs a, int orb_per_cta,
                                                    double2* __restrict__ ev) {
  constexpr int P3 = P1 * P1 * P1, ES = SplitLayout<P1, double>::ES, CS = FxTab<P1>::CS;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int sA[2 * kAcc * Cfg<P1>::E], sE[2 * Cfg<P1>::E];
  __shared__ unsigned sV[Cfg<P1>::E], sM[4 * Cfg<P1>::E], sR[2 * Cfg<P1>::E];
  const int o0 = blockIdx.y * orb_per_cta;
  const int o1 = min(o0 + orb_per_cta, a.n_orb);
  if (a.kry) {   // a CTA whose orbitals have all left the recurrence skips the element set-up
    bool any = false;
    for (int o = o0; o < o1 && !any; ++o) any = a.kry[o].status == KRY_ACTIVE;
    if (!any) return;
  }
  const int tid = threadIdx.x + blockDim.x * threadIdx.y;
  const int nthr = blockDim.x * blockDim.y;
  for (int i = tid; i < 2 * kAcc * Cfg<P1>::E; i += nthr) sA[i] = 0;
  for (int i = tid; i < 2 * Cfg<P1>::E; i += nthr) {
    sV[i % Cfg<P1>::E] = 0;
    sM[i] = sM[2 * Cfg<P1>::E + i] = sR[i] = 0;
  }
  __syncthreads();
  auto orb = [&](int o, const double2*& in, double& sc) -> bool {
    if (a.kry) {
      if (a.kry[o].status != KRY_ACTIVE) return false;
      sc = a.kry[o].s[a.kj];
    }
    in = a.in_base + (long long)o * a.in_stride;
    return true;
  };
  hbar_elem_fx<P1, kPair>(g, tab, reinterpret_cast<FxC*>(smem) + threadIdx.y * 3 * CS,
                          reinterpret_cast<float*>(smem + FxSmem<P1>::kc(blockDim.y)) + threadIdx.y * 3 * FxTab<P1>::KS,
                          reinterpret_cast<long long*>(smem + FxSmem<P1>::lines(blockDim.y)) + (size_t)threadIdx.y * ES,
                          reinterpret_cast<float*>(smem + FxSmem<P1>::tails(blockDim.y)) +
                              (size_t)threadIdx.y * SplitLayout<P1, float>::ES,
                          sA, sE, sV, sM, sR, Cfg<P1>::E, vks,
                          ((long long)blockIdx.x * blockDim.y + threadIdx.y) >> (kPair ? 1 : 0), o0, o1, orb, ev,
                          (long long)g.nx * g.ny * g.nz * P3, a.part, a.part_stride, blockIdx.x,
                          reinterpret_cast<double2*>(smem + FxSmem<P1>::pf(blockDim.y)));
}

// Batched form: a persistent grid draws the work items of one degree class from a ticket
// counter (zero at launch), as k_hbar_batch_split.
template <int P1>
__global__ void __launch_bounds__(256, 2) k_hbar_batch_fx(const BSys* __restrict__ sys,
                                                          const BItem* __restrict__ items, int n_items,
                                                          const __grid_constant__ FxTab<P1> tab,
                                                          int* __restrict__ qctr) {
  constexpr int P3 = P1 * P1 * P1, ES = SplitLayout<P1, double>::ES, CS = FxTab<P1>::CS;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int sA[2 * kAcc * Cfg<P1>::E], sE[2 * Cfg<P1>::E];
  __shared__ unsigned sV[Cfg<P1>::E], sM[4 * Cfg<P1>::E], sR[2 * Cfg<P1>::E];
  __shared__ BSys sS;
  __shared__ BItem sW;
  __shared__ int sIt;
  const int tid = threadIdx.x + blockDim.x * threadIdx.y;
  const int nthr = blockDim.x * blockDim.y;
  for (;;) {
    __syncthreads();
    if (tid == 0) {
      const int it = atomicAdd(qctr, 1);
      sIt = it;
      if (it < n_items) sW = items[it];
    }
    for (int i = tid; i < 2 * kAcc * Cfg<P1>::E; i += nthr) sA[i] = 0;
    for (int i = tid; i < 2 * Cfg<P1>::E; i += nthr) {
      sV[i % Cfg<P1>::E] = 0;
      sM[i] = sM[2 * Cfg<P1>::E + i] = sR[i] = 0;
    }
    __syncthreads();
    if (sIt >= n_items) break;
    for (int i = tid; i < (int)(sizeof(BSys) / 8); i += nthr)
      reinterpret_cast<long long*>(&sS)[i] = reinterpret_cast<const long long*>(&sys[sW.sys])[i];
    __syncthreads();
    const BItem w = sW;
    const BSys& S = sS;
    const Geom& g = S.g;
    auto orb = [&](int o, const double2*& in, double& sc) -> bool {
      const KryOrb& K = S.kry[o];
      if (K.status != KRY_ACTIVE) return false;
      const int j = K.k;
      in = bvec(S, K, o, j);
      sc = K.s[j];
      return true;
    };
    {   // an item none of whose orbitals takes a product here is skipped before the element set-up
      bool any = false;
      for (int o = w.o0; o < w.o1 && !any; ++o) {
        const double2* in_o;
        double sc_o;
        any = orb(o, in_o, sc_o);
      }
      if (!any) continue;
    }
    hbar_elem_fx<P1, false>(
        g, tab, reinterpret_cast<FxC*>(smem) + threadIdx.y * 3 * CS,
        reinterpret_cast<float*>(smem + FxSmem<P1>::kc(blockDim.y)) + threadIdx.y * 3 * FxTab<P1>::KS,
        reinterpret_cast<long long*>(smem + FxSmem<P1>::lines(blockDim.y)) + (size_t)threadIdx.y * ES,
        reinterpret_cast<float*>(smem + FxSmem<P1>::tails(blockDim.y)) + (size_t)threadIdx.y * SplitLayout<P1, float>::ES,
        sA, sE, sV, sM, sR, Cfg<P1>::E, S.vks, (long long)w.eblk * blockDim.y + threadIdx.y, w.o0, w.o1, orb,
        static_cast<double2*>(S.ev), S.n_elem * P3, S.apart, S.n_eblk, w.eblk,
        reinterpret_cast<double2*>(smem + FxSmem<P1>::pf(blockDim.y)));
  }
}

// Density rho(x_q) = sum_a occ_a |(B^(x)3 M^-1/2 psibar_a)(x_q)|^2 (Eq. 2): the three forward
// contractions of the element kernel with B', one exponent per element and orbital; the
// squares are formed and summed over the orbitals in FP64 and divided by the weights that B'
// carries.  FP64 contractions were bound by the FP64 pipe (10 orbitals, 14^3 elements, p = 6:
// 731 us; 16 orbitals, 16^3: 1.75 ms, 0.81 ms here).
template <int P1>
__global__ void __launch_bounds__(256, 2) k_density_fx(Geom g, const __grid_constant__ FxTab<P1> tab,
                                                       const double2* __restrict__ psi, int64_t stride, int n_orb,
                                                       const double* __restrict__ occ, double* __restrict__ rho) {
  constexpr int P2 = P1 * P1, P3 = P2 * P1, CS = FxTab<P1>::CS;
  constexpr int LS = SplitLayout<P1, double>::LS, PS = SplitLayout<P1, double>::PS;
  constexpr int LF = SplitLayout<P1, float>::LS, PF = SplitLayout<P1, float>::PS;
  constexpr bool kBs = kFxBs<P1>;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ FxC sB[kBs ? CS : 1];
  __shared__ unsigned sM[2 * Cfg<P1>::E];
  const int tid = threadIdx.x + blockDim.x * threadIdx.y, el = threadIdx.y;
  if (kBs)
    for (int i = tid; i < CS; i += blockDim.x * blockDim.y) sB[i] = tab.c[i];
  if (tid < 2 * Cfg<P1>::E) sM[tid] = 0;
  long long* const S1 = reinterpret_cast<long long*>(smem) + (size_t)el * SplitLayout<P1, double>::ES;
  float* const F1 = reinterpret_cast<float*>(smem + (size_t)blockDim.y * SplitLayout<P1, double>::ES * sizeof(long long)) +
                    (size_t)el * SplitLayout<P1, float>::ES;
  long long* const S2 = S1 + P1 * PS;
  float* const F2 = F1 + P1 * PF;
  const int u = threadIdx.x % P1, v = threadIdx.x / P1;
  const unsigned grp = __match_any_sync(__activemask(), el);
  const bool lead = (tid & 31) == __ffs(grp) - 1;
  int ex = 0, ey = 0, ez = 0;
  const long long eidx = (long long)blockIdx.x * blockDim.y + el;
  const bool valid = plain_elem(g, eidx, ex, ey, ez);
  const int I = ex * g.p + u, Jn = ey * g.p + v;
  const bool inIJ = valid && I >= 1 && I <= g.nix && Jn >= 1 && Jn <= g.niy;
  const double sxy = inIJ ? g.s[0][I] * g.s[1][Jn] : 0.0;
  const long long base = inIJ ? (long long)(I - 1) + (long long)g.nix * (Jn - 1) : 0;
  const long long plane = (long long)g.nix * g.niy;
  const double* const sz = g.s[2] + ez * g.p;
  const auto cB = [&](int i) { return kBs ? sB[i] : tab.c[i]; };
  const auto kB = [&](int i) { return tab.k[i]; };
  double acc[P1];
#pragma unroll
  for (int q = 0; q < P1; ++q) acc[q] = 0.0;
  __syncthreads();
  for (int o = 0; o < n_orb; ++o) {
    const double2* in = psi + (long long)o * stride;
    double2 w[P1];
    unsigned mx = 0;
#pragma unroll
    for (int c = 0; c < P1; ++c) {
      const int K = ez * g.p + c;
      w[c] = make_double2(0.0, 0.0);
      if (inIJ && K >= 1 && K <= g.niz) {
        w[c] = in[base + plane * (K - 1)];
        const double f = sxy * __ldg(sz + c);
        w[c].x *= f;
        w[c].y *= f;
      }
      mx = max(mx, max((unsigned)__double2hiint(w[c].x) & 0x7fffffffu, (unsigned)__double2hiint(w[c].y) & 0x7fffffffu));
    }
    mx = __reduce_max_sync(grp, mx);
    unsigned* const sm = sM + (o & 1) * Cfg<P1>::E;
    if (lead) atomicMax(&sm[el], mx);
    __syncthreads();
    int eb = (int)(sm[el] >> 20);
    if (threadIdx.x == 0) sM[((o & 1) ^ 1) * Cfg<P1>::E + el] = 0;   // last read before the previous orbital's stages
    const bool poison = eb == 2047;
    eb = eb < 64 ? 64 : (eb > 2046 ? 2046 : eb);
    const int ec = min(3 - kFxBits + eb - 1022, 900);   // (the squares overflow well below the limit)
    const double f = poison ? __hiloint2double(0x7ff80000, 0) : occ[o];
#pragma unroll 1
    for (int comp = 0; comp < 2; ++comp) {
      long long col[P1], t[P1];
      float cf[P1], tf[P1];
#pragma unroll
      for (int c = 0; c < P1; ++c) {
        const double x = comp ? w[c].y : w[c].x;
        col[c] = fx_from_bits((unsigned)__double2hiint(x), (unsigned)__double2loint(x), eb, cf[c]);
      }
      fx_apply<P1>(cB, kB, col, cf, [&](int q, long long x, float xf) {
        S1[q * PS + v * LS + u] = x;
        F1[q * PF + v * LF + u] = xf;
      });
      __syncthreads();
      load_line(col, S1 + v * PS + u, LS);
      load_line(cf, F1 + v * PF + u, LF);
      fx_apply<P1>(cB, kB, col, cf, [&](int q, long long x, float xf) {
        S2[v * PS + q * LS + u] = x;
        F2[v * PF + q * LF + u] = xf;
      });
      __syncthreads();
      load_line(col, S2 + v * PS + u * LS, 1);
      load_line(cf, F2 + v * PF + u * LF, 1);
      fx_apply<P1>(cB, kB, col, cf, [&](int q, long long x, float xf) {
        t[q] = x;
        tf[q] = xf;
      });
      const int es = (ec - fx_join<P1>(t, tf)) << 20;
#pragma unroll
      for (int q = 0; q < P1; ++q) {
        const double x = fx_to_double(t[q], es);
        acc[q] = fma(f * x, x, acc[q]);
      }
    }
  }
  if (valid) {
    const double wuv = tab.iw[u] * tab.iw[v];
#pragma unroll
    for (int q = 0; q < P1; ++q) rho[eidx * P3 + v * P2 + u * P1 + q] = acc[q] * (wuv * tab.iw[q]);
  }
}

template <int P1>
FxTab<P1> make_tab(const FxHost& h) {
  FxTab<P1> t;
  constexpr int CS = FxTab<P1>::CS, KS = FxTab<P1>::KS;
  for (int i = 0; i < 2 * CS; ++i) t.c[i] = fx_coef(h.c[i]);
  for (int m = 0; m < 2; ++m)
    for (int i = 0; i < KS; ++i) t.k[m * KS + i] = fx_tail_const<P1>([&](int j) { return t.c[m * CS + j]; }, i);
  t.dK = h.dK;
  t.kinf = h.kinf;
  for (int q = 0; q < P1; ++q) t.iw[q] = 1.0 / h.w[q];
  return t;
}

template <int P1>
cudaError_t elem_t(const Geom& g, const FxHost& h, const double* vks, const ApplyArgs& a, int E, int bpe, int opc,
                   double2* ev, cudaStream_t st) {
  const dim3 grid(bpe, (a.n_orb + opc - 1) / opc);
  const long long warps = (long long)bpe * grid.y * ((P1 * P1 * E + 31) / 32);
  // With less than four warps per SM one CTA's chain of stages is the launch's time: the real
  // and the imaginary parts side by side (p = 4, 6^3 elements, one orbital: 15.3 -> 11.7 us).
  // With more, both parts in turn share the set-up and the gather.
  const bool pair = 2 * E <= Cfg<P1>::E && warps < 4 * 152;
  const auto launch = [&](auto kern, int rows) {
    const size_t smem = FxSmem<P1>::bytes(rows);
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<grid, dim3(P1 * P1, rows), smem, st>>>(g, make_tab<P1>(h), vks, a, opc, ev);
    return cudaGetLastError();
  };
  return pair ? launch(k_hbar_fx<P1, true>, 2 * E) : launch(k_hbar_fx<P1, false>, E);
}

template <int P1>
cudaError_t density_t(const Geom& g, const FxHost& h, const double2* psi, int64_t stride, int n_orb, const double* occ,
                      double* rho, cudaStream_t st) {
  const long long ne = (long long)g.nx * g.ny * g.nz;
  int E = Cfg<P1>::E;
  while (E > 1 && (ne + E - 1) / E < 2 * 152) E = (E + 1) / 2;   // small meshes: spread over the SMs
  const size_t smem = (size_t)E * (SplitLayout<P1, double>::ES * sizeof(long long) + SplitLayout<P1, float>::ES * sizeof(float));
  cudaError_t e = cudaFuncSetAttribute(k_density_fx<P1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_density_fx<P1><<<(unsigned)((ne + E - 1) / E), dim3(P1 * P1, E), smem, st>>>(g, make_tab<P1>(h), psi, stride, n_orb,
                                                                                occ, rho);
  return cudaGetLastError();
}

template <int P1>
cudaError_t batch_t(const FxHost* h, const BSys* sys, const BItem* items, int n_items, int E, int grid, int* qctr,
                    cudaStream_t st, int* occ) {
  if (E < 1 || P1 * P1 * E > 256) return cudaErrorInvalidValue;
  const size_t smem = FxSmem<P1>::bytes(E);
  cudaError_t e = cudaFuncSetAttribute(k_hbar_batch_fx<P1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  if (occ) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ, k_hbar_batch_fx<P1>, P1 * P1 * E, smem);
  if (n_items <= 0) return cudaSuccess;
  k_hbar_batch_fx<P1><<<grid, dim3(P1 * P1, E), smem, st>>>(sys, items, n_items, make_tab<P1>(*h), qctr);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_hbar_fx(int P1, const Geom& g, const FxHost& h, const double* vks, const ApplyArgs& a, int E,
                           int bpe, int opc, double2* ev, cudaStream_t st) {
  switch (P1) {
    case 2: return elem_t<2>(g, h, vks, a, E, bpe, opc, ev, st);
    case 3: return elem_t<3>(g, h, vks, a, E, bpe, opc, ev, st);
    case 4: return elem_t<4>(g, h, vks, a, E, bpe, opc, ev, st);
    case 5: return elem_t<5>(g, h, vks, a, E, bpe, opc, ev, st);
    case 6: return elem_t<6>(g, h, vks, a, E, bpe, opc, ev, st);
    case 7: return elem_t<7>(g, h, vks, a, E, bpe, opc, ev, st);
    case 8: return elem_t<8>(g, h, vks, a, E, bpe, opc, ev, st);
    case 9: return elem_t<9>(g, h, vks, a, E, bpe, opc, ev, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_hbar_batch_fx(int P1, const FxHost* h, const BSys* sys, const BItem* items, int n_items, int E,
                                 int grid, int* qctr, cudaStream_t st, int* occ) {
  switch (P1) {
    case 2: return batch_t<2>(h, sys, items, n_items, E, grid, qctr, st, occ);
    case 3: return batch_t<3>(h, sys, items, n_items, E, grid, qctr, st, occ);
    case 4: return batch_t<4>(h, sys, items, n_items, E, grid, qctr, st, occ);
    case 5: return batch_t<5>(h, sys, items, n_items, E, grid, qctr, st, occ);
    case 6: return batch_t<6>(h, sys, items, n_items, E, grid, qctr, st, occ);
    case 7: return batch_t<7>(h, sys, items, n_items, E, grid, qctr, st, occ);
    case 8: return batch_t<8>(h, sys, items, n_items, E, grid, qctr, st, occ);
    case 9: return batch_t<9>(h, sys, items, n_items, E, grid, qctr, st, occ);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_density_fx(int P1, const Geom& g, const FxHost& h, const double2* psi, int64_t stride, int n_orb,
                              const double* occ, double* rho, cudaStream_t st) {
  switch (P1) {
    case 2: return density_t<2>(g, h, psi, stride, n_orb, occ, rho, st);
    case 3: return density_t<3>(g, h, psi, stride, n_orb, occ, rho, st);
    case 4: return density_t<4>(g, h, psi, stride, n_orb, occ, rho, st);
    case 5: return density_t<5>(g, h, psi, stride, n_orb, occ, rho, st);
    case 6: return density_t<6>(g, h, psi, stride, n_orb, occ, rho, st);
    case 7: return density_t<7>(g, h, psi, stride, n_orb, occ, rho, st);
    case 8: return density_t<8>(g, h, psi, stride, n_orb, occ, rho, st);
    case 9: return density_t<9>(g, h, psi, stride, n_orb, occ, rho, st);
    default: return cudaErrorInvalidValue;
  }
}

// Convolution pass with two columns per thread (FP32, every transform length;
// with its spectrum read from L2 instead of staged, the lengths of pair_l2()).
//
// The transforms are the four-step FFT of fft_core.cuh (forward FFT along
// the column with the zero-padded half pruned, product with the kernel
// spectrum, inverse FFT with the cropped half pruned; Eq. 5, Sec. IV-A),
// computed for the columns 2p and 2p + 1 of a tile together: a value pair
// PC holds the two columns' real parts in one f32x2 register pair and their
// imaginary parts in another.  Every butterfly is then a packed
// add.rn.f32x2 / sub.rn.f32x2 on operands that already sit in register
// pairs, and a product by a twiddle (the same for both columns) is four or
// five packed multiplies and adds instead of eight scalar ones; the
// shared-memory exchange moves 16 bytes per access.  Rounding: every packed
// operation rounds each lane exactly as the scalar operation would; the
// products are formed as re*c - im*s with one rounding per product and per
// sum, so results agree with the one-column kernel to FP32 rounding.
//
// Persistent CTAs hold one kernel-spectrum tile for a run of right-hand sides
// and stage the next item's input tile by TMA while the current item transforms;
// bounded mbarrier waits with the error codes of col_tma_kernel.
//
// What bounds it: FP32 and shared-memory traffic about equally (counters of one
// launch, 64 right-hand sides of 512^2, 1024 points: per 16 columns on one SM 8,200
// cycles of the FMA pipe and 7,500 of the shared-memory data pipe against 16,600
// taken), with few warps (7.5 a SM, 0.54 eligible a cycle) to overlap the two.
// Cycles per 16 columns on one SM before (one column per thread, or lane
// pairs sharing the 32-point DFTs of 512, and a spectrum tile copied or read
// for every item) and now: 128: 2,370 -> 1,930; 192: 3,930 -> 2,980 (96^3:
// 3,600 -> 2,560); 256: 3,430 -> 3,210; 320: 6,050 -> 5,210; 384: 8,500 ->
// 5,990; 512: 9,310 -> 7,290; 640: 17,700 -> 12,250; 768: 17,000 -> 13,600;
// 1024: 25,600 -> 16,600.  The 32-value plans at 168 registers and three CTAs per
// SM, their spectrum read from L2, took 8,600 (512) to 21,000 (1024).
#pragma once

namespace fwi {
namespace pair {

using u64 = unsigned long long;
// Two complex values (columns a and b): re = (re_a, re_b), im = (im_a, im_b).
struct PC {
  u64 re, im;
};

__device__ __forceinline__ u64 pk(float x, float y) {
  u64 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ void upk(u64 v, float& x, float& y) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v));
}
__device__ __forceinline__ u64 f2add(u64 a, u64 b) {
  u64 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ u64 f2sub(u64 a, u64 b) {
  u64 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ u64 f2mul(u64 a, u64 b) {
  u64 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
// a * b + c
__device__ __forceinline__ u64 f2fma(u64 a, u64 b, u64 c) {
  u64 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ u64 f2neg(u64 a) { return f2mul(a, pk(-1.f, -1.f)); }

__device__ __forceinline__ PC padd(PC a, PC b) { return {f2add(a.re, b.re), f2add(a.im, b.im)}; }
__device__ __forceinline__ PC psub(PC a, PC b) { return {f2sub(a.re, b.re), f2sub(a.im, b.im)}; }

// 16-byte shared-memory access of a pair stored as (re_a, re_b, im_a, im_b)
__device__ __forceinline__ PC lds_pc(const float4* p) {
  PC v;
  asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];"
               : "=l"(v.re), "=l"(v.im)
               : "r"(tc::smem_addr(p)));
  return v;
}
__device__ __forceinline__ void sts_pc(float4* p, PC v) {
  asm volatile("st.shared.v2.b64 [%0], {%1, %2};" ::"r"(tc::smem_addr(p)), "l"(v.re), "l"(v.im)
               : "memory");
}
// Two interleaved complex values (re_a, im_a, re_b, im_b) -> pair
__device__ __forceinline__ PC from_interleaved(float4 q) { return {pk(q.x, q.z), pk(q.y, q.w)}; }
__device__ __forceinline__ float4 to_interleaved(PC v) {
  float4 q;
  upk(v.re, q.x, q.z);
  upk(v.im, q.y, q.w);
  return q;
}

// z * w_R^J (forward) or z * conj(w_R^J) (inverse), J known at compile time.
template <int J, int R, bool INV> __device__ __forceinline__ PC ptw_ct(PC z) {
  constexpr int q = tw_quarter(J, R);
  if constexpr (q == 0) {
    return z;
  } else if constexpr (q == 2) {
    return {f2neg(z.re), f2neg(z.im)};
  } else if constexpr ((q == 1) != INV && (q == 1 || q == 3)) {
    return {z.im, f2neg(z.re)};  // * (-i)
  } else if constexpr (q == 1 || q == 3) {
    return {f2neg(z.im), z.re};  // * (+i)
  } else {
    constexpr float c = (float)tw_re(J, R);
    constexpr float s = INV ? (float)-tw_im(J, R) : (float)tw_im(J, R);
    // (re c - im s, re s + im c)
    return {f2fma(z.re, pk(c, c), f2mul(z.im, pk(-s, -s))),
            f2fma(z.re, pk(s, s), f2mul(z.im, pk(c, c)))};
  }
}
// z * (c + i s), the same twiddle for both columns, from the pair table
__device__ __forceinline__ PC ptw_tab(PC z, u64 cc, u64 ss) {
  return {f2sub(f2mul(z.re, cc), f2mul(z.im, ss)), f2fma(z.re, ss, f2mul(z.im, cc))};
}
// z * (c - i s)
__device__ __forceinline__ PC ptw_tab_conj(PC z, u64 cc, u64 ss) {
  return {f2fma(z.im, ss, f2mul(z.re, cc)), f2sub(f2mul(z.im, cc), f2mul(z.re, ss))};
}
// z * g with a different g per column: gr = (gr_a, gr_b), gi = (gi_a, gi_b)
__device__ __forceinline__ PC pmul(PC z, u64 gr, u64 gi) {
  return {f2sub(f2mul(z.re, gr), f2mul(z.im, gi)), f2fma(z.re, gi, f2mul(z.im, gr))};
}

// c * z, c the same for both columns
__device__ __forceinline__ PC pscale(PC z, float c) {
  const u64 cc = pk(c, c);
  return {f2mul(z.re, cc), f2mul(z.im, cc)};
}
// a + c z
__device__ __forceinline__ PC paxpy(float c, PC z, PC a) {
  const u64 cc = pk(c, c);
  return {f2fma(z.re, cc, a.re), f2fma(z.im, cc, a.im)};
}
// a +- i z
__device__ __forceinline__ PC padd_i(PC a, PC z) { return {f2sub(a.re, z.im), f2add(a.im, z.re)}; }
__device__ __forceinline__ PC psub_i(PC a, PC z) { return {f2add(a.re, z.im), f2sub(a.im, z.re)}; }

// In-register DFT of size R (factors 2, 3, 4, 5), natural order, in place.
template <int R, bool INV> struct PDft;
template <bool INV> struct PDft<1, INV> {
  static __device__ __forceinline__ void run(PC*) {}
};
template <bool INV> struct PDft<2, INV> {
  static __device__ __forceinline__ void run(PC* x) {
    const PC a = x[0], b = x[1];
    x[0] = padd(a, b);
    x[1] = psub(a, b);
  }
};
template <bool INV> struct PDft<4, INV> {
  static __device__ __forceinline__ void run(PC* x) {
    const PC a0 = padd(x[0], x[2]), a1 = psub(x[0], x[2]);
    const PC b0 = padd(x[1], x[3]), d = psub(x[1], x[3]);
    x[0] = padd(a0, b0);
    x[2] = psub(a0, b0);
    // X1 = a1 + w d, X3 = a1 - w d with w = -i (forward) or +i (inverse)
    if constexpr (!INV) {
      x[1] = {f2add(a1.re, d.im), f2sub(a1.im, d.re)};
      x[3] = {f2sub(a1.re, d.im), f2add(a1.im, d.re)};
    } else {
      x[1] = {f2sub(a1.re, d.im), f2add(a1.im, d.re)};
      x[3] = {f2add(a1.re, d.im), f2sub(a1.im, d.re)};
    }
  }
};
template <bool INV> struct PDft<3, INV> {
  static __device__ __forceinline__ void run(PC* x) {
    constexpr float s1 = INV ? 0.86602540378443864676f : -0.86602540378443864676f;
    const PC sp = padd(x[1], x[2]), u = pscale(psub(x[1], x[2]), s1);
    const PC t = paxpy(-0.5f, sp, x[0]);
    x[0] = padd(x[0], sp);
    x[1] = padd_i(t, u);
    x[2] = psub_i(t, u);
  }
};
template <bool INV> struct PDft<5, INV> {
  static __device__ __forceinline__ void run(PC* x) {
    // cosines and sines of 2 pi / 5 and 4 pi / 5
    constexpr float c1 = 0.30901699437494742410f, c2 = -0.80901699437494742410f;
    constexpr float s1 = INV ? 0.95105651629515357212f : -0.95105651629515357212f;
    constexpr float s2 = INV ? 0.58778525229247312917f : -0.58778525229247312917f;
    const PC a = x[0];
    const PC p1 = padd(x[1], x[4]), m1 = psub(x[1], x[4]);
    const PC p2 = padd(x[2], x[3]), m2 = psub(x[2], x[3]);
    const PC t1 = paxpy(c2, p2, paxpy(c1, p1, a)), t2 = paxpy(c1, p2, paxpy(c2, p1, a));
    const PC u1 = paxpy(s2, m2, pscale(m1, s1)), u2 = paxpy(-s1, m2, pscale(m1, s2));
    x[0] = padd(a, padd(p1, p2));
    x[1] = padd_i(t1, u1);
    x[4] = psub_i(t1, u1);
    x[2] = padd_i(t2, u2);
    x[3] = psub_i(t2, u2);
  }
};
// R = A * B: A-point DFTs over n1 (n = B n1 + n2), twiddle w_R^{n2 k1},
// B-point DFTs over n2; output index k = k1 + A k2.
template <int R, bool INV> struct PDft {
  static constexpr int A = first_factor(R);
  static constexpr int B = R / A;
  static_assert(A * B == R && B > 1, "factors 2, 3, 4, 5 only");
  static __device__ __forceinline__ void run(PC* x) {
    PC y[R];
    SFor<B>::run([&](auto n2c) {
      constexpr int n2 = decltype(n2c)::value;
      PC t[A];
#pragma unroll
      for (int n1 = 0; n1 < A; ++n1) t[n1] = x[B * n1 + n2];
      PDft<A, INV>::run(t);
      SFor<A>::run([&](auto k1c) {
        constexpr int k1 = decltype(k1c)::value;
        y[n2 * A + k1] = ptw_ct<(n2 * k1) % R, R, INV>(t[k1]);
      });
    });
#pragma unroll
    for (int k1 = 0; k1 < A; ++k1) {
      PC u[B];
#pragma unroll
      for (int n2 = 0; n2 < B; ++n2) u[n2] = y[n2 * A + k1];
      PDft<B, INV>::run(u);
#pragma unroll
      for (int k2 = 0; k2 < B; ++k2) x[k1 + A * k2] = u[k2];
    }
  }
};
// R-point DFT whose inputs x[R/2 .. R) are zero.
template <int R, bool INV> struct PDftHalfIn {
  static __device__ __forceinline__ void run(PC* x) {
    constexpr int H = R / 2;
    PC a[H], b[H];
    SFor<H>::run([&](auto nc) {
      constexpr int n = decltype(nc)::value;
      a[n] = x[n];
      b[n] = ptw_ct<n, R, INV>(x[n]);
    });
    PDft<H, INV>::run(a);
    PDft<H, INV>::run(b);
#pragma unroll
    for (int k = 0; k < H; ++k) {
      x[2 * k] = a[k];
      x[2 * k + 1] = b[k];
    }
  }
};
// R-point DFT of which only the outputs x[0 .. R/2) are formed.
template <int R, bool INV> struct PDftHalfOut {
  static __device__ __forceinline__ void run(PC* x) {
    constexpr int H = R / 2;
    PC a[H], b[H];
#pragma unroll
    for (int k = 0; k < H; ++k) {
      a[k] = x[2 * k];
      b[k] = x[2 * k + 1];
    }
    PDft<H, INV>::run(a);
    PDft<H, INV>::run(b);
    SFor<H>::run([&](auto nc) {
      constexpr int n = decltype(nc)::value;
      x[n] = padd(a[n], ptw_ct<n, R, INV>(b[n]));
    });
  }
};

}  // namespace pair

// Line plans of the two-column kernel: R1 x R2 with TL threads per column pair
// (thread t owns n2 = t + i TL in phases A and D, k1 = t + i TL in B and C).
template <int L> struct PairPlanFor;
template <> struct PairPlanFor<16> { using type = Plan<16, 4, 4, 4>; };
template <> struct PairPlanFor<32> { using type = Plan<32, 4, 8, 4>; };
template <> struct PairPlanFor<64> { using type = Plan<64, 8, 8, 8>; };
template <> struct PairPlanFor<128> { using type = Plan<128, 16, 8, 8>; };
template <> struct PairPlanFor<192> { using type = Plan<192, 12, 16, 16>; };
template <> struct PairPlanFor<256> { using type = Plan<256, 16, 16, 16>; };
template <> struct PairPlanFor<320> { using type = Plan<320, 20, 16, 20>; };
template <> struct PairPlanFor<384> { using type = Plan<384, 24, 16, 24>; };
template <> struct PairPlanFor<512> { using type = Plan<512, 32, 16, 16>; };
template <> struct PairPlanFor<640> { using type = Plan<640, 32, 20, 32>; };
template <> struct PairPlanFor<768> { using type = Plan<768, 32, 24, 32>; };
template <> struct PairPlanFor<1024> { using type = Plan<1024, 32, 32, 32>; };

// Shared memory (bytes from the 128-byte aligned base): exchange, R2 rows of
// R1 (+ 1 for tiles under 8 pairs, whose rows would otherwise start in the same
// banks) x NP pairs of 16 bytes | input staging rows_in x TC (unless it lies in
// the exchange) | kernel-spectrum tile (where staged), rows 0..L/2 in GBOX boxes
// of at most 256 rows | twiddle table L | two mbarriers and the abort flag.
// ALIAS: the input staging lies inside the exchange buffer (free until every
// thread holds its samples) where a separate one would leave one CTA per SM;
// the next item's copy then starts when the inverse transforms have read the
// exchange, behind an L2 prefetch.
template <class P, int TC> struct ColPairSmem {
  static constexpr int GBOX = (P::L / 2 + 1 + 255) / 256;
  // (several boxes: whole 128-byte units each, as TMA destinations have to be;
  // the rows past L/2 + 1 are spectrum rows nobody reads)
  static constexpr int G_BOX_ROWS =
      GBOX == 1 ? P::L / 2 + 1 : ((P::L / 2 + 1 + GBOX - 1) / GBOX + 3) / 4 * 4;
  static constexpr int G_ROWS = GBOX * G_BOX_ROWS;
  static constexpr int R1P = P::R1 + (TC < 16 ? 1 : 0);
  static constexpr bool ALIAS = (P::L == 512 && TC == 16) || P::L == 1024;
  static constexpr int ROW = TC * (int)sizeof(float2);
  static_assert(P::R2 * R1P * ROW % 128 == 0 && P::L / 2 * ROW % 128 == 0 &&
                (GBOX == 1 || G_BOX_ROWS * ROW % 128 == 0) && G_ROWS <= P::L &&
                G_BOX_ROWS <= 256, "TMA destinations and boxes");
  static constexpr size_t bytes(int rows_in, bool gs) {
    return ((size_t)P::R2 * R1P * TC + (ALIAS ? 0 : (size_t)rows_in * TC) +
            (gs ? (size_t)G_ROWS * TC : 0) + (size_t)P::L) * sizeof(float2) + 32 + 128;
  }
};

// CTAs that take adjacent column tiles of the same right-hand side together.
__host__ __device__ constexpr unsigned pair_group(unsigned ntile) {
  return ntile % 8 == 0 ? 8u : ntile % 4 == 0 ? 4u : ntile % 2 == 0 ? 2u : 1u;
}

// Work order: the (tile group, right-hand side) items, right-hand side fastest,
// are cut into one contiguous range per group of pair_group() CTAs, each of
// which takes one tile of the group.  A CTA so keeps the kernel-spectrum tile
// of one (tile, frequency) in shared memory for as many right-hand sides as its
// range holds, instead of copying it from L2 for every item (as many bytes as
// the input), and the group reads each right-hand side's rows in runs of up to
// 1 KB.  Registers: a pair value takes four; the plans of up to 24 values a
// thread run at 168 (three 128-thread CTAs per SM), those of 32 at up to 255.
template <class P> constexpr int pair_blocks(int threads) {
  return P::E > 24 ? 2 * (128 / threads > 1 ? 128 / threads : 1) : blocks_for_regs(threads, 168);
}
// GS: the spectrum is staged as above; otherwise (col_spectrum_stage = 0) every
// thread reads its column pairs from global memory (L2), at the lengths where
// that was measured against one column per thread, a launch: 16 points (8 x 512
// pixels, 1,024 right-hand sides) 49.2 -> 43.6 us, 64 (32 x 256, 1,024) 95.8 ->
// 79.1, 256 (128 x 256, 1,024) 464 -> 351 and (128 x 160 x 160, 16) 1,343 ->
// 1,182, 512 (256 x 256, 512) 600 -> 422; staged: 42.6, 77, 327, 1,003 and 403.
template <int L> constexpr bool pair_l2() { return L == 16 || L == 64 || L == 256 || L == 512; }
template <class P, int TC, bool GS>
__global__ void __launch_bounds__(TC / 2 * P::TL, pair_blocks<P>(TC / 2 * P::TL))
col_pair_kernel(const ColArgs<float> a, const __grid_constant__ CUtensorMap map,
                const __grid_constant__ CUtensorMap gmap, int rows_in, int nbox) {
  using namespace pair;
  constexpr int NP = TC / 2;  // column pairs per tile
  constexpr int R1 = P::R1, R2 = P::R2, H1 = P::H1, C1 = P::C1, C3 = P::C3, TL = P::TL;
  using SM = ColPairSmem<P, TC>;
  constexpr int R1P = SM::R1P;
  constexpr bool ALIAS = SM::ALIAS;
  extern __shared__ __align__(16) unsigned char smraw[];
  const uint32_t base_pad = (128u - (tc::smem_addr(smraw) & 127u)) & 127u;
  float4* ex = reinterpret_cast<float4*>(smraw + base_pad);        // exchange
  float2* ex_end = reinterpret_cast<float2*>(ex + R2 * R1P * NP);
  float2* stg = ALIAS ? reinterpret_cast<float2*>(ex) : ex_end;    // input staging
  float2* gst = ex_end + (ALIAS ? 0 : rows_in * TC);               // spectrum staging
  float2* tws = gst + (GS ? SM::G_ROWS * TC : 0);                  // twiddles
  uint64_t* bar = reinterpret_cast<uint64_t*>(tws + P::L);         // [0] input, [1] spectrum
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bar + 2);
  const uint32_t bar_in = tc::smem_addr(bar), bar_g = tc::smem_addr(bar + 1);
  const uint32_t stg_a = tc::smem_addr(stg), gst_a = tc::smem_addr(gst);
  const float4* stg4 = reinterpret_cast<const float4*>(stg);
  const float4* gst4 = reinterpret_cast<const float4*>(gst);
  const int cp = threadIdx.x % NP;  // column pair 2cp, 2cp + 1 of the tile
  const int t = threadIdx.x / NP;   // thread of the line
  const unsigned ntile = (unsigned)(a.ncols / TC);
  const unsigned grp = pair_group(ntile), ngrp = gridDim.x / grp;
  const unsigned nact = (unsigned)(a.active ? *a.n_active : a.nb);
  const unsigned items = ntile / grp * (unsigned)a.nplanes * nact;  // < 2^31 (fwi_create)
  const unsigned per = (items + ngrp - 1) / ngrp;
  const unsigned first = blockIdx.x / grp * per;
  const unsigned last = blockIdx.x / grp >= ngrp ? first : min(first + per, items);
  const int box_rows = rows_in / nbox;
  const uint32_t tile_bytes = (uint32_t)(rows_in * TC * sizeof(float2));
  const uint32_t g_bytes = (uint32_t)(SM::G_ROWS * TC * sizeof(float2));
  const long long ls = a.line_stride;
  int dummy_err = 0;
  int* err = a.err ? a.err : &dummy_err;
  auto has_n2 = [&](int i) { return C1 * TL == R2 || t + i * TL < R2; };
  auto has_k1 = [&](int i) { return C3 * TL == R1 || t + i * TL < R1; };

  // item -> column tile, plane, right-hand side, frequency
  struct Item { int tile, plane, rhs, l; };
  auto item_of = [&](unsigned item) {
    const unsigned q = item / nact, tg = q / (unsigned)a.nplanes;
    Item it;
    it.plane = (int)(q - tg * (unsigned)a.nplanes);
    it.tile = (int)(tg * grp + blockIdx.x % grp);
    const int slot = (int)(item - q * nact);
    it.rhs = a.active ? a.active[slot] : slot;
    it.l = a.freq_fixed >= 0 ? a.freq_fixed : (a.rhs0 + it.rhs) / a.n_elem;
    return it;
  };
  auto issue_input = [&](const Item& it) {
    tc::mbar_arrive_expect_tx(bar_in, tile_bytes);
    for (int b = 0; b < nbox; ++b)
      tc::tma_load_3d(stg_a + (uint32_t)(b * box_rows * TC * sizeof(float2)), &map,
                      2 * it.tile * TC, b * box_rows, it.rhs * a.nplanes + it.plane, bar_in);
  };
  auto prefetch_input = [&](const Item& it) {
    for (int b = 0; b < nbox; ++b)
      tc::tma_prefetch_3d(&map, 2 * it.tile * TC, b * box_rows, it.rhs * a.nplanes + it.plane);
  };
  uint32_t g_armed = 0;  // spectrum copies issued (thread 0)
  auto issue_spectrum = [&](const Item& it) {
    ++g_armed;
    tc::mbar_arrive_expect_tx(bar_g, g_bytes + (a.stall ? 16u : 0u));
    for (int b = 0; b < SM::GBOX; ++b)
      tc::tma_load_3d(gst_a + (uint32_t)(b * SM::G_BOX_ROWS * TC * sizeof(float2)), &gmap,
                      2 * it.tile * TC, b * SM::G_BOX_ROWS, it.l, bar_g);
  };

  if (threadIdx.x == 0) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map)) : "memory");
    tc::mbar_init(bar_in, 1);
    tc::mbar_init(bar_g, 1);
    *abort_flag = 0;
    tc::mbar_init_fence();
  }
  for (int i = threadIdx.x; i < P::L; i += blockDim.x) tws[i] = a.tw[i];
  __syncthreads();
  Item it = first < last ? item_of(first) : Item{0, 0, 0, 0}, nx = it;
  if (threadIdx.x == 0 && first < last) {
    issue_input(it);
    if (GS) issue_spectrum(it);
  }
  uint32_t par_in = 0, par_g = 0;
  // new_g: the item has another spectrum tile than the one before it
  bool failed = false, bad = false, new_g = GS;
  for (unsigned item = first; item < last; ++item, it = nx) {
    const bool more = item + 1 < last;
    if (more) nx = item_of(item + 1);
    const int j = it.tile * TC + 2 * cp;
    const bool ok = tc::mbar_wait(bar_in, par_in, abort_flag, err, kColErrWait);
    PC v[P::E];
    // phase-A samples x[R2 n1 + n2], n1 < R1/2 (the rest is the zero padding)
#pragma unroll
    for (int i = 0; i < C1; ++i)
      if (has_n2(i))
#pragma unroll
        for (int n1 = 0; n1 < H1; ++n1)
          v[i * R1 + n1] = from_interleaved(stg4[(R2 * n1 + t + i * TL) * NP + cp]);
    // every thread holds its samples (the input staging is free: the next copy
    // into it comes after the fence) and is done with the previous item's
    // exchange; a failed wait (this item's input, or the previous item's
    // spectrum) stops the CTA
    if constexpr (!ALIAS) tc::fence_proxy_async();
    if (__syncthreads_or(!ok || bad)) {
      failed = true;
      break;
    }
    par_in ^= 1u;
    if (threadIdx.x == 0 && more) {
      if constexpr (ALIAS) prefetch_input(nx);
      else issue_input(nx);
    }
    float2* __restrict__ out =
        a.out + it.rhs * a.out_rhs_stride + it.plane * a.out_plane_stride + j;

    // phase A: R1-point DFTs, twiddle w_L^{n2 k1}, y[n2][k1] to the exchange
#pragma unroll
    for (int i = 0; i < C1; ++i) {
      const int n2 = t + i * TL;
      if (!has_n2(i)) continue;
      PDftHalfIn<R1, false>::run(v + i * R1);
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) {
        PC z = v[i * R1 + k1];
        if (k1 > 0 && n2 > 0) {
          const float2 w = tws[n2 * k1];
          z = ptw_tab(z, pk(w.x, w.x), pk(w.y, w.y));
        }
        sts_pc(ex + (n2 * R1P + k1) * NP + cp, z);
      }
    }
    // one thread waits for a new spectrum tile; the barrier hands its
    // completion (and the copied data) to the others
    if (new_g && threadIdx.x == 0) {
      if (tc::mbar_wait(bar_g, par_g, abort_flag, err, kColErrWait)) par_g ^= 1u;
      else bad = true;
    }
    __syncthreads();
    // phase B: R2-point DFTs over n2, v[k2] = X[k1 + R1 k2]; product with the
    // kernel spectrum (rows folded onto 0..L/2): the staged tile, or columns
    // (j, j + 1) of the item's frequency
    const float4* __restrict__ gg = nullptr;
    if constexpr (!GS)
      gg = reinterpret_cast<const float4*>(a.ghat + (long long)it.l * a.ghat_freq_stride + j);
#pragma unroll
    for (int i = 0; i < C3; ++i) {
      const int k1 = t + i * TL;
      if (!has_k1(i)) continue;
      PC* u = v + i * R2;
#pragma unroll
      for (int n2 = 0; n2 < R2; ++n2) u[n2] = lds_pc(ex + (n2 * R1P + k1) * NP + cp);
      PDft<R2, false>::run(u);
#pragma unroll
      for (int k2 = 0; k2 < R2; ++k2) {
        const int row = spectrum_row<P>(k1, k2, k2);
        float4 g;
        if constexpr (GS) g = gst4[row * NP + cp];
        else g = __ldg(gg + (long long)row * (a.ncols / 2));
        u[k2] = pmul(u[k2], pk(g.x, g.z), pk(g.y, g.w));
      }
    }
    // The exchange slots (n2, k1) of a k1 belong to its thread in phases B and
    // C alike, so no barrier separates them; one before the next item's spectrum
    // tile replaces this one.
    new_g = GS && more && (nx.tile != it.tile || nx.l != it.l);
    if (new_g) {
      tc::fence_proxy_async();
      __syncthreads();
      if (threadIdx.x == 0 && !bad) issue_spectrum(nx);
    }
    // phase C: inverse DFTs over k2, twiddle w_L^{-n2 k1}, y[n2][k1]
#pragma unroll
    for (int i = 0; i < C3; ++i) {
      const int k1 = t + i * TL;
      if (!has_k1(i)) continue;
      PC* u = v + i * R2;
      PDft<R2, true>::run(u);
#pragma unroll
      for (int n2 = 0; n2 < R2; ++n2) {
        PC z = u[n2];
        if (n2 > 0 && k1 > 0) {
          const float2 w = tws[n2 * k1];
          z = ptw_tab_conj(z, pk(w.x, w.x), pk(w.y, w.y));
        }
        sts_pc(ex + (n2 * R1P + k1) * NP + cp, z);
      }
    }
    __syncthreads();
    // phase D: inverse R1-point DFTs of which the cropped half is formed
#pragma unroll
    for (int i = 0; i < C1; ++i) {
      const int n2 = t + i * TL;
      if (!has_n2(i)) continue;
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) v[i * R1 + k1] = lds_pc(ex + (n2 * R1P + k1) * NP + cp);
    }
    if constexpr (ALIAS) {
      // the exchange is free: the next item's tile may land in it (the fence
      // orders this thread's exchange accesses before the copy's writes)
      tc::fence_proxy_async();
      __syncthreads();
      if (threadIdx.x == 0 && more) issue_input(nx);
    }
#pragma unroll
    for (int i = 0; i < C1; ++i) {
      const int n2 = t + i * TL;
      if (!has_n2(i)) continue;
      PC* u = v + i * R1;
      PDftHalfOut<R1, true>::run(u);
#pragma unroll
      for (int n1 = 0; n1 < H1; ++n1)
        *reinterpret_cast<float4*>(out + (long long)(R2 * n1 + n2) * ls) = to_interleaved(u[n1]);
    }
  }
  // copies of a CTA that stopped early may still land in its shared memory: the
  // input of the item it stopped at, and the spectrum whose wait gave up, be it
  // the last item's (which no later item's `failed` follows)
  if (threadIdx.x == 0) {
    if (failed) tc::mbar_wait_drain(bar_in, par_in, err, kColErrDrain);
    tc::mbar_drain_armed(bar_g, g_armed, err, kColErrDrain);
  }
}

}  // namespace fwi

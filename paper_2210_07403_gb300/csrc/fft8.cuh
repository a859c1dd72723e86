// Register-resident FFT of power-of-two length N = 2^L (L = 4 … 13), the transform of the 2-D
// IBDL kernels. The transform length is a compile-time constant, so every index, stride and loop
// below folds to constants.
//
// Layout. A sequence is handled by Q = N/8 lanes; lane j holds the eight elements
// x[j + s·Q], s = 0 … 7, in registers, both on entry and on exit (the transform of element
// j + s·Q). A thread may hold V lanes of a sequence (j, j + Q/V, …) and FL sequences at once.
//
// Stages (Stockham autosort, no bit reversal): radix-8 stages with sub-transform lengths
// p = 1, 8, 64, … first, then one radix-2 or radix-4 stage when L is not a multiple of 3. A
// radix-8 stage with length p: butterfly j takes x[j + r·Q] (r < 8), multiplies input r by
// ω^{r·k}, k = j mod p, ω = e^{∓2πi/(8p)}, takes the 8-point DFT and writes output t to
// y[(j − k)·8 + k + t·p]. The tail stage (radix R, length N/R) runs 8/R butterflies per lane,
// i = j + m·Q, on the lane's own registers and leaves output t of butterfly m in x[m + t·8/R]:
// the same positions j + s·Q. Between stages the lanes exchange through one padded shared-memory
// buffer per sequence (N + N/8 elements: one pad after every eight keeps the stride-8 writes of the
// first stage free of bank conflicts).
//
// Twiddles come from a table (TwLayout): held in registers per lane (read once, before a kernel's
// dependency wait) or read from the table at each use.
//
// FP64 transforms are bound by the FP64 pipe (an SM sub-partition takes a fused multiply-add of a warp every 64
// cycles, a sum or a product every 76), so their stages are written for the least number of FP64 instructions: a twiddled
// radix-8 stage is three levels of radix-2 butterflies a ± w·b, and with w = c(1 + i·t), t = tan of its
// angle, p = b·(1 + i·t) and a ± c·p take six fused multiply-adds (Linzer and Feig, IEEE Trans. Signal
// Process. 41 (1993) 93–107, and Goedecker, SIAM J. Sci. Comput. 18 (1997) 1605–1611, describe such
// forms): 72 instructions instead of 84 for seven complex products and the 8-point DFT; the first
// stage's √½ factors go into its last additions (52 instead of 56). The error of c·(b_x − t·b_y)
// is that of c·b_x − s·b_y, however large t is; b·(1 + i·t) exceeds w·b by at most 1/c < n/6 (quarter
// turns, c = 0, are treated apart), which is the headroom the form takes off the FP64 range. The table then
// holds (c, t), and a lane needs four entries per radix-8 stage instead of seven. FP64 applications before /
// after: 512² Stokes star 131 / 118 µs, 2048² (finite differences, divergence dipole) 791 / 671 µs, 128³
// sphere 261 / 249 µs. The form rounds less often: rms relative error of a transform of random data, cosine and
// sine form / this one, both emulated against 80-bit arithmetic: 1.22e−16 / 1.17e−16 at 16 points, 2.00 / 1.84 at
// 512, 2.51 / 2.29 at 8192. (Of S*u nothing of it shows, the kernel tables' rounding sets its error: 64² circle
// 4.2e−15, 1024² 3.7e−14 / 3.6e−14, 128³ 2.4e−15.)
#pragma once

#include <type_traits>
#include <utility>

#include "fft.cuh"

namespace ibdl {

template <int I, int E, class F>
__device__ __forceinline__ void static_for(F&& f) {
  if constexpr (I < E) {
    f(std::integral_constant<int, I>{});
    static_for<I + 1, E>(f);
  }
}

template <int L, int V_, int E = 8>
struct F8 {
  static_assert(L >= 4 && L <= 13, "transform lengths 16 … 8192");
  static constexpr int N = 1 << L;
  static constexpr int Q = N / E;                        // lanes of a sequence (E elements each)
  static constexpr int S8 = L / 3;                       // radix-8 stages
  static constexpr int LT = L % 3;                       // log2 of the tail radix (0: none)
  static constexpr int RT = 1 << LT;
  static constexpr int NST = S8 + (LT ? 1 : 0);          // stages
  static constexpr int V = V_;                           // lanes per thread
  static_assert(Q % V == 0, "lanes per thread must divide Q");
  static constexpr int QT = Q / V;                       // threads per sequence
  static constexpr int PN = N + N / 8;                   // padded sequence length in shared memory
};

// T transforms in the fused form (table entries (cos, tan)).
template <typename T>
constexpr bool kFused8 = std::is_same<T, double>::value;

__host__ __device__ constexpr int ipow8(int s) { return s == 0 ? 1 : 8 * ipow8(s - 1); }

// The twiddle table, per stage in the order the lanes read it. A radix-8 stage S ≥ 1 with sub-length
// p = 8^S has NV = 7 values per k = j mod p (w^r, r = 1 … 7), in the fused form 4 (w, w², w⁴ and w·e^{−iπ/4});
// a tail stage has 8/RT butterflies m of RT − 1 values per lane j (w^r of i = j + m·Q), in the fused
// form log2(RT) (w, w²). The values of one k form 16-byte chunks (two FP32 values, or one of 16 bytes);
// chunk c of k lies at (offset of the stage) + c·p + k, so that the lanes of a warp read adjacent
// chunks. (Read from one table of e^{−2πi m/N} at m = r·k·N/(8p), a warp's loads touched up to 32 cache
// lines each; the L1 cache was 84 % busy in the 8192² row kernels. Applications before / after: FP32
// 8192² circle 584 / 499 µs, scalar 4096² 141 / 113, 2048² 41 / 34, Stokes 2048² 124 / 102; FP64 8192² 7774 /
// 7619, 2048² 420 / 411; float-float Stokes 2048² 424 / 373.)
template <typename T, int L>
struct TwLayout {
  static constexpr int S8 = L / 3, LT = L % 3, RT = 1 << LT, Q = (1 << L) / 8;
  static constexpr int PER = sizeof(T) == 4 ? 2 : 1;      // values per chunk
  static constexpr int N8 = kFused8<T> ? 4 : 7;           // values of a radix-8 stage
  static constexpr int NT = kFused8<T> ? LT : RT - 1;     // values of a tail butterfly
  static constexpr int NTAIL = LT ? NT * (8 / RT) : 0;
  static constexpr int C8 = (N8 + PER - 1) / PER, CT = (NTAIL + PER - 1) / PER;
  static constexpr int NTW = (S8 - 1) * N8 + NTAIL;       // values per lane
  static constexpr int CHUNKS = C8 * ((ipow8(S8) - 8) / 7) + CT * Q;
  template <int S>
  static constexpr int NV = S < S8 ? N8 : NTAIL;
  // the values of stage S on lane j
  template <int S>
  __device__ static __forceinline__ void read(const cplx<T>* __restrict__ tab, int j, cplx<T>* w) {
    constexpr int p = S < S8 ? ipow8(S) : Q, NC = S < S8 ? C8 : CT;
    const int k = S < S8 ? j & (p - 1) : j;
    const cplx<T>* t = tab + PER * (C8 * ((ipow8(S < S8 ? S : S8) - 8) / 7) + k);
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      if constexpr (PER == 2) {
        const float4 v = reinterpret_cast<const float4*>(t)[c * p];
        w[2 * c] = mk(T(v.x), T(v.y));
        if (2 * c + 1 < NV<S>) w[2 * c + 1] = mk(T(v.z), T(v.w));
      } else {
        w[c] = t[c * p];
      }
    }
  }
};

// the twiddles of one lane, in registers
template <typename T, int L>
struct TwRegs {
  using Y = TwLayout<T, L>;
  cplx<T> w[Y::NTW > 0 ? Y::NTW : 1];
  __device__ __forceinline__ void load(const cplx<T>* __restrict__ tab, int j) {
    static_for<1, Y::S8 + (Y::LT ? 1 : 0)>([&](auto st) {
      constexpr int S = decltype(st)::value;
      Y::template read<S>(tab, j, w + (S - 1) * Y::N8);
    });
  }
  template <int S>
  __device__ __forceinline__ void get(cplx<T>* v) const {
#pragma unroll
    for (int i = 0; i < Y::template NV<S>; ++i) v[i] = w[(S - 1) * Y::N8 + i];
  }
};

// the twiddles of one lane, read from the table (global memory, L1-cached) at each use
template <typename T, int L>
struct TwTable {
  const cplx<T>* __restrict__ tab;
  int j;
  __device__ __forceinline__ void load(const cplx<T>* __restrict__ t, int lane) {
    tab = t;
    j = lane;
  }
  template <int S>
  __device__ __forceinline__ void get(cplx<T>* v) const { TwLayout<T, L>::template read<S>(tab, j, v); }
};

// a·w (forward) or a·conj(w) (inverse)
template <typename T, bool INV>
__device__ __forceinline__ cplx<T> cmul_tw(cplx<T> a, cplx<T> w) {
  return INV ? mk(a.x * w.x + a.y * w.y, a.y * w.x - a.x * w.y) : mk(a.x * w.x - a.y * w.y, a.x * w.y + a.y * w.x);
}

// whether a table entry stands for −i, by its high words (off the FP64 pipe)
__device__ __forceinline__ bool quarter_turn(cplx<double> w) {
  return __double2hiint(w.x) == 0x3ff00000 && __double2hiint(w.y) == (int)0xbff00000;  // 1, −1
}

// (a, b) ← (a + w·b, a − w·b) with w = c(1 + i·t) given as (c, t) (INV: conj w; ROT: times −i, INV i).
// A quarter turn has no tangent: the table holds (1, −1) for it, which is no angle's pair, and with QTR
// (the butterflies whose twiddle can be one) p = ∓i·b then leaves the other part out. (A huge tangent
// in its place would overflow on data far below the top of the FP64 range.)
template <typename T, bool INV, bool ROT, bool QTR = false>
__device__ __forceinline__ void bfly_tan(cplx<T>& a, cplx<T>& b, cplx<T> w) {
  const T t = INV ? -w.y : w.y;
  const bool q = QTR && quarter_turn(w);
  cplx<T> p = mk(fma(-t, b.y, q ? T(0) : b.x), fma(t, b.x, q ? T(0) : b.y));
  if (ROT) p = rot90<T, INV>(p);
  b = mk(fma(-w.x, p.x, a.x), fma(-w.x, p.y, a.y));
  a = mk(fma(w.x, p.x, a.x), fma(w.x, p.y, a.y));
}

// 8-point DFT of w^r·x_r, r < 8, from w, w², w⁴ and w·e^{−iπ/4} as (cos, tan): 72 fused multiply-adds
template <typename T, bool INV>
__device__ __forceinline__ void dft8_tan(cplx<T> (&x)[8], cplx<T> w1, cplx<T> w2, cplx<T> w4, cplx<T> w1e) {
  // t mod 2 from the pairs (r, r + 4): x[r], x[r + 4]
#pragma unroll
  for (int r = 0; r < 4; ++r) bfly_tan<T, INV, false, true>(x[r], x[r + 4], w4);
  // t mod 4 from the pairs (r, r + 2): t = 0, 2 in (x0, x2), (x1, x3); 1, 3 in (x4, x6), (x5, x7)
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    bfly_tan<T, INV, false>(x[r], x[r + 2], w2);
    bfly_tan<T, INV, true>(x[r + 4], x[r + 6], w2);
  }
  bfly_tan<T, INV, false>(x[0], x[1], w1);  // outputs 0, 4
  bfly_tan<T, INV, true>(x[2], x[3], w1);   // 2, 6
  bfly_tan<T, INV, false>(x[4], x[5], w1e);  // 1, 5
  bfly_tan<T, INV, true>(x[6], x[7], w1e);   // 3, 7
  const cplx<T> y[8] = {x[0], x[4], x[2], x[6], x[1], x[5], x[3], x[7]};
#pragma unroll
  for (int t = 0; t < 8; ++t) x[t] = y[t];
}

// 8-point DFT as dft8, the odd half's √½ factors inside its last additions: 52 FP64 instructions
template <typename T, bool INV>
__device__ __forceinline__ void dft8_fma(cplx<T>* u) {
  const T c = T(0.70710678118654752440);
  cplx<T> a0 = cadd(u[0], u[4]), a1 = cadd(u[1], u[5]), a2 = cadd(u[2], u[6]), a3 = cadd(u[3], u[7]);
  const cplx<T> b0 = csub(u[0], u[4]), b1 = csub(u[1], u[5]), b2 = rot90<T, INV>(csub(u[2], u[6])), b3 = csub(u[3], u[7]);
  // √2·ω₈·b1 and √2·ω₈³·b3
  const cplx<T> p1 = INV ? mk(b1.x - b1.y, b1.x + b1.y) : mk(b1.x + b1.y, b1.y - b1.x);
  const cplx<T> p3 = INV ? mk(-(b3.x + b3.y), b3.x - b3.y) : mk(b3.y - b3.x, -(b3.x + b3.y));
  dft4<T, INV>(a0, a1, a2, a3);
  const cplx<T> t0 = cadd(b0, b2), t1 = csub(b0, b2), t2 = cadd(p1, p3), t3 = rot90<T, INV>(csub(p1, p3));
  u[0] = a0;
  u[1] = mk(fma(c, t2.x, t0.x), fma(c, t2.y, t0.y));
  u[2] = a1;
  u[3] = mk(fma(c, t3.x, t1.x), fma(c, t3.y, t1.y));
  u[4] = a2;
  u[5] = mk(fma(-c, t2.x, t0.x), fma(-c, t2.y, t0.y));
  u[6] = a3;
  u[7] = mk(fma(-c, t3.x, t1.x), fma(-c, t3.y, t1.y));
}

// stage S on one lane's registers
template <typename T, bool INV, int L, int S, class TW>
__device__ __forceinline__ void f8_stage(cplx<T> (&x)[8], const TW& tw) {
  constexpr int S8 = L / 3, LT = L % 3, RT = 1 << LT;
  cplx<T> w[8];
  if constexpr (S > 0) tw.template get<S>(w);
  if constexpr (kFused8<T>) {
    if constexpr (S == 0) {
      dft8_fma<T, INV>(x);
    } else if constexpr (S < S8) {
      dft8_tan<T, INV>(x, w[0], w[1], w[2], w[3]);
    } else if constexpr (LT == 1) {
#pragma unroll
      for (int m = 0; m < 4; ++m) bfly_tan<T, INV, false, true>(x[m], x[m + 4], w[m]);
    } else {
      // radix 4: inputs and outputs of butterfly m at x[m + 2r], r = 0 … 3
#pragma unroll
      for (int m = 0; m < 2; ++m) {
        bfly_tan<T, INV, false, true>(x[m], x[m + 4], w[2 * m + 1]);
        bfly_tan<T, INV, false, true>(x[m + 2], x[m + 6], w[2 * m + 1]);
        bfly_tan<T, INV, false>(x[m], x[m + 2], w[2 * m]);     // outputs 0, 2
        bfly_tan<T, INV, true>(x[m + 4], x[m + 6], w[2 * m]);  // outputs 1, 3
        const cplx<T> y1 = x[m + 4], y2 = x[m + 2];
        x[m + 2] = y1;
        x[m + 4] = y2;
      }
    }
  } else if constexpr (S < S8) {
    if constexpr (S > 0) {
#pragma unroll
      for (int r = 1; r < 8; ++r) x[r] = cmul_tw<T, INV>(x[r], w[r - 1]);
    }
    dft8<T, INV>(x);
  } else {
    constexpr int MB = 8 / RT;
#pragma unroll
    for (int m = 0; m < MB; ++m) {
      cplx<T> u[RT];
#pragma unroll
      for (int r = 0; r < RT; ++r) u[r] = x[m + r * MB];
#pragma unroll
      for (int r = 1; r < RT; ++r) u[r] = cmul_tw<T, INV>(u[r], w[m * (RT - 1) + r - 1]);
      if constexpr (RT == 4)
        dft4<T, INV>(u[0], u[1], u[2], u[3]);
      else
        dft2<T, INV>(u);
#pragma unroll
      for (int t = 0; t < RT; ++t) x[m + t * MB] = u[t];
    }
  }
}

// padded position of element e < N of a sequence: one pad after every 2^PS elements. A warp's access takes
// groups of 16 lanes of 8-byte elements or 8 of 16-byte ones, and the least wavefronts when a group's
// positions differ mod its size. PS = 3 gives that for 16-byte elements, and for 8-byte ones where the
// lanes of several sequences alternate in a warp; PS = 4 for 8-byte elements with one sequence per warp
// (there, 16 adjacent elements at PS = 3 meet one bank twice, half of the shared-memory wavefronts of
// the 8192² FP32 row kernels; at PS = 4 only the second stage's writes do: spread 111 / 93 µs,
// gather 98 / 84, the application 499 / 469).
template <int PS = 3>
__device__ __forceinline__ int ppos(int e) { return e + (e >> PS); }
// padded position of j + s·Q: ppos(j) + s·ppos(Q) when Q is a multiple of 2^PS (PS = 3: n ≥ 64)
template <int Q, int PS = 3>
__device__ __forceinline__ int ppos_strided(int j, int s) {
  if constexpr (Q % (1 << PS) == 0)
    return ppos<PS>(j) + s * (Q + (Q >> PS));
  else
    return ppos<PS>(j + s * Q);
}

// The same transform for one sequence with the radix-8 stages as a loop over a runtime
// sub-length p and the twiddles read from the table: one copy of
// the stage code instead of one per stage. For float-float, whose unrolled stages would not fit
// the instruction cache.
template <typename T, bool INV, int L, int V>
__device__ __forceinline__ void f8_fft_rolled(cplx<T> (&x)[1][V][8], cplx<T>* buf, int j0,
                                              const cplx<T>* __restrict__ tab, bool active) {
  using F = F8<L, V>;
#pragma unroll 1
  for (int S = 0; S < F::S8; ++S) {
    const int p = 1 << (3 * S);
    if (active) {
#pragma unroll
      for (int v = 0; v < V; ++v) {
        if (S > 0) {
          // (seven 16-byte chunks per k; 8 + … + 8^(S−1) = (p − 8)/7 values of k before this stage)
          const cplx<T>* t = tab + (p - 8) + ((j0 + v * F::QT) & (p - 1));
#pragma unroll
          for (int r = 1; r < 8; ++r) x[0][v][r] = cmul_tw<T, INV>(x[0][v][r], t[(r - 1) * p]);
        }
        dft8<T, INV>(x[0][v]);
      }
    }
    if (S + 1 < F::NST) {
      __syncthreads();
      if (active) {
#pragma unroll
        for (int v = 0; v < V; ++v) {
          const int j = j0 + v * F::QT, k = j & (p - 1);
          const int base = (j - k) * 8 + k;
#pragma unroll
          for (int t = 0; t < 8; ++t) buf[ppos(base + t * p)] = x[0][v][t];
        }
      }
      __syncthreads();
      if (active) {
#pragma unroll
        for (int v = 0; v < V; ++v) {
          const int j = j0 + v * F::QT;
#pragma unroll
          for (int s = 0; s < 8; ++s) x[0][v][s] = buf[ppos(j + s * F::Q)];
        }
      }
    }
  }
  if constexpr (F::LT > 0) {
    if (active) {
#pragma unroll
      for (int v = 0; v < V; ++v) {
        TwTable<T, L> tw;
        tw.load(tab, j0 + v * F::QT);
        f8_stage<T, INV, L, F::S8>(x[0][v], tw);
      }
    }
  }
}

// Transform of the FL sequences whose lanes j0 + v·QT (v < V) this thread holds: x[f][v][s] is
// element j + s·Q on entry and its transform on exit. buf + f·fstride is the padded shared buffer
// of sequence f. Every thread of the block must call it (it synchronises the block); `active` is
// false for threads that hold no sequence. Each lane reads its inputs before the call and writes
// its results after it only at its own positions j + s·Q, so neither needs a barrier against the
// exchanges inside.
template <typename T, bool INV, int L, int V, int FL, int PS = 3, class TW>
__device__ __forceinline__ void f8_fft(cplx<T> (&x)[FL][V][8], cplx<T>* buf, int fstride, int j0,
                                       const TW (&tw)[V], bool active) {
  using F = F8<L, V>;
  if constexpr (FL == 1 && std::is_same<TW, TwTable<T, L>>::value && sizeof(T) == 8 && !std::is_same<T, double>::value) {
    // float-float (8-byte elements that are not double): the stage loop
    f8_fft_rolled<T, INV, L, V>(reinterpret_cast<cplx<T>(&)[1][V][8]>(x), buf, j0, tw[0].tab, active);
    return;
  }
  static_for<0, F::NST>([&](auto st) {
    constexpr int S = decltype(st)::value;
    if (active) {
#pragma unroll
      for (int f = 0; f < FL; ++f)
#pragma unroll
        for (int v = 0; v < V; ++v) f8_stage<T, INV, L, S>(x[f][v], tw[v]);
    }
    if constexpr (S + 1 < F::NST) {
      constexpr int p = ipow8(S);
      __syncthreads();
      if (active) {
#pragma unroll
        for (int v = 0; v < V; ++v) {
          const int j = j0 + v * F::QT, k = j & (p - 1);
          // adding t·p (t < 8) to base carries nothing out of its low PS bits, so the padded position is
          // ppos(base) plus a constant per t
          const int pb = ppos<PS>((j - k) * 8 + k);
#pragma unroll
          for (int f = 0; f < FL; ++f)
#pragma unroll
            for (int t = 0; t < 8; ++t) buf[f * fstride + pb + t * p + ((t * p) >> PS)] = x[f][v][t];
        }
      }
      __syncthreads();
      if (active) {
#pragma unroll
        for (int v = 0; v < V; ++v) {
          const int j = j0 + v * F::QT;
#pragma unroll
          for (int f = 0; f < FL; ++f)
#pragma unroll
            for (int s = 0; s < 8; ++s) x[f][v][s] = buf[f * fstride + ppos_strided<F::Q, PS>(j, s)];
        }
      }
    }
  });
}

// ------------------------------------------------------------------------------------------
// The same transform with E = 2 or 4 elements per lane (Q = N/E lanes): radix-E stages, and for
// E = 4 and odd L a radix-2 tail. A lane's chain of operations is shorter (64 points: 34 FP64
// instructions per transform with E = 2, 124 with E = 8) and a sequence spreads over more warps, at
// the price of more exchanges and somewhat more operations in all: for single problems too small to
// fill the GPU. FP64 (E = 2) and float-float only.
// ------------------------------------------------------------------------------------------
__host__ __device__ constexpr int ipow(int b, int e) { return e == 0 ? 1 : b * ipow(b, e - 1); }

// Twiddles: NV values per stage S ≥ 1 and k = j mod E^S (E = 2: w; E = 4: w, w², w³), then for the tail two per
// lane j (w of i = j, j + Q); 16-byte values, value c of k at offset(S) + c·E^S + k.
template <typename T, int L, int E>
struct FewLayout {
  static_assert(E == 2 || !kFused8<T>, "four elements per lane: float-float only (no fused radix-4 stage)");
  static constexpr int LE = E == 2 ? 1 : 2, NS = L / LE, LT = L % LE, Q = (1 << L) / E;
  static constexpr int NV = E - 1, NT = LT ? 2 : 0;
  __host__ __device__ static constexpr int offset(int S) { return NV * ((ipow(E, S) - E) / (E - 1)); }
  static constexpr int NTW = NV * (NS - 1) + NT;
};

template <typename T, int L, int E>
struct TwFew {
  using Y = FewLayout<T, L, E>;
  cplx<T> w[Y::NTW];
  __device__ __forceinline__ void load(const cplx<T>* __restrict__ tab, int j) {
    static_for<1, Y::NS>([&](auto st) {
      constexpr int S = decltype(st)::value, p = ipow(E, S);
#pragma unroll
      for (int c = 0; c < Y::NV; ++c) w[(S - 1) * Y::NV + c] = tab[Y::offset(S) + c * p + (j & (p - 1))];
    });
#pragma unroll
    for (int m = 0; m < Y::NT; ++m) w[(Y::NS - 1) * Y::NV + m] = tab[Y::offset(Y::NS) + m * Y::Q + j];
  }
};

// (a, b) ← (a + w·b, a − w·b)
template <typename T, bool INV>
__device__ __forceinline__ void bfly(cplx<T>& a, cplx<T>& b, cplx<T> w) {
  if constexpr (kFused8<T>) {
    bfly_tan<T, INV, false, true>(a, b, w);
  } else {
    const cplx<T> t = cmul_tw<T, INV>(b, w);
    b = csub(a, t);
    a = cadd(a, t);
  }
}

template <typename T, bool INV, int L, int E>
__device__ __forceinline__ void few_fft(cplx<T> (&x)[E], cplx<T>* buf, int j, const TwFew<T, L, E>& tw, bool active) {
  using Y = FewLayout<T, L, E>;
  constexpr int NST = Y::NS + (Y::LT ? 1 : 0), Q = Y::Q;
  static_for<0, NST>([&](auto st) {
    constexpr int S = decltype(st)::value;
    if (active) {
      if constexpr (E == 2) {
        if constexpr (S == 0)
          dft2<T, INV>(x);
        else
          bfly<T, INV>(x[0], x[1], tw.w[S - 1]);
      } else if constexpr (S == Y::NS) {  // tail: butterflies i = j, j + Q
        bfly<T, INV>(x[0], x[2], tw.w[(S - 1) * Y::NV]);
        bfly<T, INV>(x[1], x[3], tw.w[(S - 1) * Y::NV + 1]);
      } else if constexpr (S == 0) {
        dft4<T, INV>(x[0], x[1], x[2], x[3]);
      } else {
#pragma unroll
        for (int r = 1; r < 4; ++r) x[r] = cmul_tw<T, INV>(x[r], tw.w[(S - 1) * Y::NV + r - 1]);
        dft4<T, INV>(x[0], x[1], x[2], x[3]);
      }
    }
    if constexpr (S + 1 < NST) {
      constexpr int p = ipow(E, S);
      __syncthreads();
      if (active) {
        const int k = j & (p - 1), b = (j - k) * E + k;
#pragma unroll
        for (int t = 0; t < E; ++t) buf[ppos(b + t * p)] = x[t];
      }
      __syncthreads();
      if (active) {
#pragma unroll
        for (int s = 0; s < E; ++s) x[s] = buf[ppos_strided<Q>(j, s)];
      }
    }
  });
}

// the transform of one sequence with E elements per lane
template <typename T, bool INV, int L, int V, int E, int PS = 3, class TW>
__device__ __forceinline__ void fft_lanes(cplx<T> (&x)[1][V][E], cplx<T>* buf, int j0, const TW (&tw)[V], bool active) {
  if constexpr (E == 8)
    f8_fft<T, INV, L, V, 1, PS>(x, buf, 0, j0, tw, active);
  else
    few_fft<T, INV, L, E>(x[0][0], buf, j0, tw[0], active);
}

}  // namespace ibdl

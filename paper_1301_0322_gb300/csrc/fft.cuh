// Shared-memory Stockham FFT engine for the PM solver (sm_103a).
//
// One thread block transforms a batch of independent 1-D sequences of length N.  Each thread
// owns E elements (E/R butterflies of radix R per stage); T = N/E threads cooperate on one
// sequence.  The first stage reads its inputs straight from the caller (global memory or
// shared memory), the last stage writes straight to the caller; intermediate stages exchange
// through shared memory (Stockham autosort: output in natural order, no bit reversal).
//
// Conventions: forward = exp(-2 pi i n k / N), inverse = exp(+2 pi i n k / N), neither scaled.
// Twiddles come from a float2 table tw[m] = exp(-2 pi i m / NT) computed in float64 on the
// host; stage twiddles exp(-2 pi i m / N) are read at tw[m * TWS] with NT = N * TWS.
#pragma once
#include <cstdint>
#include <type_traits>
#include <utility>

namespace cola {

// Complex arithmetic with every rounding spelled out (__fadd_rn / __fmul_rn are never fused
// into an FMA by the compiler): a kernel body then rounds identically in every kernel it is
// inlined into, so the single-box and the ensemble kernels give bit-identical results.
__device__ __forceinline__ float2 c_add(float2 a, float2 b) { return make_float2(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y)); }
__device__ __forceinline__ float2 c_sub(float2 a, float2 b) { return make_float2(__fsub_rn(a.x, b.x), __fsub_rn(a.y, b.y)); }
__device__ __forceinline__ float2 c_mul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, __fmul_rn(-a.y, b.y)), fmaf(a.x, b.y, __fmul_rn(a.y, b.x)));
}
__device__ __forceinline__ float2 c_conj(float2 a) { return make_float2(a.x, -a.y); }
__device__ __forceinline__ float2 c_scale(float2 a, float s) { return make_float2(__fmul_rn(a.x, s), __fmul_rn(a.y, s)); }
// a + r b and a - r b with r = -i (forward sign) or +i (inverse sign)
template <bool INV>
__device__ __forceinline__ float2 c_add_rot(float2 a, float2 b) {
  return INV ? make_float2(__fsub_rn(a.x, b.y), __fadd_rn(a.y, b.x)) : make_float2(__fadd_rn(a.x, b.y), __fsub_rn(a.y, b.x));
}
template <bool INV>
__device__ __forceinline__ float2 c_sub_rot(float2 a, float2 b) {
  return c_add_rot<!INV>(a, b);
}
__device__ __forceinline__ float2 c_fma(float s, float2 a, float2 b) { return make_float2(fmaf(s, a.x, b.x), fmaf(s, a.y, b.y)); }
// a + i s b
__device__ __forceinline__ float2 c_fma_i(float s, float2 b, float2 a) { return make_float2(fmaf(-s, b.y, a.x), fmaf(s, b.x, a.y)); }

// Two complex values at once, as the pair of their real parts and the pair of their imaginary
// parts: the arithmetic of a transform over two columns then runs in packed float32
// instructions (add, mul, fma .f32x2), each of which rounds its two lanes as the scalar one
// does, so both columns get the bits of the scalar transform for half of its instructions
// (twiddles, addresses and exchange accesses are shared as well).
struct alignas(16) cpair {
  float2 re, im;
};
__device__ __forceinline__ unsigned long long p_bits(float2 a) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y));
  return r;
}
__device__ __forceinline__ float2 p_value(unsigned long long v) {
  float2 d;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(v));
  return d;
}
__device__ __forceinline__ float2 p_add(float2 a, float2 b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(p_bits(a)), "l"(p_bits(b)));
  return p_value(r);
}
__device__ __forceinline__ float2 p_sub(float2 a, float2 b) {
  unsigned long long r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(p_bits(a)), "l"(p_bits(b)));
  return p_value(r);
}
__device__ __forceinline__ float2 p_mul(float2 a, float2 b) {
  unsigned long long r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(p_bits(a)), "l"(p_bits(b)));
  return p_value(r);
}
__device__ __forceinline__ float2 p_fma(float2 a, float2 b, float2 c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(p_bits(a)), "l"(p_bits(b)), "l"(p_bits(c)));
  return p_value(r);
}
// A product that may feed an add, as two scalar instructions (the same time in the float32 pipe):
// the compiler fuses a packed product into a following packed add, .rn or not, which would round
// once where the scalar code rounds twice.
__device__ __forceinline__ float2 p_mul_rn(float2 a, float2 b) { return make_float2(__fmul_rn(a.x, b.x), __fmul_rn(a.y, b.y)); }
__device__ __forceinline__ float2 p_dup(float s) { return make_float2(s, s); }
__device__ __forceinline__ cpair c_add(cpair a, cpair b) { return {p_add(a.re, b.re), p_add(a.im, b.im)}; }
__device__ __forceinline__ cpair c_sub(cpair a, cpair b) { return {p_sub(a.re, b.re), p_sub(a.im, b.im)}; }
// both lanes by the same factor w (rounded as c_mul(float2, float2))
__device__ __forceinline__ cpair c_mul(cpair a, float2 w) {
  const float2 wr = p_dup(w.x), wi = p_dup(w.y), nwi = p_dup(-w.y);
  return {p_fma(a.re, wr, p_mul(a.im, nwi)), p_fma(a.re, wi, p_mul(a.im, wr))};
}
// lane by lane: a.lane0 * s.x, a.lane1 * s.y
__device__ __forceinline__ cpair c_scale(cpair a, float2 s) { return {p_mul_rn(a.re, s), p_mul_rn(a.im, s)}; }
template <bool INV>
__device__ __forceinline__ cpair c_add_rot(cpair a, cpair b) {
  return INV ? cpair{p_sub(a.re, b.im), p_add(a.im, b.re)} : cpair{p_add(a.re, b.im), p_sub(a.im, b.re)};
}
template <bool INV>
__device__ __forceinline__ cpair c_sub_rot(cpair a, cpair b) {
  return c_add_rot<!INV>(a, b);
}
__device__ __forceinline__ cpair c_fma(float s, cpair a, cpair b) {
  return {p_fma(p_dup(s), a.re, b.re), p_fma(p_dup(s), a.im, b.im)};
}
__device__ __forceinline__ cpair c_fma_i(float s, cpair b, cpair a) {
  return {p_fma(p_dup(-s), b.im, a.re), p_fma(p_dup(s), b.re, a.im)};
}

// Compile-time sine/cosine (Taylor series in double; arguments in [0, 2 pi)) for the constant
// twiddles inside the small in-register DFTs.
constexpr double kPi = 3.14159265358979323846264338327950288;
constexpr double cx_cos(double x) {
  double term = 1.0, sum = 1.0;
  for (int n = 1; n < 40; ++n) {
    term *= -x * x / ((2.0 * n - 1.0) * (2.0 * n));
    sum += term;
  }
  return sum;
}
constexpr double cx_sin(double x) {
  double term = x, sum = x;
  for (int n = 1; n < 40; ++n) {
    term *= -x * x / ((2.0 * n) * (2.0 * n + 1.0));
    sum += term;
  }
  return sum;
}

template <int R, int K, bool INV>
struct ConstTw {
  static constexpr float re = (float)cx_cos(2.0 * kPi * K / R);
  static constexpr float im = (INV ? 1.0f : -1.0f) * (float)cx_sin(2.0 * kPi * K / R);
};

// x * exp(-+2 pi i K / R) (a quarter turn is left to c_add_rot / c_sub_rot)
template <int R, int K, bool INV, class V>
__device__ __forceinline__ V mul_const_tw(V x) {
  if constexpr (K == 0) {
    return x;
  } else {
    return c_mul(x, make_float2(ConstTw<R, K, INV>::re, ConstTw<R, K, INV>::im));
  }
}

// ---- small in-register DFTs (V: float2, one value, or cpair, two at once) -----------------
template <int R, bool INV>
struct DFT;

template <bool INV>
struct DFT<2, INV> {
  template <class V>
  __device__ __forceinline__ static void run(V* v) {
    const V a = v[0], b = v[1];
    v[0] = c_add(a, b);
    v[1] = c_sub(a, b);
  }
};

template <bool INV>
struct DFT<3, INV> {
  template <class V>
  __device__ __forceinline__ static void run(V* v) {
    // omega = exp(-+2 pi i / 3) = -1/2 + i s,  s = -+sqrt(3)/2
    constexpr float s = INV ? 0.866025403784438647f : -0.866025403784438647f;
    const V t1 = c_add(v[1], v[2]);
    const V t2 = c_fma(-0.5f, t1, v[0]);
    const V t3 = c_sub(v[1], v[2]);
    v[0] = c_add(v[0], t1);
    v[1] = c_fma_i(s, t3, t2);
    v[2] = c_fma_i(-s, t3, t2);
  }
};

template <bool INV>
struct DFT<4, INV> {
  template <class V>
  __device__ __forceinline__ static void run(V* v) {
    const V t0 = c_add(v[0], v[2]), t1 = c_sub(v[0], v[2]);
    const V t2 = c_add(v[1], v[3]), t3 = c_sub(v[1], v[3]);
    v[0] = c_add(t0, t2);
    v[2] = c_sub(t0, t2);
    v[1] = c_add_rot<INV>(t1, t3);
    v[3] = c_sub_rot<INV>(t1, t3);
  }
};

// Even composite radices R = 2H (6, 8, 12, 16): one radix-2 decimation-in-time split.
template <int R, bool INV>
struct DFT {
  static_assert(R % 2 == 0 && R <= 16, "unsupported radix");
  static constexpr int H = R / 2;
  template <int K, class V>
  __device__ __forceinline__ static void combine_one(V* v, const V& e, const V& o) {
    if constexpr (4 * K == R) {
      v[K] = c_add_rot<INV>(e, o);
      v[K + H] = c_sub_rot<INV>(e, o);
    } else {
      const V p = mul_const_tw<R, K, INV>(o);
      v[K] = c_add(e, p);
      v[K + H] = c_sub(e, p);
    }
  }
  template <class V, int... K>
  __device__ __forceinline__ static void combine(V* v, const V* e, const V* o, std::integer_sequence<int, K...>) {
    (combine_one<K>(v, e[K], o[K]), ...);
  }
  template <class V>
  __device__ __forceinline__ static void run(V* v) {
    V e[H], o[H];
#pragma unroll
    for (int i = 0; i < H; ++i) {
      e[i] = v[2 * i];
      o[i] = v[2 * i + 1];
    }
    DFT<H, INV>::run(e);
    DFT<H, INV>::run(o);
    combine(v, e, o, std::make_integer_sequence<int, H>{});
  }
};

// ---- size table: radix list (product N) and elements per thread E --------------------------
template <int... Rs>
struct Radices {};

template <int N>
struct FFTConf;
#define COLA_FFT_CONF(N_, E_, ...)            \
  template <>                                 \
  struct FFTConf<N_> {                        \
    static constexpr int N = N_;              \
    static constexpr int E = E_;              \
    static constexpr int T = N_ / E_;         \
    using radices = Radices<__VA_ARGS__>;     \
  };
COLA_FFT_CONF(16, 16, 16)
COLA_FFT_CONF(24, 24, 8, 3)
COLA_FFT_CONF(32, 8, 8, 4)
COLA_FFT_CONF(48, 12, 4, 4, 3)
COLA_FFT_CONF(64, 8, 8, 8)
COLA_FFT_CONF(96, 24, 8, 12)
COLA_FFT_CONF(128, 16, 16, 8)
COLA_FFT_CONF(192, 24, 8, 8, 3)
COLA_FFT_CONF(256, 16, 16, 16)
COLA_FFT_CONF(384, 24, 8, 8, 6)
COLA_FFT_CONF(512, 8, 8, 8, 8)
COLA_FFT_CONF(768, 24, 8, 8, 12)
COLA_FFT_CONF(1024, 16, 16, 16, 4)
COLA_FFT_CONF(1536, 24, 8, 8, 8, 3)
COLA_FFT_CONF(2048, 16, 16, 16, 8)
#undef COLA_FFT_CONF

// Radix variants: FFTConfV<N, 0> is FFTConf<N>; FFTConfV<N, 1> is a second factorisation with a
// different number of elements per thread (the ensemble autotuner times both).
template <int N, int V>
struct FFTConfV : FFTConf<N> {};
#define COLA_FFT_ALT(N_, E_, ...)             \
  template <>                                 \
  struct FFTConfV<N_, 1> {                    \
    static constexpr int N = N_;              \
    static constexpr int E = E_;              \
    static constexpr int T = N_ / E_;         \
    using radices = Radices<__VA_ARGS__>;     \
  };
COLA_FFT_ALT(32, 4, 4, 4, 2)
COLA_FFT_ALT(48, 24, 8, 6)
COLA_FFT_ALT(64, 16, 16, 4)
COLA_FFT_ALT(96, 12, 4, 4, 6)
COLA_FFT_ALT(128, 8, 8, 4, 4)
COLA_FFT_ALT(192, 12, 4, 4, 12)
COLA_FFT_ALT(256, 8, 8, 8, 4)
#undef COLA_FFT_ALT

template <class L>
struct FirstRadix;
template <int R0, int... Rs>
struct FirstRadix<Radices<R0, Rs...>> {
  static constexpr int value = R0;
};

// padded index of the row-layout exchange buffers: the first Stockham stage stores with stride
// R0 (its radix) between consecutive threads, so one pad slot per R0 entries (per 8 for R0 <= 8)
// puts those stores on distinct banks (row pitch xrow_ld, 8 mod 16, leaves room for either)
template <int R0>
__device__ __forceinline__ int xpad(int n) {
  constexpr int shift = R0 >= 16 ? 4 : 3;
  return n + (n >> shift);
}
template <int R0, int... Rs>
__host__ __device__ constexpr int last_radix_of(Radices<R0, Rs...>) {
  int last = R0;
  for (int r : {R0, Rs...}) last = r;
  return last;
}
template <class C>
__host__ __device__ constexpr int first_radix() {
  return FirstRadix<typename C::radices>::value;
}
template <int M>
__host__ __device__ constexpr int xrow_ld() {
  return ((M + 1 + ((M + 1) >> 3) + 1) + 15) / 16 * 16 + 8;
}

// ---- stage twiddle tables in shared memory ------------------------------------------------
// A stage of radix R after NS combined points multiplies input r of butterfly j (0 < r < R) by
// w^r, w = exp(-2 pi i (j mod NS) / (NS R)).  From the base table these are R - 1 scattered
// 8-byte loads per butterfly; a block may instead copy every stage's twiddles once into shared
// memory, butterfly by butterfly, and read them as 16-byte pairs.  Row pitch stw_pitch(R) float2
// (an even count, 2 mod 4): eight consecutive butterflies' pair loads fall on distinct banks.
// A tight table (TIGHT) gives radix-4 stages pitch 4 instead of 6: two-way bank conflicts on
// the pair loads, a third less shared memory for the largest stage of a 1024-point transform.
__host__ __device__ constexpr int stw_pitch(int R, bool tight = false) {
  const int pairs = R / 2;  // ceil((R - 1) / 2)
  return (tight && R == 4) ? 4 : 2 * pairs + ((pairs % 2 == 0) ? 2 : 0);
}
template <int... Rs>
__host__ __device__ constexpr int stw_offset_of(Radices<Rs...>, int ns_target, bool tight = false) {
  int ns = 1, off = 0;
  for (int r : {Rs...}) {
    if (ns == ns_target) return off;
    if (ns > 1) off += ns * stw_pitch(r, tight);
    ns *= r;
  }
  return off;
}
// float2 entries of the table of configuration C
template <class C, bool TIGHT = false>
__host__ __device__ constexpr int stw_size() {
  return stw_offset_of(typename C::radices{}, C::N, TIGHT);
}

// Fill the table of configuration C from the base table tw (stage twiddle m at tw[m * TWS]):
// threads tid = 0 .. nth - 1 of the block; the first use comes after the transform's first
// block barrier, so the fill needs no barrier of its own.
template <int N, int TWS, bool TIGHT, int... Rs>
__device__ __forceinline__ void stw_fill_stages(Radices<Rs...>, float2* dst, const float2* __restrict__ tw,
                                                int tid, int nth) {
  int ns = 1, off = 0;
  (
      [&] {
        constexpr int R = Rs;
        if (ns > 1) {
          const int p = stw_pitch(R, TIGHT), cnt = ns * (R - 1), step = N / (ns * R);
          for (int i = tid; i < cnt; i += nth) {
            const int j = i / (R - 1), r = i - j * (R - 1) + 1;
            dst[off + j * p + r - 1] = __ldg(tw + (int64_t)j * r * step * TWS);
          }
          off += ns * p;
        }
        ns *= R;
      }(),
      ...);
}
template <class C, int TWS, bool TIGHT = false>
__device__ __forceinline__ void stw_fill(float2* dst, const float2* __restrict__ tw, int tid, int nth) {
  stw_fill_stages<C::N, TWS, TIGHT>(typename C::radices{}, dst, tw, tid, nth);
}

// twiddle source reading the shared-memory table of configuration C (16-byte aligned)
template <class C, bool TIGHT = false>
struct SmemTw {
  const float2* base;
  template <int R, int NS, bool INV, class V>
  __device__ __forceinline__ void apply(unsigned j, V* x) const {
    constexpr int off = stw_offset_of(typename C::radices{}, NS, TIGHT), p = stw_pitch(R, TIGHT);
    const float4* q = reinterpret_cast<const float4*>(base + off + j * p);
#pragma unroll
    for (int k = 0; k < R / 2; ++k) {
      const float4 w2 = q[k];
      const int r = 2 * k + 1;
      x[r] = c_mul(x[r], make_float2(w2.x, INV ? -w2.y : w2.y));
      if (r + 1 < R) x[r + 1] = c_mul(x[r + 1], make_float2(w2.z, INV ? -w2.w : w2.w));
    }
  }
};

// ---- Stockham stages --------------------------------------------------------------------
// exchange slot base + off, where off is a constant once the loops are unrolled and the two share
// no bit below 16: the buffer's own at(base, off) where it has one (a permuted layout)
template <class Mem, class = void>
struct HasAt : std::false_type {};
template <class Mem>
struct HasAt<Mem, std::void_t<decltype(std::declval<const Mem&>().at(0, 0))>> : std::true_type {};
template <class Mem>
__device__ __forceinline__ decltype(auto) mem_at(Mem& mem, int base, int off) {
  if constexpr (HasAt<Mem>::value) return mem.at(base, off);
  else return mem(base + off);
}
// barrier of the threads that share an exchange buffer: the buffer's own sync() where it has one
// (a part of the block), else the block's
template <class Mem, class = void>
struct HasSync : std::false_type {};
template <class Mem>
struct HasSync<Mem, std::void_t<decltype(std::declval<const Mem&>().sync())>> : std::true_type {};
template <class Mem>
__device__ __forceinline__ void stage_sync(const Mem& mem) {
  if constexpr (HasSync<Mem>::value) mem.sync();
  else __syncthreads();
}

template <int N, int E, int TWS, bool INV>
struct Stockham {
  static constexpr int T = N / E;

  // Butterfly j = t + T q of a stage (0 <= t < T).  Two compile-time cases spare the per-element
  // division by NS: if NS divides T, j / NS = t / NS + q T / NS and j mod NS = t mod NS for every
  // q; if NS >= T E / R, every j is below NS (j / NS = 0, j mod NS = j).
  template <int R, int NS>
  __device__ __forceinline__ static unsigned j_mod(unsigned t, int q) {
    if constexpr (T % NS == 0) return t % NS;
    else if constexpr (NS >= T * (E / R)) return t + T * q;
    else return (t + T * q) % NS;
  }

  // twiddle and in-register DFT of every butterfly this thread owns (butterfly j = t + T q,
  // inputs v[q R + r] = x[j + r N/R]), for a stage of radix R after NS points were combined
  // (tw: the base table, or an SmemTw stage table)
  template <int R, int NS, class V, class TW>
  __device__ __forceinline__ static void compute(V (&v)[E], int t, const TW& tw) {
#pragma unroll
    for (int q = 0; q < E / R; ++q) {
      if constexpr (NS > 1) {
        const unsigned jj = j_mod<R, NS>((unsigned)t, q);
        if constexpr (!std::is_class<TW>::value) {
#pragma unroll
          for (int r = 1; r < R; ++r) {
            float2 w = __ldg(tw + jj * (r * (N / (NS * R)) * TWS));
            if (INV) w.y = -w.y;
            v[q * R + r] = c_mul(v[q * R + r], w);
          }
        } else {
          tw.template apply<R, NS, INV>(jj, &v[q * R]);
        }
      }
      DFT<R, INV>::run(&v[q * R]);
    }
  }

  // output position of element r of butterfly j = t + T q
  template <int R, int NS>
  __device__ __forceinline__ static int out_index(int t, int q, int r) {
    if constexpr (T % NS == 0) {
      const unsigned ut = (unsigned)t;
      return (int)((ut / NS) * (NS * R) + ut % NS) + q * (T * R) + r * NS;
    } else if constexpr (NS >= T * (E / R)) {
      return t + T * q + r * NS;
    } else {
      const int j = t + T * q;
      return (j / NS) * NS * R + (j % NS) + r * NS;
    }
  }

  // out_index as a part that depends on the thread and one that does not (constant after unrolling)
  template <int R, int NS>
  __device__ __forceinline__ static int out_base(int t) {
    if constexpr (T % NS == 0) return (int)(((unsigned)t / NS) * (NS * R) + (unsigned)t % NS);
    else return t;
  }
  template <int R, int NS>
  __device__ __forceinline__ static constexpr int out_off(int q, int r) {
    if constexpr (T % NS == 0) return q * (T * R) + r * NS;
    else return T * q + r * NS;
  }
  // exchange after the stage (R, NS): this thread's outputs to the buffer, the next stage's inputs from it
  template <int R, int NS, int R2, class V, class Mem>
  __device__ __forceinline__ static void exchange(V (&v)[E], int t, Mem& mem) {
    constexpr bool split = T % NS == 0 || NS >= T * (E / R);
    const int base = split ? out_base<R, NS>(t) : 0;
#pragma unroll
    for (int q = 0; q < E / R; ++q)
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if constexpr (split) mem_at(mem, base, out_off<R, NS>(q, r)) = v[q * R + r];
        else mem_at(mem, out_index<R, NS>(t, q, r), 0) = v[q * R + r];
      }
    stage_sync(mem);
#pragma unroll
    for (int q = 0; q < E / R2; ++q)
#pragma unroll
      for (int r = 0; r < R2; ++r) v[q * R2 + r] = mem_at(mem, t, T * q + r * (N / R2));
  }

  // Run the stages NS.. of the radix list.  v holds the inputs of the first listed stage.
  // mem(n) -> V& : exchange buffer slot for element n of this thread's sequence.
  // store(n, x)       : final output of element n.
  template <int NS, int R, int... Rest, class V, class TW, class Mem, class Store>
  __device__ __forceinline__ static void run(V (&v)[E], int t, const TW& tw, Mem& mem, Store& store) {
    compute<R, NS>(v, t, tw);
    if constexpr (sizeof...(Rest) == 0) {
      static_assert(NS * R == N, "radix list does not multiply to N");
      stage_sync(mem);
#pragma unroll
      for (int q = 0; q < E / R; ++q)
#pragma unroll
        for (int r = 0; r < R; ++r) store(out_index<R, NS>(t, q, r), v[q * R + r]);
    } else {
      stage_sync(mem);
      exchange<R, NS, FirstRadix<Radices<Rest...>>::value>(v, t, mem);
      run<NS * R, Rest...>(v, t, tw, mem, store);
    }
  }

  // The stages NS.. with the result left in registers, in the last stage's order.  after_reads()
  // is called once this thread has read its inputs of the last stage.
  template <int NS, int R, int... Rest, class V, class TW, class Mem, class Hook>
  __device__ __forceinline__ static void run_regs(V (&v)[E], int t, const TW& tw, Mem& mem, Hook& after_reads) {
    compute<R, NS>(v, t, tw);
    if constexpr (sizeof...(Rest) > 0) {
      stage_sync(mem);
      exchange<R, NS, FirstRadix<Radices<Rest...>>::value>(v, t, mem);
      if constexpr (sizeof...(Rest) == 1) after_reads();
      run_regs<NS * R, Rest...>(v, t, tw, mem, after_reads);
    } else {
      static_assert(NS * R == N && NS > 1, "radix list of at least two stages that multiplies to N");
    }
  }
  template <int... Rs, class V, class TW, class Mem, class Hook>
  __device__ __forceinline__ static void run_regs_all(Radices<Rs...>, V (&v)[E], int t, const TW& tw, Mem& mem,
                                                      Hook& after_reads) {
    run_regs<1, Rs...>(v, t, tw, mem, after_reads);
  }

  template <int... Rs, class V, class TW, class Mem, class Store>
  __device__ __forceinline__ static void run_all(Radices<Rs...>, V (&v)[E], int t, const TW& tw, Mem& mem,
                                                 Store& store) {
    run<1, Rs...>(v, t, tw, mem, store);
  }
};

// Convenience wrapper: load the first-stage inputs with load(n) and run the whole transform.
template <int N, int TWS, bool INV, class C = FFTConf<N>, class TW, class Load, class Mem, class Store>
__device__ __forceinline__ void fft_1d(int t, const TW& tw, Load& load, Mem& mem, Store& store) {
  static_assert(C::N == N, "configuration of another length");
  constexpr int E = C::E, T = C::T;
  constexpr int R0 = FirstRadix<typename C::radices>::value;
  decltype(load(0)) v[E];  // float2 or cpair
#pragma unroll
  for (int q = 0; q < E / R0; ++q)
#pragma unroll
    for (int r = 0; r < R0; ++r) v[q * R0 + r] = load(t + T * q + r * (N / R0));
  Stockham<N, E, TWS, INV>::run_all(typename C::radices{}, v, t, tw, mem, store);
}

// Transform of values in registers: u[m] is element n = t + T m (0 <= m < E) before and after.
// Both the first stage's inputs and the last stage's outputs of a thread are the elements
// congruent to t modulo T, so a thread can go from one transform to the next without an exchange.
// (The first exchange starts with a block barrier; none follows the last one's reads.)
// after_reads() runs when this thread has read the last stage's inputs.
template <int N, int TWS, bool INV, class C = FFTConf<N>, class V, class TW, class Mem, class Hook>
__device__ __forceinline__ void fft_regs(V (&u)[C::E], int t, const TW& tw, Mem& mem, Hook& after_reads) {
  static_assert(C::N == N, "configuration of another length");
  constexpr int E = C::E;
  constexpr int R0 = FirstRadix<typename C::radices>::value, RL = last_radix_of(typename C::radices{});
  V v[E];
#pragma unroll
  for (int q = 0; q < E / R0; ++q)
#pragma unroll
    for (int r = 0; r < R0; ++r) v[q * R0 + r] = u[q + r * (E / R0)];
  Stockham<N, E, TWS, INV>::run_regs_all(typename C::radices{}, v, t, tw, mem, after_reads);
#pragma unroll
  for (int q = 0; q < E / RL; ++q)
#pragma unroll
    for (int r = 0; r < RL; ++r) u[q + r * (E / RL)] = v[q * RL + r];
}
template <int N, int TWS, bool INV, class C = FFTConf<N>, class V, class TW, class Mem>
__device__ __forceinline__ void fft_regs(V (&u)[C::E], int t, const TW& tw, Mem& mem) {
  auto none = [] {};
  fft_regs<N, TWS, INV, C>(u, t, tw, mem, none);
}

}  // namespace cola

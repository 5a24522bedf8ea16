// Kernels for problems too small to fill the GPU with the 32x32 and larger tiles of lba_kernel.cuh.
//
// There a launch takes as long as one CTA's chain of K steps, and the step itself, not the machine's rate, is what
// counts.  The two accumulation orders leave different ways out:
//   lba_split_kernel  chunks of 16: the chunk sums C_j do not depend on each other, so the G warps of a CTA each form every
//                     G-th chunk sum of one output tile, hand them over through shared memory, and fold G chunks per round in
//                     chunk order, a few outputs per thread: T <- Q_acc(C_j + T).  K is divided by G; a fold is one
//                     addition where a chunk is sixteen.  A warp loads and decodes its own slabs: one barrier per round.
//   lba_chain_kernel  sequential: nothing can be divided, so every thread carries as few chains as a packed instruction
//                     allows (one pair), and other warps decode meanwhile.
// Results are those of the packed kernel bit for bit: the same steps, in the same order.
#pragma once
#include "lba_kernel.cuh"

namespace lba {

// One FMAq step on a pair of outputs and the fold, with the constants they need.  SAT: Q_prod cuts and saturates (each a
// no-op where unreachable); RNE as in lba_contract_packed_kernel.
template <bool SAT, int RNE>
struct PairSteps {
  u64 cc, acc_k1, acc_k2, prod_k1, prod_k2;
  uint32_t mask, pmask;
  float sat, psat;

  __device__ __forceinline__ explicit PairSteps(const Problem& p)
      : cc(pack2(p.c, p.c)), acc_k1(pack2(p.acc_k1, p.acc_k1)), acc_k2(pack2(p.acc_k2, p.acc_k2)),
        prod_k1(pack2(p.prod_k1, p.prod_k1)), prod_k2(pack2(p.prod_k2, p.prod_k2)), mask(p.qa.mask), pmask(p.qp.mask),
        sat(p.qa.sat), psat(p.qp.sat) {}

  __device__ __forceinline__ u64 product(u64 a, u64 b) const { return cut(mul2_ftz(b, a)); }
  __device__ __forceinline__ u64 cut(u64 pr) const {
    if (SAT) {
      if (RNE) pr = rne2_fp(pr, prod_k1, prod_k2);
      float lo, hi;
      unpack2(pr, lo, hi);
      if (!RNE) {
        lo = and_bits(lo, pmask);
        hi = and_bits(hi, pmask);
      }
      pr = pack2(clamp_mag(lo, psat), clamp_mag(hi, psat));
    }
    return pr;
  }
  template <bool CLAMP>
  __device__ __forceinline__ u64 round(u64 t) const {
    float lo, hi;
    if (RNE == 0) {
      unpack2(t, lo, hi);
      lo = and_bits(lo, mask);
      hi = and_bits(hi, mask);
    } else {
      if (RNE == 1) {
        t = rne2_fp(t, acc_k1, acc_k2);
      } else {
        unpack2(t, lo, hi);
        t = rne2_bf16(lo, hi);
      }
      if (!CLAMP) return t;
      unpack2(t, lo, hi);
    }
    if (CLAMP) {
      lo = clamp_mag(lo, sat);
      hi = clamp_mag(hi, sat);
    }
    return pack2(lo, hi);
  }
  template <bool CLAMP>
  __device__ __forceinline__ u64 step(u64 a, u64 b, u64 s) const {
    return add<CLAMP>(product(a, b), s);
  }
  template <bool CLAMP>
  __device__ __forceinline__ u64 add(u64 pr, u64 s) const {
    return round<CLAMP>(RNE ? fma2_rn_ftz(cc, pr, s) : fma2_rz_ftz(cc, pr, s));
  }
  __device__ __forceinline__ u64 fold(u64 c, u64 t) const {
    return round<true>(RNE ? add2_rn_ftz(c, t) : add2_rz_ftz(c, t));
  }
};

// sixteen bytes of a row -> scaled binary32, k-major in shared memory, `stride` elements from one k to the next; returns the
// squared 2-norm, scaled
__device__ __forceinline__ float stage_row(const Problem& p, const uint4& row, float mul, float* dst, int stride) {
  const auto store = [&](int k, u64 v) { unpack2(v, dst[k * stride], dst[(k + 1) * stride]); };
  const u64 mul2 = pack2(mul, mul);
  const float n2 = p.in_m4e3 ? decode_row<true>(row, mul2, mul2, store) : decode_row<false>(row, mul2, mul2, store);
  return n2 == 0.0f ? 0.0f : n2 * p.nrm_scale;  // (the scale may be infinite)
}

// micro-tile operands of one k-step: TM rows from a0, each as both halves of a factor (see both2), TN columns from b0
template <int TM, int TN>
__device__ __forceinline__ void load_step(const float* a0, const float* b0, u64 (&a)[TM], u64 (&b2)[TN / 2]) {
  static_assert(TM == 2 || TM == 4, "one load");
  const typename std::conditional<TM == 4, ulonglong2, ulonglong1>::type v = *reinterpret_cast<decltype(&v)>(a0);
  both2(v.x, a[0], a[1]);
  if constexpr (TM == 4) both2(v.y, a[2], a[3]);
#pragma unroll
  for (int j = 0; j < TN; j += 4) {
    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(b0 + j);
    b2[j / 2] = v.x;
    b2[j / 2 + 1] = v.y;
  }
}

// back to a real value, +0 for every zero, scales and bias in binary32
__device__ __forceinline__ float finish(const Problem& p, float s, float sa, int64_t n) {
  float y = __fmul_rn(__fmul_rn(s, p.un1), p.un2);
  y = (y == 0.0f) ? 0.0f : y;
  const float r = __fmul_rn(__fmul_rn(y, sa), p.sb[p.sb_per_col ? n : 0]);
  return p.bias ? __fadd_rn(r, p.bias[n]) : r;
}

// ------------------------------------------------------------------ chunks of 16: chunk sums spread over the warps of a CTA
template <int BM, int BN, int TM, int TN, int G>
struct SplitShape {
  static_assert((BM / TM) * (BN / TN) == 32, "one warp holds the whole tile");
  static constexpr int OUTS = BM * BN / (32 * G) < 2 ? 2 : BM * BN / (32 * G);  // outputs a thread folds
  static constexpr int FOLDERS = BM * BN / OUTS;                                 // threads that fold
  static_assert(OUTS == 2 || OUTS == 4, "consecutive columns of one row");
  static constexpr bool TWO_ROWS = BM == 32;  // a lane decodes a row of A and a row of B, or one of either
  static constexpr size_t A_BYTES = sizeof(float) * BK * BM, B_BYTES = sizeof(float) * BK * BN;
  static constexpr size_t SMEM = G * (A_BYTES + B_BYTES) + sizeof(float) * 2 * G * BM * BN;
};

template <int BM, int BN, int TM, int TN, int G, bool SAT, int RNE, int LD>
__global__ void __launch_bounds__(32 * G) lba_split_kernel(const Problem p) {
  typedef SplitShape<BM, BN, TM, TN, G> S;
  constexpr int TX = BN / TN, PN = TN / 2, OUTS = S::OUTS;
  typedef RowLoader<BM, BN, 32, LD> Loader;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  float (*const As)[BM] = reinterpret_cast<float (*)[BM]>(smem_raw + w * (S::A_BYTES + S::B_BYTES));
  float (*const Bs)[BN] = reinterpret_cast<float (*)[BN]>(smem_raw + w * (S::A_BYTES + S::B_BYTES) + S::A_BYTES);
  float* const sums = reinterpret_cast<float*>(smem_raw + G * (S::A_BYTES + S::B_BYTES));  // [2][G][BM * BN]
  const int tx = lane % TX, ty = lane / TX;
  const int64_t m0 = (int64_t)blockIdx.x * BM, n0 = (int64_t)blockIdx.y * BN;
  const int nslab = (int)((p.K + BK - 1) / BK);
  const int rounds = (nslab + G - 1) / G;
  const PairSteps<SAT, RNE> steps(p);

  Loader loader;
  after_previous();
  loader.init(p, lane, m0, n0);
  uint4 raw[Loader::LPT];
  for (int i = 0; i < w; ++i) loader.skip_slab(p);
  if (w < nslab) loader.fetch_apart(p, lane, w, raw);

  u64 t2[OUTS / 2];
#pragma unroll
  for (int o = 0; o < OUTS / 2; ++o) t2[o] = 0ull;

  for (int q = 0; q < rounds; ++q) {
    const int s = q * G + w;
    float* const mine = sums + ((q & 1) * G + w) * (BM * BN);
    if (s < nslab) {
      float na = 0.0f, nb = 0.0f;
      if constexpr (S::TWO_ROWS) {
        static_assert(!S::TWO_ROWS || (BM == 32 && BN == 32), "a row of A and a row of B per lane");
        na = stage_row(p, loader.take(p, 0, s, raw[0]), p.pk_a, &As[0][lane], BM);
        nb = stage_row(p, loader.take(p, Loader::LPT - 1, s, raw[Loader::LPT - 1]), p.pk_b, &Bs[0][lane], BN);
      } else {
        static_assert(S::TWO_ROWS || (BM == 16 && BN == 16), "a row of A or of B per lane");
        const bool is_a = lane < BM;
        const float n2 = stage_row(p, loader.take(p, 0, s, raw[0]), is_a ? p.pk_a : p.pk_b,
                                    is_a ? &As[0][lane] : &Bs[0][lane - BM], BM);
        na = is_a ? n2 : 0.0f;
        nb = is_a ? 0.0f : n2;
      }
      na = __uint_as_float(__reduce_max_sync(0xFFFFFFFFu, __float_as_uint(na)));
      nb = __uint_as_float(__reduce_max_sync(0xFFFFFFFFu, __float_as_uint(nb)));
      __syncwarp();
      if (s + G < nslab) {
#pragma unroll 1
        for (int i = 1; i < G; ++i) loader.skip_slab(p);
        loader.fetch_apart(p, lane, s + G, raw);
      }
      // the chunk starts from zero: |S_i| <= ||x|| ||w|| (see the packed kernel)
      const float grow = sqrt_approx(na * nb) * 1.01f * p.slab_factor;
      u64 acc[TM][PN];
      auto slab = [&](auto clamp_tag) {
        constexpr bool CLAMP = decltype(clamp_tag)::value;
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
          for (int j = 0; j < PN; ++j) acc[i][j] = 0ull;
        u64 a2[2][TM], b2[2][PN];  // the operands of the next step are on their way while a step is computed
        load_step<TM, TN>(&As[0][ty * TM], &Bs[0][tx * TN], a2[0], b2[0]);
#pragma unroll (CLAMP ? 1 : 4)
        for (int kk = 0; kk < BK; kk += 2) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            if (kk + h + 1 < BK) load_step<TM, TN>(&As[kk + h + 1][ty * TM], &Bs[kk + h + 1][tx * TN], a2[h ^ 1], b2[h ^ 1]);
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
              for (int j = 0; j < PN; ++j) acc[i][j] = steps.template step<CLAMP>(a2[h][i], b2[h][j], acc[i][j]);
          }
        }
      };
      if (grow < p.clamp_lim) slab(std::false_type());
      else slab(std::true_type());
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < PN; j += 2) {
          u64* const dst = reinterpret_cast<u64*>(mine + (ty * TM + i) * BN + tx * TN + 2 * j);
          *reinterpret_cast<ulonglong2*>(dst) = make_ulonglong2(acc[i][j], acc[i][j + 1]);
        }
    }
    __syncthreads();  // the next round writes the other half of `sums`, and the one after that follows its barrier
    if (tid >= S::FOLDERS) continue;  // whole warps
    const int have = nslab - q * G < G ? nslab - q * G : G;
    const float* const row = sums + (q & 1) * G * (BM * BN) + tid * OUTS;
#pragma unroll
    for (int j = 0; j < G; ++j) {
      if (j < have) {
        const u64* const c = reinterpret_cast<const u64*>(row + j * (BM * BN));
        if constexpr (OUTS == 2) {
          t2[0] = steps.fold(*c, t2[0]);
        } else {
          const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(c);
          t2[0] = steps.fold(v.x, t2[0]);
          t2[OUTS / 2 - 1] = steps.fold(v.y, t2[OUTS / 2 - 1]);
        }
      }
    }
  }

  const int64_t m = m0 + tid * OUTS / BN, n = n0 + tid * OUTS % BN;
  if (tid >= S::FOLDERS || m >= p.M) return;
  float o[OUTS];
#pragma unroll
  for (int i = 0; i < OUTS / 2; ++i) unpack2(t2[i], o[2 * i], o[2 * i + 1]);
  const float sa = p.sa[p.sa_per_row ? m : 0];
  float* const dst = p.out + (int64_t)blockIdx.z * p.batch_out + m * p.N + n;
#pragma unroll
  for (int i = 0; i < OUTS; ++i)
    if (n + i < p.N) o[i] = finish(p, o[i], sa, n + i);
  if (n + OUTS - 1 < p.N && (reinterpret_cast<uintptr_t>(dst) & (4 * OUTS - 1)) == 0) {
    if constexpr (OUTS == 2) *reinterpret_cast<float2*>(dst) = make_float2(o[0], o[1]);
    else *reinterpret_cast<float4*>(dst) = make_float4(o[0], o[1], o[2], o[OUTS - 1]);
  } else {
#pragma unroll
    for (int i = 0; i < OUTS; ++i)
      if (n + i < p.N) dst[i] = o[i];
  }
}

// ------------------------------------------------------------------ sequential: one pair of chains per thread
// 16 x 16 outputs.  Four warps carry the chains; four more decode, each every fourth slab, because one warp takes three
// times as long to decode a slab of the tile's 32 rows as the chains take to consume it.  They meet every four slabs.
// Twelve slabs are kept: the four being consumed, the four after them (a consumer reads eight steps ahead) and the four
// being decoded.  The chain itself is one FMA and one mask per step: a consumer loads the operands of eight steps in one
// go, while it adds the products of the eight before, and multiplies them in the second half of those, so that
// neither shared-memory latency nor the multiplication sits in the chain.
constexpr int CHAIN_SLABS = 4;
constexpr int CHAIN_THREADS = 128 + 32 * CHAIN_SLABS;

template <bool SAT, int RNE, int LD>
__global__ void __launch_bounds__(CHAIN_THREADS) lba_chain_kernel(const Problem p) {
  constexpr int BM = 16, BN = 16, RING = 3 * CHAIN_SLABS;
  typedef RowLoader<BM, BN, 32, LD> Loader;
  static_assert(Loader::LPT == 1, "a lane decodes one row");
  __shared__ __align__(16) float As[RING][BK][BM];
  __shared__ __align__(16) float Bs[RING][BK][BN];
  __shared__ float bound[RING];  // ||x|| ||w|| of the slab's longest rows, as a fraction of 2^(e_max + 1)
  const int tid = threadIdx.x;
  const int64_t m0 = (int64_t)blockIdx.x * BM, n0 = (int64_t)blockIdx.y * BN;
  const int nslab = (int)((p.K + BK - 1) / BK);
  const int supers = (nslab + CHAIN_SLABS - 1) / CHAIN_SLABS;

  after_previous();
  if (tid >= 128) {
    const int lane = tid & 31, w = (tid - 128) >> 5;
    Loader loader;
    loader.init(p, lane, m0, n0);
    uint4 raw[1];
    for (int i = 0; i < w; ++i) loader.skip_slab(p);
    if (w < nslab) loader.fetch_apart(p, lane, w, raw);
    auto produce = [&](int s, int slot) {
      const uint4 row = loader.take(p, 0, s, raw[0]);
      if (s + CHAIN_SLABS < nslab) {
#pragma unroll 1
        for (int i = 1; i < CHAIN_SLABS; ++i) loader.skip_slab(p);
        loader.fetch_apart(p, lane, s + CHAIN_SLABS, raw);
      }
      float* const dst = lane < BM ? &As[slot][0][lane] : &Bs[slot][0][lane - BM];
      const float n2 = stage_row(p, row, lane < BM ? p.pk_a : p.pk_b, dst, BM);
      const unsigned na = __reduce_max_sync(0xFFFFFFFFu, lane < BM ? __float_as_uint(n2) : 0u);
      const unsigned nb = __reduce_max_sync(0xFFFFFFFFu, lane < BM ? 0u : __float_as_uint(n2));
      if (lane == 0) bound[slot] = sqrt_approx(__uint_as_float(na) * __uint_as_float(nb)) * 1.01f;
    };
    if (w < nslab) produce(w, w);
    if (CHAIN_SLABS + w < nslab) produce(CHAIN_SLABS + w, CHAIN_SLABS + w);
    __syncthreads();
    int slot = 2 * CHAIN_SLABS + w;
    for (int S = 0; S < supers; ++S) {
      const int s = (S + 2) * CHAIN_SLABS + w;
      if (s < nslab) produce(s, slot);
      slot = slot + CHAIN_SLABS < RING ? slot + CHAIN_SLABS : w;
      __syncthreads();
    }
    return;
  }

  const int tx = tid % 8, ty = tid / 8;
  const PairSteps<SAT, RNE> steps(p);
  u64 acc = 0ull;
  float u = 0.0f;  // upper bound of max |acc|, as a fraction of 2^(e_max + 1) (see the packed kernel)
  constexpr int H = BK / 2;
  float a[H];
  u64 b[H], pr[H];
  auto load = [&](int slot, int h) {
#pragma unroll
    for (int i = 0; i < H; ++i) {
      a[i] = As[slot][h * H + i][ty];
      b[i] = *reinterpret_cast<const u64*>(&Bs[slot][h * H + i][2 * tx]);
    }
  };
  __syncthreads();
  load(0, 0);
#pragma unroll
  for (int i = 0; i < H; ++i) pr[i] = steps.product(pack2(a[i], a[i]), b[i]);
  int slot = 0;
  // whether the clamp can act in a slab (see the packed kernel) is decided while the slab before it runs
  float grow = bound[0];
  bool fast = __all_sync(0xFFFFFFFFu, grow * p.slab_factor < p.clamp_lim);
  for (int S = 0; S < supers; ++S) {
    const int s_end = (S + 1) * CHAIN_SLABS < nslab ? (S + 1) * CHAIN_SLABS : nslab;
#pragma unroll 1
    for (int s = S * CHAIN_SLABS; s < s_end; ++s) {
      const int next = slot + 1 < RING ? slot + 1 : 0;
      const float grow_next = bound[next];
      auto slab = [&](auto clamp_tag) {
        constexpr bool CLAMP = decltype(clamp_tag)::value;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          load(h == 0 ? slot : next, h ^ 1);  // (after the last slab: a slot that nothing uses)
#pragma unroll
          for (int i = 0; i < H / 2; ++i) acc = steps.template add<CLAMP>(pr[i], acc);
          u64 nx[H];
#pragma unroll
          for (int i = H / 2; i < H; ++i) {
            acc = steps.template add<CLAMP>(pr[i], acc);
#pragma unroll
            for (int e = 2 * i - H; e < 2 * i - H + 2; ++e) nx[e] = steps.product(pack2(a[e], a[e]), b[e]);
          }
#pragma unroll
          for (int i = 0; i < H; ++i) pr[i] = nx[i];
        }
      };
      u = fminf((u + grow) * p.slab_factor, 1.0f);
      bool fast_next = __all_sync(0xFFFFFFFFu, (u + grow_next) * p.slab_factor < p.clamp_lim);
      if (fast) slab(std::false_type());
      else slab(std::true_type());
      if (!fast_next) {  // the carried bound may just be loose
        float lo, hi;
        unpack2(acc, lo, hi);
        u = fmaxf(fabsf(lo), fabsf(hi)) * p.inv_top;
        fast_next = __all_sync(0xFFFFFFFFu, (u + grow_next) * p.slab_factor < p.clamp_lim);
      }
      fast = fast_next;
      grow = grow_next;
      slot = next;
    }
    __syncthreads();
  }

  const int64_t m = m0 + ty, n = n0 + 2 * tx;
  if (m >= p.M) return;
  const float sa = p.sa[p.sa_per_row ? m : 0];
  float* const dst = p.out + (int64_t)blockIdx.z * p.batch_out + m * p.N + n;
  float o[2];
  unpack2(acc, o[0], o[1]);
  const bool both = n + 1 < p.N;
  if (n < p.N) o[0] = finish(p, o[0], sa, n);
  if (both) o[1] = finish(p, o[1], sa, n + 1);
  if (both && (reinterpret_cast<uintptr_t>(dst) & 7) == 0) {
    *reinterpret_cast<float2*>(dst) = make_float2(o[0], o[1]);
  } else {
    if (n < p.N) dst[0] = o[0];
    if (both) dst[1] = o[1];
  }
}

template <int RNE>
cudaError_t launch_small(int tile, int load, const Problem& p, cudaStream_t stream);

}  // namespace lba

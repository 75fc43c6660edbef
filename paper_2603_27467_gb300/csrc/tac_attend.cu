// Attention straight from TurboAngle records, for sm_103a.
//
// The consumer of the Sec. 3.1 reconstruction (the paper evaluates its codes
// through a model's attention but describes no kernel for it).  H and D are
// orthogonal and H is symmetric, so for a decoded key k^ = D H y^,
//   q . k^ = (H D q) . y^,      y^_2i + i y^_2i+1 = r^_i exp(2 pi i k_i / n),
// and the output sum_t p_t v^_t = D H (sum_t p_t y^V_t).  Scores are taken
// against the rotated query and values are accumulated in the rotated domain:
// one transform per query and one per output instead of one per cached token.
//
// Two kernels (flash-decoding split over tokens):
//   attend_partial  persistent CTAs of 8 warps over units of 256 tokens of one
//                   job; a CTA takes a contiguous range of units and a warp 32
//                   tokens of each (a batch).  Both contractions run on the
//                   tensor cores (mma.sync m16n8k16, fp16 operands, fp32 sums):
//                   the operands are decoded straight into the registers of the
//                   fragments, so nothing decoded touches memory.  Operands are
//                   split into fp16 parts that together keep what fp32 would:
//                   a decoded value r^ (cos, sin), in units of the power of two of
//                   its record, into hi (a multiple of 2^-10), the residue of the
//                   product rounded to fp16 and, in jobs of few tokens, what that
//                   leaves; the queries and the softmax weights into a multiple of
//                   2^-6 of the largest and two residues (all of an fp32 number to
//                   2^-28 of the largest).  The parts of a query or a weight
//                   are columns of the other operand (two of them side by side, in
//                   the same lane's accumulators).  hi times the first part sums
//                   exactly on the tensor cores, whose sums are truncated to 24
//                   bits (measured); the smaller products are added in fp32.
//   attend_combine  one CTA per (job, query): merges the units' partial results
//                   of the job, divides, applies D H (fp32 butterfly) and
//                   stores the row.
// Bound: instruction issue: 95 warp-instructions a token-head (d = 128, 4
// queries), 50 of them to decode and split its 128 pairs (table offset 2, lookup
// 1, norm code 3, products and split 3, packing 2 for each), issued in 60 % of the
// cycles at 16 warps per SM (128 registers).  Of a long call (128 heads of 32768
// tokens, 560 us) merging every unit is 7 % and the third parts of queries and
// weights 4 % (timing copies without them); handing a unit's sums over by
// mbarriers and merging them half a batch later instead of two CTA barriers takes
// 4 % off at d = 64 and spills at d = 128 (batch of 16 sequences 174 -> 192 us).
// Copies are bulk copies, one lane a segment (six cp.async loops took 2000 cycles
// of a batch's 12 000).
// 16 sequences of 1k to 32k tokens (8 KV heads, 4 queries each, 244 MB of records)
// take 174 us (1.4 TB/s), 229 us with fp32 products on the CUDA cores (114
// instructions, 10 - 12 warps, a warp walking 256 tokens alone); 8 heads of 4097
// tokens 16.5 and 59 us; 128 heads of 8192 tokens at d = 64 96 and 144 us.  The
// error of fp32 outputs against 64 bits is 0.56 to 1.0 times that of the fp32
// products over 105 shapes (1 to 8 queries, 1 to 32000 tokens, every norm storage,
// 3 draws each), 0.77 times on average.  Two fp16 parts of everything and sums over a CTA's units
// took 158, 20.5 and 84 us (484 us for the long call) and had 0.74 to 2.5 times that error.
// Every unit is merged and written by itself, in a fixed order, so a job's outputs
// do not depend on the other jobs of the call or on how the units fall to the CTAs.
// Codebooks (n, norm bits, norm mode) are runtime parameters: K and V may
// differ, and any codebook the encoder supports is accepted.
#include <algorithm>
#include <atomic>

#include <cuda_fp16.h>

#include "tac_attend.cuh"

namespace tac {

template <int V>
struct IC { static constexpr int value = V; };

constexpr int kAttWarps = 8;                  // warps per CTA
constexpr int kAttThreads = 32 * kAttWarps;
constexpr int kAttUnit = TAC_ATTEND_SPLIT;    // tokens of a unit: one batch for each warp
// Jobs of at most this many tokens split the decoded values in three parts.  With
// two a value keeps 2^-23 of its record's scale, which shows where few tokens share
// the softmax: 1.0 to 1.13 times the error of fp32 products up to 40 tokens (fp32
// norms), 0.66 to 1.0 times with three.  The third part costs 4 instructions a
// pair; from 257 tokens on two parts are at 0.79 to 0.95 times (eight shapes of 12000
// to 32768 tokens, 10 draws each; single draws from 0.5 to 1.5).
constexpr int kAttThree = kAttUnit;
constexpr float kLog2e = 1.4426950408889634f;
static_assert(kAttUnit == kAttWarps * kAttBatch, "a unit is one batch per warp");

// QT column tiles of four queries each (up to 4 QT queries).
template <int D, int QT>
struct Att {
  static constexpr int P = D / 2, NQ = 4 * QT;
  static constexpr int KP = P / 4, KS = KP / 2;   // K: pairs of a token a lane decodes (4 lanes a token), mma steps
  static constexpr int VP = P / 8;            // V: pairs of a token a lane decodes (8 lanes a token)
  // Shared memory: rotated queries as the fragments their mma steps load, their
  // scales, the warps' barriers, the warps' (max, sum, 1/unit) of a unit | K table
  // | V table | per warp: batch constants, weights, staged batch.  A warp's sums
  // of a unit are merged from the place of its staged V rows.
  static constexpr int Q_S = KS / 2 * QT * 2 * 512, Q_MB = Q_S + 32, Q_RED = Q_MB + 16 * kAttWarps;
  static constexpr int QB = Q_RED + 3 * kAttWarps * NQ * 4;
  static constexpr int W_KC = 0;              // float2 per token: (A, B) of K's norms
  static constexpr int W_VC = W_KC + kAttBatch * 8;
  static constexpr int W_KS = W_VC + kAttBatch * 8;   // float per token: 2^e of K's record
  static constexpr int W_VS = W_KS + kAttBatch * 4;
  static constexpr int W_W = W_VS + kAttBatch * 4;    // weights: [2][QT][8 + 4 columns][16 tokens] halves
  static constexpr int W_STG = W_W + 2 * QT * 12 * 32;
  static constexpr int MERGE = NQ * D * 4;            // a warp's sums
  static int smem(int stage, int tables) { return QB + tables + kAttWarps * (W_STG + stage); }
  static_assert(QB % 16 == 0 && W_STG % 16 == 0, "alignment");
};

// Decoded values are scaled by 2^kYExp of their record's power of two, which
// keeps their residues normal fp16 numbers.
constexpr int kYExp = 14;

// Bin centres (cos, sin)(2 pi k / n) of every supported n times 2^kYExp, rounded
// from fp64 by the host compiler.
namespace cx {
struct CentreTable { float2 v[kTabEntries]; };
constexpr CentreTable make_centre_table() {
  CentreTable t{};
  for (int idx = 0; idx < kTabEntries; ++idx) {
    const int n = tab_n_of(idx), k = idx - tab_offset_n(n);
    const CS cs = cos_sin_q8(8 * k, n);
    t.v[idx] = float2{(float)cs.c * (1 << kYExp), (float)cs.s * (1 << kYExp)};
  }
  return t;
}
}  // namespace cx
__device__ const cx::CentreTable g_centre = cx::make_centre_table();

// A shared-memory 16-byte load the compiler may not hoist or merge: keeps a
// loop-invariant operand in shared memory instead of in registers.
__device__ __forceinline__ uint4 lds_reload(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
  return v;
}

__device__ __forceinline__ uint32_t rotr(uint32_t x, int s) { return __funnelshift_r(x, x, s); }

__device__ __forceinline__ uint32_t h2_bits(__half2 h) { return *reinterpret_cast<const uint32_t*>(&h); }
__device__ __forceinline__ __half2 h2_of(uint32_t u) { return *reinterpret_cast<const __half2*>(&u); }

// d += a b: one m16n8k16 step, fp16 operands, fp32 accumulators.
__device__ __forceinline__ void mma_f16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// d = a b: the same from zero accumulators.
__device__ __forceinline__ void mma_f16_zero(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%10, %10, %10, %10};\n"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}

// 2^k, k clamped to [-126, 126], and 2^x for an integer-valued x (0 below 2^-126).
__device__ __forceinline__ float exp2i(int k) { return __uint_as_float((uint32_t)(127 + min(max(k, -126), 126)) << 23); }
__device__ __forceinline__ float exp2_whole(float x) { return x < -126.f ? 0.f : exp2i((int)fminf(x, 126.f)); }
// The exponent of a nonnegative fp32 number (-127 for zero and subnormals).
__device__ __forceinline__ int exp_of(float x) { return (int)((__float_as_uint(x) >> 23) & 0xFFu) - 127; }

// The split of (r, r) * cs, |r cs| < 2^(1 + kYExp): nh = -(hi of both), hi a
// multiple of 2^(kYExp - 10), lo the residue.
__device__ __forceinline__ void split_pair(float r, float2 cs, float2& nh, float2& lo) {
  constexpr float M = 12288.f * (1 << kYExp);  // 1.5 * 2^(13 + kYExp)
  const float2 rr = make_float2(r, r);
  const float2 q = __ffma2_rn(rr, cs, make_float2(M, M));
  nh = __ffma2_rn(q, make_float2(-1.f, -1.f), make_float2(M, M));
  lo = __ffma2_rn(rr, cs, nh);
}

// x = a + b + c, three fp16 numbers, to 2^-33 of 2^13 <= |x| < 2^15 at worst.
__device__ __forceinline__ void split_three(float x, float first, __half& a, __half& b, __half& c) {
  a = __float2half_rn(first);
  const float r = x - __half2float(a);
  b = __float2half_rn(r);
  c = __float2half_rn(r - __half2float(b));
}

// Batch constants of one token from its header: r^ 2^-e = A c + B for the norm
// code c (log mode: its log2), e the exponent of the larger of the two norms.
__device__ __forceinline__ void norm_consts(float2 h, float inv_l, bool lg, float2& ab, float& scale) {
  const bool spread = h.y > h.x;
  const int e = min(max(exp_of(spread ? h.y : h.x), kYExp - 126), 126);
  const float sc = exp2i(-e);
  scale = exp2i(e - kYExp);
  if (lg) {
    const float lo = lg2_approx(h.x);
    ab = make_float2(spread ? (lg2_approx(h.y) - lo) * inv_l : 0.f, lo - (float)e);
  } else {
    ab = make_float2(spread ? (h.y - h.x) * inv_l * sc : 0.f, h.x * sc);
  }
}

// A warp's staged batches arrive by bulk copies (cp.async.bulk) that signal an
// mbarrier of its own.  A wait gives up after 2^16 tries (each suspends the
// warp for a while) and returns false; the warp then copies nothing more, its
// results are NaN, and it waits (as long at most) for its copies before it leaves.
__device__ __forceinline__ uint32_t smem_addr(const void* ptr) { return (uint32_t)__cvta_generic_to_shared(ptr); }
__device__ __forceinline__ void mbar_init(uint32_t bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint32_t bar, int bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void* src, int bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  for (int i = 0; i < (1 << 16); ++i) {
    uint32_t done;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(done) : "r"(bar), "r"(parity) : "memory");
    if (done) return true;
  }
  return false;
}
// Shared memory written by ordinary stores is next written by bulk copies.
__device__ __forceinline__ void fence_async_proxy() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// The last, partial batch of a job: rows < 32 rows of row_bytes bytes, the rest
// of the 32 zero-filled.
static __device__ __noinline__ void copy_tail(const uint8_t* src, uint8_t* dst, int row_bytes, int rows, int lane) {
  const int full = kAttBatch * row_bytes, valid = rows * row_bytes;
  for (int c = lane * 16; c < full; c += 512) {
    const int n = min(max(valid - c, 0), 16);
    cp_async16(dst + c, n > 0 ? src + c : src, n);
  }
}

// In-place unnormalized Walsh-Hadamard transform of a row of d floats in
// shared memory (Sylvester order), by the lanes of a warp.
template <int D>
__device__ __forceinline__ void warp_fwht(float* row, int lane) {
#pragma unroll
  for (int lh = 0; (1 << lh) < D; ++lh) {
    __syncwarp();
#pragma unroll
    for (int e = lane; e < D / 2; e += 32) {
      const int i = ((e >> lh) << (lh + 1)) + (e & ((1 << lh) - 1));
      const float a = row[i], b = row[i + (1 << lh)];
      row[i] = a + b;
      row[i + (1 << lh)] = a - b;
    }
  }
  __syncwarp();
}

template <int D, int QT>
__global__ void __launch_bounds__(kAttThreads, QT == 1 ? 2 : 1)
    attend_partial(const __grid_constant__ AttParams p, float* ws) {
  using C = Att<D, QT>;
  constexpr int P = C::P, NQ = C::NQ, KP = C::KP, KS = C::KS, VP = C::VP;
  extern __shared__ __align__(128) uint8_t smem[];
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // warp-uniform for the compiler too
  const int g = lane >> 2, t = lane & 3;           // the fragments' row group and column pair
  uint32_t* const qfrag = reinterpret_cast<uint32_t*>(smem);                 // [KS / 2][QT][2][lane] uint4
  float* const qscale = reinterpret_cast<float*>(smem + C::Q_S);             // 2^e of each query
  float2* const red = reinterpret_cast<float2*>(smem + C::Q_RED);            // [warp][query]: max, 1/unit of a unit's sums
  float* const redl = reinterpret_cast<float*>(red + kAttWarps * NQ);        // and the sum
  float2* const tk = reinterpret_cast<float2*>(smem + C::QB);
  uint8_t* const wbase = smem + C::QB + p.tab_k + p.tab_v;
  float2* const tv = reinterpret_cast<float2*>(smem + C::QB + p.tab_k);
  uint8_t* const pw = wbase + warp * (C::W_STG + p.stage);
  float2* const kc = reinterpret_cast<float2*>(pw + C::W_KC);
  float2* const vc = reinterpret_cast<float2*>(pw + C::W_VC);
  float* const ksc = reinterpret_cast<float*>(pw + C::W_KS);
  float* const vsc = reinterpret_cast<float*>(pw + C::W_VS);
  uint8_t* const stk = pw + C::W_STG;

  // the combine kernel may be launched from now on (it waits for this grid's end)
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  // the CTA's units
  const int per = p.nunits / p.nctas, extra = p.nunits % p.nctas, cta = blockIdx.x;
  int u = cta * per + min(cta, extra);
  const int u_end = u + per + (cta < extra ? 1 : 0);
  int tab_nk = 0, tab_nv = 0;                      // codebooks the tables hold

  int jb = p.first_job[cta];
  const uint32_t bar_k = smem_addr(smem + C::Q_MB) + 16 * warp, bar_v = bar_k + 8;
  uint32_t phase_k = 0, phase_v = 0;               // parity of the next completion
  bool dead = false;                               // a wait ran out
  if (lane == 0) {
    mbar_init(bar_k);
    mbar_init(bar_v);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  for (; u < u_end; ++jb) {                        // a segment: the CTA's units of one job
    const AttJob& J = p.job[jb];
    const int nunits = (int)((J.tokens + kAttUnit - 1) / kAttUnit);
    const int u_stop = min(u_end, J.unit0 + nunits);
    const int nq = J.nq;
    const int ak = P * J.wk / 8, nbk = P * J.bk / 8, av = P * J.wv / 8, nbv = P * J.bv / 8;
    const int hkb = J.mk != TAC_NORM_FP32 ? 8 : 0, hvb = J.mv != TAC_NORM_FP32 ? 8 : 0;
    uint8_t* const st_kn = stk + kAttBatch * ak;
    uint8_t* const st_kh = st_kn + kAttBatch * nbk;
    uint8_t* const st_va = st_kh + kAttBatch * hkb;
    uint8_t* const st_vn = st_va + kAttBatch * av;
    uint8_t* const st_vh = st_vn + kAttBatch * nbv;
    int64_t row0 = (int64_t)(u - J.unit0) * kAttUnit + warp * kAttBatch;
    const int64_t seg_rows = min(J.tokens, (int64_t)(u_stop - J.unit0) * kAttUnit);   // the segment's end
    int unit = u - J.unit0;                        // within the job
    u = u_stop;

    // ---- staging: lane s of 6 copies the 32 rows of segment s (K angle | norm |
    // header, V angle | norm | header) of a whole batch; the last, partial batch
    // of the job comes by cp.async ----
    const bool is_v = lane >= 3;
    const int sg = is_v ? lane - 3 : lane;
    const int c_row = lane >= 6 ? 0 : sg == 0 ? (is_v ? av : ak) : sg == 1 ? (is_v ? nbv : nbk) : (is_v ? hvb : hkb);
    const uint8_t* c_src = sg == 0 ? (is_v ? J.vc : J.kc) : sg == 1 ? (is_v ? J.vn : J.kn) : (is_v ? J.vh : J.kh);
    c_src += row0 * c_row;                         // advances with the K (V) batches
    const uint32_t c_dst =
        smem_addr(sg == 0 ? (is_v ? st_va : stk) : sg == 1 ? (is_v ? st_vn : st_kn) : (is_v ? st_vh : st_kh));
    auto issue = [&](bool v, int64_t row, uint32_t bar, int bytes) {
      const bool mine = (is_v == v) && lane < 6 && c_row > 0;
      if (dead) return;
      if (row + kAttBatch <= seg_rows) {
        if (lane == 0) mbar_expect(bar, bytes);
        __syncwarp();
        if (mine) bulk_copy(c_dst, c_src, kAttBatch * c_row, bar);
      } else if (row < seg_rows) {
        const int rows = (int)(seg_rows - row);
        for (int x = 0; x < 3; ++x) {
          const int from = (v ? 3 : 0) + x, rb = __shfl_sync(0xffffffffu, c_row, from);
          const uint8_t* src = reinterpret_cast<const uint8_t*>(
              __shfl_sync(0xffffffffu, (unsigned long long)(uintptr_t)c_src, from));
          uint8_t* dst = x == 0 ? (v ? st_va : stk) : x == 1 ? (v ? st_vn : st_kn) : (v ? st_vh : st_kh);
          copy_tail(src, dst, rb, rows, lane);
        }
        cp_async_commit();
      }
      if (mine) c_src += kAttUnit * c_row;
    };
    const int bytes_k = kAttBatch * (ak + nbk + hkb), bytes_v = kAttBatch * (av + nbv + hvb);
    // waits for the batch of rows [row, row + 32)
    auto landed = [&](int64_t row, uint32_t bar, uint32_t& phase) {
      if (row + kAttBatch <= seg_rows) {
        if (!dead) dead = !__all_sync(0xffffffffu, mbar_wait(bar, phase));
        if (!dead) phase ^= 1u;
      } else {
        cp_async_wait<0>();
      }
      __syncwarp();
    };
    fence_async_proxy();
    __syncthreads();                               // the previous segment is done with the queries and the tables
    issue(false, row0, bar_k, bytes_k);
    issue(true, row0, bar_v, bytes_v);

    // ---- bin-centre tables (cos, sin)(2 pi k / n), 2^lgr copies: entry k copy c
    // at k 2^lgr + c; entries n..2^W-1 repeat entry n-1 (codes >= n clamp) ----
    const int lgrk = J.lgrk, lgrv = J.lgrv;
    if (tab_nk != J.nk || tab_nv != J.nv) {
      const int ek = 1 << J.wk, ev = 1 << J.wv;
      for (int e = tid; e < (ek << lgrk) + (ev << lgrv); e += kAttThreads) {
        const bool v = e >= ek << lgrk;
        const int at = v ? e - (ek << lgrk) : e, n = v ? J.nv : J.nk;
        (v ? tv : tk)[at] = g_centre.v[tab_offset_n(n) + min(at >> (v ? lgrv : lgrk), n - 1)];
      }
      tab_nk = J.nk;
      tab_nv = J.nv;
    }
    // ---- rotated queries q' = H D_K q * scale * log2(e), one warp a query,
    // scaled by 2^-e into [-2^14, 2^14) and split in three: a multiple of 2^8 (six
    // bits), then two fp16 residues.  Columns 2 a and 2 a + 1 of a fragment are the
    // first two parts of query a; the third (negated) is column 2 a of a fragment
    // of its own.  The word of a slot (the halves of its pair) lands where its mma
    // step loads it: the run of KP slots of lane t, step by step.  Step ks takes
    // two slots of every lane's run: neighbours, or (4-bit norms, whose codes are
    // unpacked four apart) slots four apart ----
    const bool k4 = J.ck <= 1;
    if (warp < NQ) {
      float y[D / 32];                             // elements lane + 32 k
      const int64_t off = (int64_t)warp * J.q_stride + lane;
#pragma unroll
      for (int k = 0; k < D / 32; ++k) {
        float x = 0.f;
        if (warp < nq)
          x = p.q_bf16 ? __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(J.q)[off + 32 * k])
                       : reinterpret_cast<const float*>(J.q)[off + 32 * k];
        y[k] = (J.sk[k] >> lane) & 1u ? -x : x;
      }
#pragma unroll
      for (int h = 1; h < D / 32; h <<= 1)
#pragma unroll
        for (int k = 0; k < D / 32; ++k)
          if (!(k & h)) {
            const float a = y[k], b = y[k + h];
            y[k] = a + b;
            y[k + h] = a - b;
          }
#pragma unroll
      for (int h = 1; h < 32; h <<= 1) {
        const float sg_ = lane & h ? -1.f : 1.f;
#pragma unroll
        for (int k = 0; k < D / 32; ++k)
          y[k] = __fmaf_rn(sg_, y[k], __shfl_xor_sync(0xffffffffu, y[k], h));
      }
      const float qs = J.scale * kLog2e * rsqrtf((float)D);
      float mx = 0.f;
#pragma unroll
      for (int k = 0; k < D / 32; ++k) {
        y[k] *= qs;
        mx = fmaxf(mx, fabsf(y[k]));
      }
#pragma unroll
      for (int o = 16; o >= 1; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      const int e = min(max(exp_of(mx) - 13, -126), 126);
      const float sc = exp2i(-e);
#pragma unroll
      for (int k = 0; k < D / 32; ++k) {
        const float a = y[k] * sc, b = __shfl_down_sync(0xffffffffu, a, 1);
        if (!(lane & 1)) {                         // pair 16 k + lane / 2
          constexpr float M = 3221225472.f;        // 1.5 * 2^31: sums round to multiples of 2^8
          __half a1, a2, a3, b1, b2, b3;
          split_three(a, __fsub_rn(__fadd_rn(a, M), M), a1, a2, a3);
          split_three(b, __fsub_rn(__fadd_rn(b, M), M), b1, b2, b3);
          const int i = pair_slot<D>(16 * k + lane / 2), r = i % KP;
          const int at = k4 ? (r & ~7) + 2 * (r & 3) + ((r >> 2) & 1) : r;
          uint32_t* const w = qfrag + (((at >> 2) * QT + (warp >> 2)) * 64 + 8 * (warp & 3) + i / KP) * 4 + (at & 3);
          w[0] = h2_bits(__halves2half2(a1, b1));
          w[16] = h2_bits(__halves2half2(a2, b2));
          w[128] = h2_bits(__halves2half2(__hneg(a3), __hneg(b3)));
          w[144] = 0u;
        }
      }
      if (lane == 0) qscale[warp] = exp2i(e);
    }
    __syncthreads();

    // ---- lane constants ----
    // K: lane (g, t) decodes slots KP t .. KP t + KP - 1 of tokens g and g + 8 of
    // each 16; codes 4 q .. 4 q + 3 start at bit wk (KP t + 4 q) of the row.  A
    // code becomes the byte offset of its table entry (copy lane % 2^lgr) by one
    // rotate and one mask.
    const int wk = J.wk, Tk = 3 + lgrk;
    const uint32_t kC = (uint32_t)(lane & ((1 << lgrk) - 1)) << 3;
    const uint32_t kM = ((1u << wk) - 1u) << Tk;
    int kra[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) kra[j] = (wk * j - Tk) & 31;
    const uint8_t* const tkb = reinterpret_cast<const uint8_t*>(tk);
    int koff[KP / 4], ksh[KP / 4];                 // word and shift of codes 4 q .. 4 q + 3
#pragma unroll
    for (int q = 0; q < KP / 4; ++q) {
      const int bit = wk * (KP * t + 4 * q);
      koff[q] = (bit >> 5) * 4;
      ksh[q] = bit & 31;
    }
    // V: lane (g, t) decodes slots VP g .. VP g + VP - 1 of tokens 4 t .. 4 t + 3 of each 16.
    const int wv = J.wv, Tv = 3 + lgrv;
    const uint32_t vC = (uint32_t)(lane & ((1 << lgrv) - 1)) << 3;
    const uint32_t vM = ((1u << wv) - 1u) << Tv;
    int vra[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) vra[j] = (wv * j - Tv) & 31;
    const uint8_t* const tvb = reinterpret_cast<const uint8_t*>(tv);
    int voff[VP / 4], vsh[VP / 4];
#pragma unroll
    for (int q = 0; q < VP / 4; ++q) {
      const int bit = wv * (VP * g + 4 * q);
      voff[q] = (bit >> 5) * 4;
      vsh[q] = bit & 31;
    }
    const uint32_t qlane = smem_addr(qfrag) + 16 * lane;
    const float kinv = J.inv_lk, vinv = J.inv_lv;
    const bool klog = J.mk == TAC_NORM_LOG, vlog = J.mv == TAC_NORM_LOG;
    // The lane's queries: 4 x + t.
    float qsc[QT];
#pragma unroll
    for (int x = 0; x < QT; ++x) qsc[x] = qscale[4 * x + t];

    // fp32 norms: no header; the largest norm of each token of the batch sets its scale.
    auto fp32_consts = [&](const uint8_t* norms, int row_bytes, float2* ab, float* scale) {
      for (int i = 0; i < kAttBatch / 4; ++i) {
        const int tok = 4 * i + (lane >> 3);
        const float* nr = reinterpret_cast<const float*>(norms + tok * row_bytes) + VP * (lane & 7);
        float mx = 0.f;
#pragma unroll
        for (int k = 0; k < VP; k += 4) {
          const float4 v = *reinterpret_cast<const float4*>(nr + k);
          mx = fmaxf(fmaxf(fmaxf(mx, fabsf(v.x)), fmaxf(fabsf(v.y), fabsf(v.z))), fabsf(v.w));
        }
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        const int e = min(max(exp_of(mx), kYExp - 126), 126);
        if ((lane & 7) == 0) {
          ab[tok] = make_float2(exp2i(-e), 0.f);
          scale[tok] = exp2i(e - kYExp);
        }
      }
    };

    // Scores of the staged batch.  Rows of the fragments are tokens, columns the
    // parts of the queries, the steps run over the slots.  hi is a multiple of 2^-10
    // below 2 and the queries' first part of 2^8 up to 2^14, so that their products
    // and all sums of them are whole multiples of 2^-2 below 2^22 (64 pairs, each
    // at most 2 sqrt(2) 2^14): exact, although the tensor cores' sums are truncated
    // to 24 bits.  The other parts are 2^-7 of it or less and are added last, in fp32.
    // sv[x]: tokens 16 (i / 2) + 8 (i & 1) + g, query 4 x + t.
    auto scores = [&](float (&sv)[QT][4], auto kc_, auto three_) {
      constexpr int KC = decltype(kc_)::value;
      constexpr bool THREE = decltype(three_)::value != 0;
      constexpr bool F32 = KC == 4, LOG = KC == 1 || KC == 3;
      constexpr int KB = KC <= 1 ? 4 : 8, KW = F32 ? 1 : KP * KB / 32;
#pragma unroll
      for (int x2 = 0; x2 < QT; ++x2) sv[x2][2] = sv[x2][3] = 0.f;
#pragma unroll 1
      for (int mt = 0; mt < 2; ++mt) {
        uint32_t x[2][KP / 4], nw[2][KW];
        float2 ab[2];
        const float* nf[2] = {nullptr, nullptr};
#pragma unroll
        for (int rr = 0; rr < 2; ++rr) {
          const int row = 16 * mt + 8 * rr + g;
          const uint8_t* arow = stk + row * ak;
#pragma unroll
          for (int q = 0; q < KP / 4; ++q) {
            const uint32_t* aw = reinterpret_cast<const uint32_t*>(arow + koff[q]);
            x[rr][q] = __funnelshift_r(aw[0], aw[1], ksh[q]);
          }
          ab[rr] = kc[row];
          const uint8_t* nr = st_kn + row * nbk;
          if constexpr (F32) {
            nf[rr] = reinterpret_cast<const float*>(nr) + KP * t;
          } else if constexpr (KW == 4) {
            const uint4 v = *reinterpret_cast<const uint4*>(nr + 16 * t);
            nw[rr][0] = v.x; nw[rr][1] = v.y; nw[rr][2] = v.z; nw[rr][3] = v.w;
          } else if constexpr (KW == 2) {
            const uint2 v = *reinterpret_cast<const uint2*>(nr + 8 * t);
            nw[rr][0] = v.x; nw[rr][1] = v.y;
          } else {
            nw[rr][0] = *reinterpret_cast<const uint32_t*>(nr + 4 * t);
          }
        }
        float ch[QT][2][4], cl[QT][4];             // hi times parts 1 | 2 (two chains), the rest
#pragma unroll
        for (int x2 = 0; x2 < QT; ++x2)
#pragma unroll
          for (int i = 0; i < 4; ++i) ch[x2][0][i] = ch[x2][1][i] = cl[x2][i] = 0.f;
        uint4 bq[QT][2];
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) {
          if ((ks & 1) == 0) {
#pragma unroll
            for (int x2 = 0; x2 < QT; ++x2)
#pragma unroll
              for (int f = 0; f < 2; ++f) bq[x2][f] = lds_reload(qlane + ((ks / 2 * QT + x2) * 2 + f) * 512);
          }
          uint32_t ah[4], al[4], al2[4];
#pragma unroll
          for (int rr = 0; rr < 2; ++rr) {
            float rv[2];
            if constexpr (F32) {
              const float2 v = *reinterpret_cast<const float2*>(nf[rr] + 2 * ks);
              rv[0] = v.x * ab[rr].x;
              rv[1] = v.y * ab[rr].x;
            } else {
              uint32_t hb;
              if constexpr (KB == 8) hb = __byte_perm(nw[rr][ks >> 1], 0x64646464u, (ks & 1) ? 0x4342 : 0x4140);
              else hb = ((nw[rr][ks >> 2] >> (4 * (ks & 3))) & 0x000F000Fu) | 0x64006400u;
              const float2 cc = __half22float2(__hsub2(h2_of(hb), h2_of(0x64006400u)));
              rv[0] = __fmaf_rn(cc.x, ab[rr].x, ab[rr].y);
              rv[1] = __fmaf_rn(cc.y, ab[rr].x, ab[rr].y);
              if constexpr (LOG) { rv[0] = ex2_ftz(rv[0]); rv[1] = ex2_ftz(rv[1]); }
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const int i = (KB == 4 && !F32) ? 8 * (ks >> 2) + (ks & 3) + 4 * h : 2 * ks + h;
              const uint32_t o = (rotr(x[rr][i >> 2], kra[i & 3]) & kM) | kC;
              float2 nh, lo;
              split_pair(rv[h], *reinterpret_cast<const float2*>(tkb + o), nh, lo);
              ah[2 * h + rr] = h2_bits(__floats2half2_rn(nh.x, nh.y));
              const __half2 hl = __floats2half2_rn(lo.x, lo.y);
              al[2 * h + rr] = h2_bits(hl);
              if constexpr (THREE) {
                const float2 fl = __half22float2(hl);
                al2[2 * h + rr] = h2_bits(__floats2half2_rn(lo.x - fl.x, lo.y - fl.y));
              }
            }
          }
#pragma unroll
          for (int x2 = 0; x2 < QT; ++x2) {
            const uint4 q12 = bq[x2][0], q3 = bq[x2][1];
            const uint32_t b0 = ks & 1 ? q12.z : q12.x, b1 = ks & 1 ? q12.w : q12.y;
            mma_f16(ch[x2][ks & 1], ah, b0, b1);
            mma_f16(cl[x2], al, b0, b1);
            if constexpr (THREE) mma_f16(cl[x2], al2, b0, b1);
            mma_f16(cl[x2], ah, ks & 1 ? q3.z : q3.x, ks & 1 ? q3.w : q3.y);
          }
        }
#pragma unroll
        for (int x2 = 0; x2 < QT; ++x2)
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            sv[x2][i] = sv[x2][2 + i];
            const float rest = (cl[x2][2 * i] + cl[x2][2 * i + 1]) - (ch[x2][0][2 * i + 1] + ch[x2][1][2 * i + 1]);
            sv[x2][2 + i] = rest - (ch[x2][0][2 * i] + ch[x2][1][2 * i]);
          }
      }
    };

    // Values: acc += sum_t w_t y^V_t.  Rows of the fragments are the (cos, sin) of
    // slot VP g + j, columns the parts of the queries' weights (as the queries'
    // parts above), the steps run over the tokens.  THREE: a value's residue is
    // split once more (see kAttThree).
    float acc[QT][VP][4];
    auto values = [&](auto vc_, auto three_) {
      constexpr int VC = decltype(vc_)::value;
      constexpr bool THREE = decltype(three_)::value != 0;
      constexpr bool F32 = VC == 4, LOG = VC == 1 || VC == 3;
      constexpr int VB = VC <= 1 ? 4 : 8;
      constexpr bool N16 = VB == 4 && VP == 4 && !F32;   // a lane's norms of a token in 16 bits
      constexpr int VW = F32 ? 1 : (VP * VB + 31) / 32;
#pragma unroll 1
      for (int kk = 0; kk < 2; ++kk) {
        uint32_t x[4][VP / 4], nw[4][VW];
        float2 ab[4];
        const float* nf[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int tok = 16 * kk + 4 * t + i;
          const uint8_t* arow = st_va + tok * av;
#pragma unroll
          for (int q = 0; q < VP / 4; ++q) {
            const uint32_t* aw = reinterpret_cast<const uint32_t*>(arow + voff[q]);
            x[i][q] = __funnelshift_r(aw[0], aw[1], vsh[q]);
          }
          ab[i] = vc[tok];
          const uint8_t* nr = st_vn + tok * nbv;
          nf[i] = reinterpret_cast<const float*>(nr) + VP * g;
          if constexpr (F32) {
          } else if constexpr (VW == 2) {
            const uint2 v = *reinterpret_cast<const uint2*>(nr + 8 * g);
            nw[i][0] = v.x; nw[i][1] = v.y;
          } else if constexpr (N16) {
            nw[i][0] = *reinterpret_cast<const uint16_t*>(nr + 2 * g);
          } else {
            nw[i][0] = *reinterpret_cast<const uint32_t*>(nr + 4 * g);
          }
        }
        if constexpr (N16) {                       // the norms of two tokens in one word
          nw[0][0] |= nw[1][0] << 16;
          nw[2][0] |= nw[3][0] << 16;
        }
        uint32_t b[QT][2], nb[QT][2], nb3[QT][2];
#pragma unroll
        for (int x2 = 0; x2 < QT; ++x2) {
          const uint8_t* wt = pw + C::W_W + (kk * QT + x2) * 384 + 8 * t;
          const uint2 v = *reinterpret_cast<const uint2*>(wt + g * 32);
          const uint2 v3 = *reinterpret_cast<const uint2*>(wt + 256 + (g >> 1) * 32);
          b[x2][0] = v.x; b[x2][1] = v.y;
          nb[x2][0] = v.x ^ 0x80008000u; nb[x2][1] = v.y ^ 0x80008000u;
          nb3[x2][0] = g & 1 ? 0u : v3.x; nb3[x2][1] = g & 1 ? 0u : v3.y;
        }
#pragma unroll
        for (int jj = 0; jj < VP / 2; ++jj) {      // two slots at a time
          const int ja = (VB == 4 && !F32 && !N16) ? 8 * (jj >> 2) + (jj & 3) : 2 * jj;
          const int js[2] = {ja, (VB == 4 && !F32 && !N16) ? ja + 4 : ja + 1};
          float rv[4][2];
          if constexpr (N16) {
#pragma unroll
            for (int i = 0; i < 4; i += 2)
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                const uint32_t hb = ((nw[i][0] >> (4 * js[h])) & 0x000F000Fu) | 0x64006400u;
                const float2 cc = __half22float2(__hsub2(h2_of(hb), h2_of(0x64006400u)));
                rv[i][h] = __fmaf_rn(cc.x, ab[i].x, ab[i].y);
                rv[i + 1][h] = __fmaf_rn(cc.y, ab[i + 1].x, ab[i + 1].y);
              }
          } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              if constexpr (F32) {
                const float2 v = *reinterpret_cast<const float2*>(nf[i] + 2 * jj);
                rv[i][0] = v.x * ab[i].x;
                rv[i][1] = v.y * ab[i].x;
              } else {
                uint32_t hb;
                if constexpr (VB == 8) hb = __byte_perm(nw[i][(jj >> 1) % VW], 0x64646464u, (jj & 1) ? 0x4342 : 0x4140);
                else hb = ((nw[i][0] >> (4 * (jj & 3))) & 0x000F000Fu) | 0x64006400u;
                const float2 cc = __half22float2(__hsub2(h2_of(hb), h2_of(0x64006400u)));
                rv[i][0] = __fmaf_rn(cc.x, ab[i].x, ab[i].y);
                rv[i][1] = __fmaf_rn(cc.y, ab[i].x, ab[i].y);
              }
            }
          }
          if constexpr (LOG) {
#pragma unroll
            for (int i = 0; i < 4; ++i) { rv[i][0] = ex2_ftz(rv[i][0]); rv[i][1] = ex2_ftz(rv[i][1]); }
          }
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int j = js[h];
            uint32_t ah[4], al[4], al2[4];
#pragma unroll
            for (int i = 0; i < 4; i += 2) {
              float2 n0, l0, n1, l1;
              const uint32_t o0 = (rotr(x[i][j >> 2], vra[j & 3]) & vM) | vC;
              const uint32_t o1 = (rotr(x[i + 1][j >> 2], vra[j & 3]) & vM) | vC;
              split_pair(rv[i][h], *reinterpret_cast<const float2*>(tvb + o0), n0, l0);
              split_pair(rv[i + 1][h], *reinterpret_cast<const float2*>(tvb + o1), n1, l1);
              ah[i] = h2_bits(__floats2half2_rn(n0.x, n1.x));
              ah[i + 1] = h2_bits(__floats2half2_rn(n0.y, n1.y));
              const __half2 lx = __floats2half2_rn(l0.x, l1.x), ly = __floats2half2_rn(l0.y, l1.y);
              al[i] = h2_bits(lx);
              al[i + 1] = h2_bits(ly);
              if constexpr (THREE) {
                const float2 fx = __half22float2(lx), fy = __half22float2(ly);
                al2[i] = h2_bits(__floats2half2_rn(l0.x - fx.x, l1.x - fx.y));
                al2[i + 1] = h2_bits(__floats2half2_rn(l0.y - fy.x, l1.y - fy.y));
              }
            }
#pragma unroll
            for (int x2 = 0; x2 < QT; ++x2) {
              float c[4];
              mma_f16_zero(c, al, b[x2][0], b[x2][1]);
              if constexpr (THREE) mma_f16(c, al2, b[x2][0], b[x2][1]);
              mma_f16(c, ah, nb3[x2][0], nb3[x2][1]);
              if constexpr (THREE) {               // hi times part 1 (exact) apart from the rest
                float ch[4];
                mma_f16_zero(ch, ah, nb[x2][0], nb[x2][1]);
                c[1] = (c[1] + ch[1]) + c[0];
                c[3] = (c[3] + ch[3]) + c[2];
                c[0] = ch[0];
                c[2] = ch[2];
              } else {
                mma_f16(c, ah, nb[x2][0], nb[x2][1]);
              }
              float2* a2 = reinterpret_cast<float2*>(acc[x2][j]);
              a2[0] = add2(a2[0], make_float2(c[0], c[1]));
              a2[1] = add2(a2[1], make_float2(c[2], c[3]));
            }
          }
        }
      }
    };

    const bool three = J.tokens <= kAttThree;
    for (; ; ++unit, row0 += kAttUnit) {             // a unit: one batch for each warp
      float m_[QT], l_[QT], iu[QT];                  // its max (whole), sum of 2^(s - m), and 1 / the sums' unit
#pragma unroll
      for (int x = 0; x < QT; ++x) {
        m_[x] = -INFINITY;
        l_[x] = 0.f;
        iu[x] = 1.f;
#pragma unroll
        for (int j = 0; j < VP; ++j)
#pragma unroll
          for (int i = 0; i < 4; ++i) acc[x][j][i] = 0.f;
      }
      if (row0 < seg_rows) {
        const int valid = (int)min((int64_t)kAttBatch, J.tokens - row0);
        landed(row0, bar_k, phase_k);                // this batch's K rows
        if (hkb) norm_consts(reinterpret_cast<const float2*>(st_kh)[lane], kinv, klog, kc[lane], ksc[lane]);
        else fp32_consts(st_kn, nbk, kc, ksc);
        __syncwarp();
        float sv[QT][4];
        switch (J.ck + (three ? 8 : 0)) {
          case 0: scores(sv, IC<0>{}, IC<0>{}); break;
          case 1: scores(sv, IC<1>{}, IC<0>{}); break;
          case 2: scores(sv, IC<2>{}, IC<0>{}); break;
          case 3: scores(sv, IC<3>{}, IC<0>{}); break;
          case 4: scores(sv, IC<4>{}, IC<0>{}); break;
          case 8: scores(sv, IC<0>{}, IC<1>{}); break;
          case 9: scores(sv, IC<1>{}, IC<1>{}); break;
          case 10: scores(sv, IC<2>{}, IC<1>{}); break;
          case 11: scores(sv, IC<3>{}, IC<1>{}); break;
          default: scores(sv, IC<4>{}, IC<1>{}); break;
        }
        auto token = [&](int i) { return 16 * (i >> 1) + 8 * (i & 1) + g; };
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int tok = token(i);
          const float ks = ksc[tok];
#pragma unroll
          for (int x = 0; x < QT; ++x) sv[x][i] = tok < valid ? sv[x][i] * (qsc[x] * ks) : -INFINITY;
        }
        __syncwarp();                                // every lane is done with the K rows
        issue(false, row0 + kAttUnit, bar_k, bytes_k);
        landed(row0, bar_v, phase_v);                // this batch's V rows
        if (hvb) norm_consts(reinterpret_cast<const float2*>(st_vh)[lane], vinv, vlog, vc[lane], vsc[lane]);
        else fp32_consts(st_vn, nbv, vc, vsc);
        __syncwarp();
        // ---- softmax (base 2) of the batch against the whole number above its
        // largest score; weights 2^(s - m) 2^e scaled by the power of two that
        // brings the largest to [2^14, 2^15), in three fp16 parts ----
#pragma unroll
        for (int x = 0; x < QT; ++x) {
          float mx = fmaxf(fmaxf(sv[x][0], sv[x][1]), fmaxf(sv[x][2], sv[x][3]));
#pragma unroll
          for (int o = 4; o < 32; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
          m_[x] = J.tokens <= kAttBatch ? mx : ceilf(mx);
          float w[4], wm = 0.f;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float pr = ex2_approx(sv[x][i] - m_[x]);
            l_[x] += pr;
            w[i] = pr * vsc[token(i)];
            wm = fmaxf(wm, w[i]);
          }
#pragma unroll
          for (int o = 4; o < 32; o <<= 1) wm = fmaxf(wm, __shfl_xor_sync(0xffffffffu, wm, o));
          const int k = min(max(14 - exp_of(wm), -126), 126);
          const float unit_ = exp2i(k);
          iu[x] = exp2i(-k);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            __half w1, w2, w3;
            const float ws_ = w[i] * unit_;
            constexpr float M = 6442450944.f;      // 1.5 * 2^32: sums round to multiples of 2^9
            split_three(ws_, __fsub_rn(__fadd_rn(ws_, M), M), w1, w2, w3);
            const int tok = token(i);
            __half* const wt = reinterpret_cast<__half*>(pw + C::W_W + ((tok >> 4) * QT + x) * 384) + (tok & 15);
            wt[32 * t] = w1;
            wt[32 * t + 16] = w2;
            wt[128 + 16 * t] = __hneg(w3);
          }
        }
        __syncwarp();
        switch (J.cv + (three ? 8 : 0)) {
          case 0: values(IC<0>{}, IC<0>{}); break;
          case 1: values(IC<1>{}, IC<0>{}); break;
          case 2: values(IC<2>{}, IC<0>{}); break;
          case 3: values(IC<3>{}, IC<0>{}); break;
          case 4: values(IC<4>{}, IC<0>{}); break;
          case 8: values(IC<0>{}, IC<1>{}); break;
          case 9: values(IC<1>{}, IC<1>{}); break;
          case 10: values(IC<2>{}, IC<1>{}); break;
          case 11: values(IC<3>{}, IC<1>{}); break;
          default: values(IC<4>{}, IC<1>{}); break;
        }
#pragma unroll
        for (int x = 0; x < QT; ++x)
#pragma unroll
          for (int o = 4; o < 32; o <<= 1) l_[x] += __shfl_xor_sync(0xffffffffu, l_[x], o);
      }
      __syncwarp();                                  // every lane is done with the V rows and the weights
      // ---- merge the warps' sums of the unit in a fixed order: its record depends on
      // nothing but the job's own rows and queries ----
      float2* const mrg = reinterpret_cast<float2*>(st_va);   // [x][j][lane], in the place of the V rows
#pragma unroll
      for (int x = 0; x < QT; ++x)
#pragma unroll
        for (int j = 0; j < VP; ++j)
          mrg[(x * VP + j) * 32 + lane] = make_float2(acc[x][j][0] + acc[x][j][1], acc[x][j][2] + acc[x][j][3]);
      if (g == 0) {
#pragma unroll
        for (int x = 0; x < QT; ++x) {
          const int at = warp * NQ + 4 * x + t;
          red[at] = make_float2(m_[x], iu[x]);
          redl[at] = dead ? __int_as_float(0x7FC00000) : l_[x];
        }
      }
      __syncthreads();
      float* const rec = ws + J.ws + (int64_t)unit * nq * att_rec_floats(D);
      const uint8_t* const m0 = reinterpret_cast<const uint8_t*>(mrg) - (size_t)warp * (C::W_STG + p.stage);
#pragma unroll
      for (int e0 = 0; e0 < QT * VP * 32; e0 += kAttThreads) {
        const int e = e0 + tid, x = e / (VP * 32), j = (e >> 5) % VP, a = 4 * x + t;
        if (e < QT * VP * 32 && a < nq) {
          float2 mw[kAttWarps];
          float M = -INFINITY;
#pragma unroll
          for (int w = 0; w < kAttWarps; ++w) {
            mw[w] = red[w * NQ + a];
            M = fmaxf(M, mw[w].x);
          }
          float2 s2 = make_float2(0.f, 0.f);
#pragma unroll
          for (int w = 0; w < kAttWarps; ++w) {
            mw[w].x = ex2_ftz(mw[w].x - M);          // of a whole number (or -infinity): exact
            const float f = mw[w].x * mw[w].y;
            const float2 v = reinterpret_cast<const float2*>(m0 + (size_t)w * (C::W_STG + p.stage))[e];
            s2 = __ffma2_rn(v, make_float2(f, f), s2);
          }
          float* const ra = rec + a * att_rec_floats(D);
          *reinterpret_cast<float2*>(ra + 2 + 2 * slot_pair<D>(VP * g + j)) = s2;
          if (j == 0 && g == 0) {
            float l = 0.f;
#pragma unroll
            for (int w = 0; w < kAttWarps; ++w) l = __fmaf_rn(redl[w * NQ + a], mw[w].x, l);
            *reinterpret_cast<float2*>(ra) = make_float2(M, l);
          }
        }
      }
      fence_async_proxy();
      __syncthreads();                               // the merge is done with the warps' memory
      if (unit + 1 == u_stop - J.unit0) break;
      issue(true, row0 + kAttUnit, bar_v, bytes_v);
    }
  }
  if (dead) {                                        // the copies issued and not waited for
    (void)mbar_wait(bar_k, phase_k);
    (void)mbar_wait(bar_v, phase_v);
  }
}

// One CTA of 4 warps per (job, query): warp w merges units w, w + 4, ...
// against the row's overall max, the warps' sums are added in shared memory,
// and warp 0 normalizes, applies D H (fp32 butterfly) and stores the row.
template <int D, typename TO>
__global__ void __launch_bounds__(128) attend_combine(const __grid_constant__ AttParams p, const float* ws) {
  constexpr int ESZ = (int)sizeof(TO);
  constexpr int E = D / 32;
  __shared__ float part[4][D];
  __shared__ float red[4][2];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const AttJob& J = p.job[blockIdx.y];
  const int a = blockIdx.x;
  if (a >= J.nq) return;
  const int nsp = (int)((J.tokens + kAttUnit - 1) / kAttUnit);
  const float* recs = ws + J.ws + (int64_t)a * att_rec_floats(D);
  const int64_t stride = (int64_t)J.nq * att_rec_floats(D);   // between units
  // launched while the partial kernel runs: wait for its results
  asm volatile("griddepcontrol.wait;" ::: "memory");
  float M = -INFINITY;
  for (int s = threadIdx.x; s < nsp; s += 128) M = fmaxf(M, recs[s * stride]);
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
  if (lane == 0) red[warp][0] = M;
  __syncthreads();
  M = fmaxf(fmaxf(red[0][0], red[1][0]), fmaxf(red[2][0], red[3][0]));
  float Ls = 0.f;
  float y[E];
#pragma unroll
  for (int e = 0; e < E; ++e) y[e] = 0.f;
#pragma unroll 4
  for (int s = warp; s < nsp; s += 4) {
    const float* ra = recs + s * stride;
    const float f = ex2_approx(ra[0] - M);
    Ls = __fmaf_rn(ra[1], f, Ls);
#pragma unroll
    for (int e = 0; e < E; ++e) y[e] = __fmaf_rn(ra[2 + lane + 32 * e], f, y[e]);
  }
#pragma unroll
  for (int e = 0; e < E; ++e) part[warp][lane + 32 * e] = y[e];
  if (lane == 0) red[warp][1] = Ls;
  __syncthreads();
  if (warp != 0) return;
  const float inv = 1.f / (red[0][1] + red[1][1] + red[2][1] + red[3][1]);
  float* row = part[0];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int j = lane + 32 * e;
    row[j] = (part[0][j] + part[1][j] + part[2][j] + part[3][j]) * inv;
  }
  warp_fwht<D>(row, lane);
  const float sc = rsqrtf((float)D);
  uint8_t* orow = reinterpret_cast<uint8_t*>(J.out) + (int64_t)a * J.out_stride * ESZ;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int j = lane + 32 * e;
    float v = row[j] * sc;
    if ((J.sv[j >> 5] >> (j & 31)) & 1u) v = -v;
    if constexpr (ESZ == 2) reinterpret_cast<__nv_bfloat16*>(orow)[j] = __float2bfloat16_rn(v);
    else reinterpret_cast<float*>(orow)[j] = v;
  }
}

// Launches the partial and combine kernels for one group of jobs.  The grid
// is every CTA that fits on the device at once, or one per unit.
template <int D, typename TQ, int QT>
static cudaError_t launch_attend_t(const AttParams& p_in, int nq_max, float* ws, int sms, cudaStream_t st) {
  using C = Att<D, QT>;
  auto kp = attend_partial<D, QT>;
  // per device, set on the first launch; atomic so that host threads making
  // first calls at once do not race (each sets the same values)
  static std::atomic<int> regs[64];
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (regs[dev].load(std::memory_order_acquire) == 0) {
    cudaError_t e = cudaFuncSetAttribute(kp, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    if (e != cudaSuccess) return e;
    cudaFuncAttributes fa;
    e = cudaFuncGetAttributes(&fa, kp);
    if (e != cudaSuccess) return e;
    regs[dev].store(fa.numRegs > 0 ? fa.numRegs : 1, std::memory_order_release);
  }
  AttParams p = p_in;
  p.stage = p.tab_k = p.tab_v = 0;
  for (int j = 0; j < p.njobs; ++j) {
    const AttJob& J = p.job[j];
    p.stage = std::max(p.stage, att_stage_bytes(D, J.wk, J.bk, J.mk, J.wv, J.bv, J.mv, C::MERGE));
    p.tab_k = std::max(p.tab_k, 8 << (J.wk + J.lgrk));
    p.tab_v = std::max(p.tab_v, 8 << (J.wv + J.lgrv));
  }
  const int smem = C::smem(p.stage, p.tab_k + p.tab_v);
  const int regs_cta = ((regs[dev].load(std::memory_order_relaxed) * 32 + 255) / 256) * 256 * kAttWarps;
  const int per_sm = std::max(1, std::min(228 * 1024 / (smem + 1024), 65536 / regs_cta));
  p.nctas = (int32_t)std::min<int64_t>(std::min<int64_t>(p.nunits, (int64_t)sms * per_sm), kAttMaxCtas);
  if (p.nctas < 1) return cudaSuccess;
  const int per = p.nunits / p.nctas, extra = p.nunits % p.nctas;
  for (int c = 0, j = 0; c < p.nctas; ++c) {
    while (j + 1 < p.njobs && p.job[j + 1].unit0 <= c * per + std::min(c, extra)) ++j;
    p.first_job[c] = (uint8_t)j;
  }
  kp<<<p.nctas, kAttThreads, smem, st>>>(p, ws);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  // the combine kernel starts as the partial kernel's CTAs leave and waits for
  // its results on the device: its launch latency overlaps the partial kernel
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)nq_max, (unsigned)p.njobs);
  cfg.blockDim = dim3(128);
  cfg.stream = st;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, attend_combine<D, TQ>, p, (const float*)ws);
}

// The workspace of tac_attend_multi_static: one array per device, in the
// module image (no allocation at call time).
static __device__ __align__(256) float g_attend_ws[TAC_ATTEND_STATIC_WS_BYTES / 4];

// Address of g_attend_ws on the current device, resolved once per device.
cudaError_t attend_static_workspace(float** ws) {
  constexpr int kMaxDevices = 64;
  static std::atomic<void*> cache[kMaxDevices];
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  void* a = cache[dev].load(std::memory_order_acquire);
  if (!a) {
    e = cudaGetSymbolAddress(&a, g_attend_ws);
    if (e != cudaSuccess) return e;
    if (!a || (reinterpret_cast<uintptr_t>(a) & 255)) return cudaErrorInvalidSymbol;
    cache[dev].store(a, std::memory_order_release);   // racing first calls store the same address
  }
  *ws = static_cast<float*>(a);
  return cudaSuccess;
}

// nq_max: the largest query count of the jobs (the kernel is built for up to 4 and up to 8).
cudaError_t launch_attend(int d, int dtype, int nq_max, const AttParams& p, float* ws, int sms,
                          cudaStream_t st) {
  const bool bf = dtype == TAC_BF16;
#define TAC_ATT_NQ(DD, T)                                                                 \
  return nq_max <= 4 ? launch_attend_t<DD, T, 1>(p, nq_max, ws, sms, st)              \
                     : launch_attend_t<DD, T, 2>(p, nq_max, ws, sms, st);
  if (d == 64) { if (bf) { TAC_ATT_NQ(64, __nv_bfloat16) } else { TAC_ATT_NQ(64, float) } }
  if (d == 128) { if (bf) { TAC_ATT_NQ(128, __nv_bfloat16) } else { TAC_ATT_NQ(128, float) } }
#undef TAC_ATT_NQ
  return cudaErrorInvalidValue;
}

}  // namespace tac

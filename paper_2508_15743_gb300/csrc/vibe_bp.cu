// K1 -- persistent serial-schedule min-sum BP ensemble with the ensemble selection fused in.
//
// One warp decodes one shot at a time and pulls shots from a global counter until the batch is
// done. For its shot the warp runs the K members one after another (Sec. III.D.2): member i keeps its
// variable-to-check messages in the warp's slice of shared memory, sweeps its steps (k_steps in
// vibe_graph.cu: up to 32 edges of columns that share no check, one lane per edge) and stops as soon
// as H e = s (Algorithm 1).
//
// Correction limit (Sec. III.D.2 step 3). The candidates are the first M converged members in
// (iteration, member) order. Running members in index order, member i can only enter that set by
// converging before the M-th candidate's iteration, so it gets the budget t_M - 1 once M candidates
// exist (T before). Members whose budget is 0 are skipped. This is the lock-step rule of the paper
// without the waiting: every member's trajectory is independent of the others, so the candidate set
// and the chosen correction are identical, and no sweep that cannot change the result is run.
//
// Ranking (step 4): the chosen candidate minimises W(e) = sum over e_j = 1 of lambda_j (float, ascending
// j), ties to the earlier candidate. With no converged member (step 5) the warp accumulates
// LLR^i / ||LLR^i||_2 over all members in index order and hands (1/K) * sum to the LSD kernel.
//
// Arithmetic is the oracle's to the bit: fixed per-node operation order, __fadd_rn/__fmul_rn (no
// contraction), min and sign exact. Stored messages are never -0 (a sum that starts at lambda_v > 0
// cannot round to -0 in FP32; FP16 stores map -0 to +0), so the sign bit of a message equals x < 0.
#include <algorithm>
#include <type_traits>

#include "vibe_internal.cuh"

namespace vibe {
namespace {

// A stored message in shared memory, and the row scan: |x| minimum with the XOR of the signs as its
// sign over the 16-byte chunks of a row, as a float (min.xorsign.abs does both at once; a NaN -- the sum
// of +inf and -inf -- never wins and has sign 0).
template <typename MT>
struct Msg;

__device__ __forceinline__ float minx(float a, float b) {
  float d;
  asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
  return d;
}
__device__ __forceinline__ uint32_t minx2(uint32_t a, uint32_t b) {   // two halves
  uint32_t d;
  asm("min.xorsign.abs.f16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}

template <>
struct Msg<float> {
  static constexpr int kBytes = 4;
  static constexpr int kSpc = 4;   // slots per 16-byte chunk of a row
  static constexpr uint32_t kInf = kInfBits;
  static constexpr bool kDrop = true;   // the scan leaves the own slot out itself (rows of known length)
  __device__ __forceinline__ static void store(uint32_t a, uint32_t b) { sts32(a, b); }
  __device__ __forceinline__ static uint32_t round(float x) { return __float_as_uint(x); }
  __device__ __forceinline__ static void store(float* p, float x) { *p = x; }
  __device__ __forceinline__ static float value(float x) { return x; }
  template <int NCH>
  __device__ __forceinline__ static float scan(uint32_t row, int nch, uint32_t pos) {
    float v = __int_as_float(0x7f800000);
    auto chunk = [&](uint32_t a, uint32_t drop) {
      const uint4 q = lds128(a);
      const float inf = __uint_as_float(kInfBits);
      const float x = (drop & 1u) ? inf : __uint_as_float(q.x), y = (drop & 2u) ? inf : __uint_as_float(q.y);
      const float z = (drop & 4u) ? inf : __uint_as_float(q.z), w = (drop & 8u) ? inf : __uint_as_float(q.w);
      v = minx(v, minx(minx(x, y), minx(z, w)));
    };
    if (NCH) {
      const uint32_t own = 1u << pos;
#pragma unroll
      for (int i = 0; i < NCH; ++i) chunk(row + 16 * i, own >> (4 * i));
    } else {
      for (int i = 0; i < nch; ++i) chunk(row + 16 * i, 0u);
    }
    return v;
  }
};

template <>
struct Msg<__half> {
  static constexpr int kBytes = 2;
  static constexpr int kSpc = 8;
  static constexpr uint32_t kInf = 0x7c00u;
  static constexpr bool kDrop = false;
  __device__ __forceinline__ static void store(uint32_t a, uint32_t b) { sts16(a, b); }
  __device__ __forceinline__ static uint32_t round(float x) {   // -0 as +0
    const uint32_t h = (uint32_t)__half_as_ushort(__float2half_rn(x));
    return h == 0x8000u ? 0u : h;
  }
  __device__ __forceinline__ static void store(__half* p, float x) {
    *reinterpret_cast<unsigned short*>(p) = (unsigned short)round(x);
  }
  __device__ __forceinline__ static float value(__half x) { return __half2float(x); }
  template <int NCH>
  __device__ __forceinline__ static float scan(uint32_t row, int nch, uint32_t) {
    uint32_t v = 0x7c007c00u;
    auto chunk = [&](uint32_t a) {
      const uint4 q = lds128(a);
      v = minx2(v, minx2(minx2(q.x, q.y), minx2(q.z, q.w)));
    };
    if (NCH) {
#pragma unroll
      for (int i = 0; i < NCH; ++i) chunk(row + 16 * i);
    } else {
      for (int i = 0; i < nch; ++i) chunk(row + 16 * i);
    }
    return __half2float(__ushort_as_half((unsigned short)minx2(v, v >> 16)));
  }
};

__device__ __forceinline__ bool is_finite_bits(float x) {
  return (__float_as_uint(x) & 0x7f800000u) != 0x7f800000u;
}

// One parallel (flooding) iteration of Algorithm 1 on the warp's FP32 message image.
// Check pass: a lane takes whole rows; from the smallest magnitude, the second smallest, the slot
// holding the smallest and the sign parity of the row's variable-to-check messages it overwrites each
// real slot with that edge's check-to-variable message (minimum and sign product over the other
// slots: exactly the exclusion over N(c) \ v). Column pass: a lane takes whole columns and turns its
// own slots into the new variable-to-check messages with the sums of the serial update. Every column
// reads only its own slots, so the passes need no second image. Parity pass: (H e)_c XOR s_c from
// the decisions (many columns touch a check in the column pass); returns whether the lane met an
// unsatisfied check.
// Its cost is instructions (18.4 G warp instructions for 60,000 shots of an all-flooding d=7 ensemble before, 13.2 G
// in the form that read the tables from the parameter space): the row's swizzle is found once per row, from a row pitch
// known at compile time, and a column's entries are one load. All flooding, d=7 phenomenological, K=8, T=20, 200,000
// shots: FP32 86.1 -> 45.5 ms, FP16 (layer_sweep) 82.0 -> 59.2; all layered 199.9 -> 125.3 and 146.7 -> 106.1.
// The csc_ent entries of column v (entries past its degree are not used). Where DP <= 4 every problem of the launch
// has the pitch 4: one load.
template <int DP>
__device__ __forceinline__ void column_entries(const uint32_t* csc, size_t pitch, int v, int deg, uint32_t (&ent)[DP]) {
  if constexpr (DP <= 4) {
    const uint4 x = __ldg(reinterpret_cast<const uint4*>(csc) + v);
    const uint32_t e[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
    for (int k = 0; k < DP; ++k) ent[k] = e[k];
  } else {
#pragma unroll
    for (int k = 0; k < DP; ++k) ent[k] = k < deg ? __ldg(csc + v * pitch + k) : 0u;
  }
}

__device__ __forceinline__ uint32_t syn_bit(const uint32_t* s32, int c) { return (s32[c >> 5] >> (c & 31)) & 1u; }

template <int DP, int NCH>
__device__ __forceinline__ bool flood_sweep(const Tables& t, float alpha, float* msgs, uint8_t* dec8,
                                            const uint32_t* s32, float* lpost, int lane) {
  const int m = t.m, n = t.n;
  // copies of t's fields: the stores below might alias t, which would make every use a load
  const int32_t *rowptr = t.rowptr, *colidx = t.colidx, *colptr = t.colptr;
  const uint32_t* csc = t.csc_ent;
  const float* lam = t.lam;
  const size_t pitch = (size_t)t.DP;
  const uint32_t RP = NCH ? (uint32_t)(NCH * Msg<float>::kSpc) : (uint32_t)t.RP;
  for (int c = lane; c < m; c += 32) {
    const int deg = __ldg(rowptr + c + 1) - __ldg(rowptr + c);
    float* row = msgs + (size_t)c * RP;
    const uint32_t swz = row_position((uint32_t)c, 0u, (int)RP, 4);   // slot j is at j ^ swz
    float m1 = __int_as_float(0x7f800000), m2 = m1;
    int a1 = -1;
    uint32_t sx = 0;
    for (int j = 0; j < deg; ++j) {
      const float x = row[(uint32_t)j ^ swz];
      const float ax = fabsf(x);
      sx ^= __float_as_uint(x) >> 31;
      if (ax < m1) { m2 = m1; m1 = ax; a1 = j; }
      else if (ax < m2) m2 = ax;
    }
    for (int j = 0; j < deg; ++j) {
      const uint32_t pos = (uint32_t)j ^ swz;
      const float x = row[pos];
      const float mn = j == a1 ? m2 : m1;
      const uint32_t neg = (sx ^ (__float_as_uint(x) >> 31) ^ syn_bit(s32, c)) & 1u;
      const float mag = __fmul_rn(alpha, mn);
      row[pos] = neg ? -mag : mag;
    }
  }
  __syncwarp();
  for (int v = lane; v < n; v += 32) {
    const int deg = __ldg(colptr + v + 1) - __ldg(colptr + v);
    uint32_t ent[DP];
    column_entries<DP>(csc, pitch, v, deg, ent);
    float* slot[DP];
    float cv[DP];
#pragma unroll
    for (int k = 0; k < DP; ++k) {
      slot[k] = msgs;
      cv[k] = 0.0f;
      if (k < deg) {
        slot[k] = msgs + (size_t)(ent[k] >> 9) * RP + (ent[k] & 0xffu);
        cv[k] = *slot[k];
      }
    }
    const float lamv = __ldg(lam + v);
    float L = lamv;
#pragma unroll
    for (int k = 0; k < DP; ++k)
      if (k < deg) L = __fadd_rn(L, cv[k]);
    float pre = lamv;   // lambda + m_0 + ... + m_{k-1}, the shared head of every exclusion sum
#pragma unroll
    for (int k = 0; k < DP; ++k) {
      if (k < deg) {
        float a = pre;
#pragma unroll
        for (int k2 = k + 1; k2 < DP; ++k2)
          if (k2 < deg) a = __fadd_rn(a, cv[k2]);
        *slot[k] = a;
        pre = __fadd_rn(pre, cv[k]);
      }
    }
    dec8[v] = L <= 0.0f ? 1u : 0u;
    if (lpost) lpost[v] = L;
  }
  __syncwarp();
  bool bad = false;
  for (int c = lane; c < m; c += 32) {
    uint32_t p = syn_bit(s32, c);
    for (int e = __ldg(rowptr + c); e < __ldg(rowptr + c + 1); ++e) p ^= dec8[__ldg(colidx + e)];
    bad |= p != 0u;
  }
  __syncwarp();
  return bad;
}

// One iteration of a schedule over check layers, with the check-to-variable messages in their own
// float image cv (same slot layout as the message image msgs): the layered schedule (the oracle's
// reading R10; layers from the graph builder) or, with flood set, the parallel schedule as a single
// layer of all checks (Algorithm 1's other branch, reading R8), which FP16 message storage needs:
// there the check-to-variable messages of an iteration are float temporaries and only the stored
// variable-to-check messages are rounded.
// Per layer, a check pass (lane per check of the layer: smallest and second-smallest magnitude, the
// slot of the smallest and the sign parity of the row's variable-to-check messages give each edge's
// minimum and sign product over the other edges, scaled by alpha and signed by the syndrome bit) and a
// column pass (lane per column of the layer's checks, which share no column: the serial update's
// exclusion sums over the column's current cv entries, stored as its new variable-to-check messages).
// Then every posterior (lambda plus the column's cv entries in ascending check order), decision and
// check parity. cv holds zeros when a layered member starts (init in run_member).
template <typename MT, int DP, int NCH>
__device__ __forceinline__ bool layer_sweep(const Tables& t, float alpha, bool flood, MT* msgs, float* cv,
                                            uint8_t* dec8, const uint32_t* s32, float* lpost, int lane) {
  const int m = t.m, n = t.n;
  // copies of t's fields: the stores below might alias t, which would make every use a load
  const int32_t *rowptr = t.rowptr, *colidx = t.colidx, *colptr = t.colptr, *layer_ptr = t.layer_ptr,
                *layer_chk = t.layer_chk, *layer_vptr = t.layer_vptr, *layer_var = t.layer_var;
  const uint32_t* csc = t.csc_ent;
  const float* lam = t.lam;
  const size_t pitch = (size_t)t.DP;
  const uint32_t RP = NCH ? (uint32_t)(NCH * Msg<MT>::kSpc) : (uint32_t)t.RP;
  const int nl = flood ? 1 : t.nlayer;
  for (int l = 0; l < nl; ++l) {
    const int c0 = flood ? 0 : __ldg(layer_ptr + l), c1 = flood ? m : __ldg(layer_ptr + l + 1);
    for (int q = c0 + lane; q < c1; q += 32) {
      const int c = flood ? q : __ldg(layer_chk + q);
      const int deg = __ldg(rowptr + c + 1) - __ldg(rowptr + c);
      const MT* row = msgs + (size_t)c * RP;
      float* crow = cv + (size_t)c * RP;
      const uint32_t swz = row_position((uint32_t)c, 0u, (int)RP, Msg<MT>::kSpc);   // slot j is at j ^ swz
      float m1 = __int_as_float(0x7f800000), m2 = m1;
      int a1 = -1;
      uint32_t sx = 0;
      for (int j = 0; j < deg; ++j) {
        const float x = Msg<MT>::value(row[(uint32_t)j ^ swz]);
        const float ax = fabsf(x);
        sx ^= __float_as_uint(x) >> 31;
        if (ax < m1) { m2 = m1; m1 = ax; a1 = j; }
        else if (ax < m2) m2 = ax;
      }
      for (int j = 0; j < deg; ++j) {
        const uint32_t pos = (uint32_t)j ^ swz;
        const float x = Msg<MT>::value(row[pos]);
        const uint32_t neg = (sx ^ (__float_as_uint(x) >> 31) ^ syn_bit(s32, c)) & 1u;
        const float mag = __fmul_rn(alpha, j == a1 ? m2 : m1);
        crow[pos] = neg ? -mag : mag;
      }
    }
    __syncwarp();
    const int v0 = flood ? 0 : __ldg(layer_vptr + l), v1 = flood ? n : __ldg(layer_vptr + l + 1);
    for (int q = v0 + lane; q < v1; q += 32) {
      const int v = flood ? q : __ldg(layer_var + q);
      const int deg = __ldg(colptr + v + 1) - __ldg(colptr + v);
      uint32_t slot[DP], ent[DP];
      column_entries<DP>(csc, pitch, v, deg, ent);
      float c2v[DP];
#pragma unroll
      for (int k = 0; k < DP; ++k) {
        slot[k] = 0u;
        c2v[k] = 0.0f;
        if (k < deg) {
          slot[k] = (ent[k] >> 9) * RP + (ent[k] & 0xffu);
          c2v[k] = cv[slot[k]];
        }
      }
      float pre = __ldg(lam + v);   // lambda + m_0 + ... + m_{k-1}, the shared head of every exclusion sum
#pragma unroll
      for (int k = 0; k < DP; ++k) {
        if (k < deg) {
          float a = pre;
#pragma unroll
          for (int k2 = k + 1; k2 < DP; ++k2)
            if (k2 < deg) a = __fadd_rn(a, c2v[k2]);
          Msg<MT>::store(msgs + slot[k], a);
          pre = __fadd_rn(pre, c2v[k]);
        }
      }
    }
    __syncwarp();
  }
  for (int v = lane; v < n; v += 32) {
    const int deg = __ldg(colptr + v + 1) - __ldg(colptr + v);
    float L = __ldg(lam + v);
    uint32_t ent[DP];
    column_entries<DP>(csc, pitch, v, deg, ent);
#pragma unroll
    for (int k = 0; k < DP; ++k)
      if (k < deg) L = __fadd_rn(L, cv[(ent[k] >> 9) * RP + (ent[k] & 0xffu)]);
    dec8[v] = L <= 0.0f ? 1u : 0u;
    if (lpost) lpost[v] = L;
  }
  __syncwarp();
  bool bad = false;
  for (int c = lane; c < m; c += 32) {
    uint32_t p = syn_bit(s32, c);
    for (int e = __ldg(rowptr + c); e < __ldg(rowptr + c + 1); ++e) p ^= dec8[__ldg(colidx + e)];
    bad |= p != 0u;
  }
  __syncwarp();
  return bad;
}

// Warps per SM the register budget targets. Shared-memory wavefronts bound the kernel, which this many
// warps keep busy; the FP32 states of the d=9 phenomenological problem fill shared memory at 20.
template <typename MT, int DP>
struct MinBlocks { static constexpr int value = (DP <= 8 ? 20 : 16) / kBpWarpsPerCta; };

// What a member's run is told and what it reports.
struct ImageRun {
  int budget;               // sweeps at most
  bool soft, keep_last;     // the posterior after every sweep / after sweep T
  const int* conv;          // pair mode: the shot's converged members (pair_should_stop), else NULL
  float* lpost;             // global: n posteriors
  uint32_t* st;             // the steps' decision words: shared (generic address) or global
  int ran;                  // result: sweeps run
};

constexpr int kRecSteps = 2;   // steps fetched together, one group ahead

// One serial sweep of a member over its ns steps on the message image at shared address msgs. A lane
// holds one edge of a step (its check is no other lane's): it scans its row with +inf -- a magnitude that
// never wins a minimum, sign bit 0 -- in the place of its own slot, which gives the minimum and sign
// product over the other slots exactly (FP32 rows of up to four chunks put it in while scanning, which
// saves the 3.5 wavefronts of a scattered store; FP16 rows, where the halves cost more instructions than
// that, and longer rows have it written to the slot first), gets
// the column's other messages from their lanes, forms its exclusion sum in the order of Algorithm 1 and
// stores the new message in its slot. Decisions are one
// word per step (on the lane of the column's last edge); check parities are flipped, and the word
// stored, only when one changes.
// What bounds it: shared-memory wavefronts (90 % of their peak with FP32 messages; with FP16 77 %, and issue at
// 67 %). The lanes' rows are random; the order of a step's columns (k_step_order) brings a 16-byte row load of 32
// lanes from ~9.5 wavefronts to ~8 (ideal 4). With one lane per column a sweep of the d=9 phenomenological problem
// took 42 chunks of 187 warp instructions and 2800 wavefronts in all; its 62 steps take 95 (FP16 84) and 33
// wavefronts (FP16 20) each, by the profiler's counters. Measured, 32768 shots of it (K=16, T=30):
// 96.7 -> 61.7 ms with FP32 messages (73.1 before the order and without the dropped slot), 78.1 -> 48.0 ms with
// FP16; the 4.8.8 code, whose rows of 10 now take three chunks instead of four, 40 -> 13 ms.
// NCH: 16-byte chunks of a row (0: from the tables). par32 holds the check parities.
template <typename MT, int DP, int NCH, bool LP>
__device__ __forceinline__ void step_sweep(const Tables& t, const uint32_t* soff, const int ns, const size_t first,
                                           const float alpha, const uint32_t msgs, const uint32_t s32,
                                           const uint32_t par32, uint32_t* st, float* lp, const int lane) {
  const int nch = NCH ? NCH : t.RP / Msg<MT>::kSpc;
  const uint32_t row_bytes = (uint32_t)nch * 16u;
  // the chunk swizzle of row_position(): slot ^ ((check >> a) & (n - 1)) * slots per chunk
  const uint32_t swz_mask = (nch == 2 || nch == 4 || nch == 8) ? (uint32_t)nch - 1u : 0u;
  const int swz_shift = nch == 2 ? 2 : nch == 4 ? 1 : 0;
  const uint2* trec = t.xrec + first + lane;
  const uint32_t* tlnk = t.xlnk + first + lane;
  const bool wide = DP > 16 && t.DP > 16;
  uint32_t o[kRecSteps + 1], on[kRecSteps + 1];   // first slots of this group's steps and the next one's
  uint2 r[kRecSteps], rn[kRecSteps];
  uint32_t ln[kRecSteps], lnn[kRecSteps];
  auto fetch = [&](const uint32_t (&off)[kRecSteps + 1], uint2 (&rec)[kRecSteps], uint32_t (&lnk)[kRecSteps]) {
#pragma unroll
    for (int u = 0; u < kRecSteps; ++u) {
      rec[u] = make_uint2(0u, 0u);
      lnk[u] = 0u;
      if (off[u] + (uint32_t)lane < off[u + 1]) {
        rec[u] = __ldg(trec + off[u]);
        lnk[u] = __ldg(tlnk + off[u]);
      }
    }
  };
#pragma unroll
  for (int u = 0; u <= kRecSteps; ++u) {
    o[u] = __ldg(soff + u);
    on[u] = __ldg(soff + kRecSteps + u);
  }
  fetch(o, r, ln);
  for (int s0 = 0; s0 < ns; s0 += kRecSteps) {
    fetch(on, rn, lnn);
    uint32_t of[kRecSteps];   // the offsets after the next group's
#pragma unroll
    for (int u = 0; u < kRecSteps; ++u) of[u] = __ldg(soff + s0 + 2 * kRecSteps + 1 + u);
#pragma unroll
    for (int u = 0; u < kRecSteps; ++u) {
      const uint32_t old = s0 + u < ns ? st[s0 + u] : 0u;
      const uint32_t c = r[u].x >> 18;
      const uint32_t row = msgs + c * row_bytes;
      uint32_t pos = r[u].x & 0xffu;
      if (NCH == 0 || NCH == 2 || NCH == 4 || NCH == 8) pos ^= ((c >> swz_shift) & swz_mask) * (uint32_t)Msg<MT>::kSpc;
      const uint32_t own = row + pos * (uint32_t)Msg<MT>::kBytes;
      const bool act = (int)ln[u] < 0;
      if (!(Msg<MT>::kDrop && NCH) && act) Msg<MT>::store(own, Msg<MT>::kInf);
      const uint32_t sw = lds32(s32 + ((c >> 5) << 2));
      const float mn = Msg<MT>::template scan<NCH>(row, nch, pos);
      const uint32_t mcv = __float_as_uint(__fmul_rn(alpha, mn)) ^ (__funnelshift_l(0u, sw, ~c) & 0x80000000u);
      float acc = __uint_as_float(r[u].y);
      // links of columns of more than 16 checks: first lane | k << 5 | degree - 1 << 10
      uint32_t incl = ln[u] >> 5, lastl = (ln[u] >> kLnkLastLane) & 31u;
      if (wide) {
        const uint32_t k = (ln[u] >> 5) & 31u, dm1 = (ln[u] >> 10) & 31u;
        incl = ((2u << dm1) - 1u) & ~(1u << k);
        lastl = (ln[u] + dm1) & 31u;
      } else if (DP > 16) {
        incl &= 0xffffu;
      }
#pragma unroll
      for (int j = 0; j < DP; ++j)
        acc = add_if(acc, __uint_as_float(__shfl_sync(kFull, mcv, (int)ln[u] + j)), incl & (1u << j));
      const float L = __fadd_rn(acc, __uint_as_float(mcv));   // on the last edge's lane: the posterior
      const uint32_t dec = __ballot_sync(kFull, (ln[u] & kLnkLast) && L <= 0.0f);
      if (act) Msg<MT>::store(own, Msg<MT>::round(acc));
      const uint32_t ch = dec ^ old;
      if (ch) {   // some column of the step changed its decision
        if (act && ((ch >> lastl) & 1u)) red_xor_shared(par32 + ((c >> 5) << 2), 1u << (c & 31));
        if (lane == 0) st[s0 + u] = dec;
      }
      if (LP) {
        if (ln[u] & kLnkLast) lp[__ldg(t.xcolid + first + o[u] + lane)] = L;
        else if (ln[u] == 0u && o[u] + (uint32_t)lane < o[u + 1])   // column without checks
          lp[__ldg(t.xcolid + first + o[u] + lane)] = __uint_as_float(r[u].y);
      }
      __syncwarp();
    }
#pragma unroll
    for (int u = 0; u < kRecSteps; ++u) { r[u] = rn[u]; ln[u] = lnn[u]; }
#pragma unroll
    for (int u = 0; u <= kRecSteps; ++u) o[u] = on[u];
    on[0] = on[kRecSteps];
#pragma unroll
    for (int u = 0; u < kRecSteps; ++u) on[u + 1] = of[u];
  }
}

// One member (index i) of the shot whose syndrome words are in the warp's shared memory at byte offset
// smem_off: initialises the member's message image and runs up to `budget` sweeps, stopping at the first
// that leaves H e = s, or in pair mode before a sweep that no longer counts. Returns the converging sweep
// (0 if none); leaves the decisions in the step words (serial member) or the decision bytes, and the
// posterior of the last sweep in lpost when soft output is on or `keep_last` is set and the member
// reached sweep T. Not inlined: the sweep gets its own registers, whatever the caller keeps.
template <typename MT, int DP, int NCH>
__device__ __noinline__ int run_member(const Tables& t, int i, int smem_off, ImageRun& R) {
  extern __shared__ __align__(16) unsigned char smem[];
  unsigned char* base = smem + smem_off;
  const int lane = __shfl_sync(kFull, (int)(threadIdx.x & 31), (int)(threadIdx.x & 31));
  const uint32_t sbase = __shfl_sync(kFull, (uint32_t)__cvta_generic_to_shared(smem) + (uint32_t)smem_off, lane);
  const int n = t.n, m = t.m, T = t.T, mw = t.mw;
  const int n4 = (n + 3) >> 2;
  const int msg_vec = (int)(((size_t)m * t.RP * sizeof(MT)) / 16);
  const uint32_t* s32 = reinterpret_cast<const uint32_t*>(base + t.off_s);
  uint32_t* par = reinterpret_cast<uint32_t*>(base + t.off_par);
  const bool flood = i < t.n_flood;
  const bool layered = !flood && i < t.n_flood + t.n_layered;
  const int ns = __ldg(t.stepcnt + i);
  // member init: messages from the prior image, decisions 0, parity = s
  {
    const uint4* src = reinterpret_cast<const uint4*>(t.msg_init);
    for (int q = lane; q < msg_vec; q += 32) sts128(sbase + t.off_msg + 16 * q, __ldg(src + q));
    if (flood || layered) {
      uint32_t* d32 = reinterpret_cast<uint32_t*>(base + t.off_dec);
      for (int q = lane; q < n4; q += 32) d32[q] = 0u;
    } else {
      for (int q = lane; q < ns; q += 32) R.st[q] = 0u;
    }
    for (int q = lane; q < mw; q += 32) par[q] = s32[q];
  }
  float* cv = t.off_cv >= 0 ? reinterpret_cast<float*>(base + t.off_cv) : nullptr;
  if (layered) {   // the layered member's check-to-variable messages start at zero
    uint4* c4 = reinterpret_cast<uint4*>(cv);
    const int cv_vec = (int)(((size_t)m * t.RP * 4) / 16);
    for (int q = lane; q < cv_vec; q += 32) c4[q] = make_uint4(0u, 0u, 0u, 0u);
  }
  __syncwarp();

  const size_t first = (size_t)i * t.SP;
  const uint32_t* soff = t.soff + (size_t)i * t.soff_pitch;
  const float alpha = __ldg(t.alpha_m + i);   // member i's scaling factor
  const int budget = R.budget;
  int conv = 0, ran = 0;
  for (int it = 1; it <= budget; ++it) {
    if (R.conv && pair_should_stop(R.conv, t.K, t.M, i, it, lane)) break;
    // the posterior is needed after the last possible sweep of a member that may end without
    // converging (LLR average) and, for soft output, after every sweep
    float* lp = (R.soft || (it == T && R.keep_last)) ? R.lpost : nullptr;
    bool bad = false;
    if (flood || layered) {
      MT* msgs = reinterpret_cast<MT*>(base + t.off_msg);
      uint8_t* dec8 = base + t.off_dec;
      if (std::is_same<MT, float>::value && flood)
        bad = flood_sweep<DP, NCH>(t, alpha, reinterpret_cast<float*>(msgs), dec8, s32, lp, lane);
      else
        bad = layer_sweep<MT, DP, NCH>(t, alpha, flood, msgs, cv, dec8, s32, lp, lane);
    } else {
      if (lp)
        step_sweep<MT, DP, NCH, true>(t, soff, ns, first, alpha, sbase + t.off_msg, sbase + t.off_s, sbase + t.off_par,
                                      R.st, lp, lane);
      else
        step_sweep<MT, DP, NCH, false>(t, soff, ns, first, alpha, sbase + t.off_msg, sbase + t.off_s, sbase + t.off_par,
                                       R.st, nullptr, lane);
      for (int q = lane; q < mw; q += 32) bad |= lds32(sbase + t.off_par + 4 * q) != 0u;
      __syncwarp();
    }
    ran = it;
    if (!__any_sync(kFull, bad)) { conv = it; break; }
  }
  R.ran = ran;
  return conv;
}

// The decisions a converged member left, as bits in column order in shared memory, and W(e) = sum of
// lambda_j over e_j = 1, ascending j.
__device__ __forceinline__ float member_bits(const Tables& t, int i, unsigned char* base, const uint32_t* st,
                                             uint32_t* bits, int lane) {
  const int n = t.n, nw = t.nw;
  if (i < t.n_flood + t.n_layered) {
    const uint8_t* dec8 = base + t.off_dec;
    for (int w = 0; w < nw; ++w) {
      const int v = 32 * w + lane;
      const uint32_t word = __ballot_sync(kFull, v < n && dec8[v] != 0);
      if (lane == 0) bits[w] = word;
    }
  } else {
    const uint32_t* soff = t.soff + (size_t)i * t.soff_pitch;
    const uint32_t* colid = t.xcolid + (size_t)i * t.SP;
    const int ns = __ldg(t.stepcnt + i);
    for (int w = lane; w < nw; w += 32) bits[w] = 0u;
    __syncwarp();
    for (int s = lane; s < ns; s += 32) {
      uint32_t d = st[s];
      if (!d) continue;
      const uint32_t o = __ldg(soff + s);
      while (d) {
        const uint32_t v = __ldg(colid + o + (uint32_t)__ffs(d) - 1u);
        atomicOr(bits + (v >> 5), 1u << (v & 31));
        d &= d - 1u;
      }
    }
  }
  __syncwarp();
  float W = 0.0f;
  for (int w = 0; w < nw; ++w) {
    uint32_t x = bits[w];
    while (x) {
      W = __fadd_rn(W, __ldg(t.lam + 32 * w + __ffs(x) - 1));
      x &= x - 1;
    }
  }
  return W;
}

// The syndrome of a shot as words in shared memory (bits past m cleared); returns whether it is not zero.
__device__ __forceinline__ bool load_syndrome(const Tables& t, const uint32_t* syn, uint32_t* s32, int lane) {
  uint32_t any = 0;
  for (int w = lane; w < t.mw; w += 32) {
    const int rem = t.m - 32 * w;
    const uint32_t x = __ldg(syn + w) & (rem >= 32 ? 0xffffffffu : ((1u << rem) - 1u));
    s32[w] = x;
    any |= x;
  }
  any = __any_sync(kFull, any != 0u);
  __syncwarp();
  return any != 0u;
}

// Decodes one shot of problem t with the warp (the body of the persistent loop below). smem_off: the
// warp's shared memory; acc, lpost, cand_post, gst: its global scratch.
template <typename MT, int DP, int NCH>
__device__ __forceinline__ void decode_shot(const BpArgs& a, const Tables& t, uint32_t shot, unsigned char* base,
                                            int smem_off, float* acc, float* lpost, float* cand_post, uint32_t* gst,
                                            int lane, unsigned long long& my_iters, unsigned long long& my_shots,
                                            unsigned long long& my_fail) {
  const int n = t.n, K = t.K, M = t.M, T = t.T, nw = t.nw, kw = t.kw;
  uint32_t* cand = reinterpret_cast<uint32_t*>(base + t.off_cand);
  uint32_t* st = t.off_st >= 0 ? reinterpret_cast<uint32_t*>(base + t.off_st) : gst;
  const bool any = load_syndrome(t, a.syn + (size_t)shot * a.syn_stride, reinterpret_cast<uint32_t*>(base + t.off_s), lane);
  ++my_shots;
  uint32_t* out_corr = a.corr + (size_t)shot * a.corr_stride;

  if (!any && !a.want_soft) {
    // s = 0: every member converges in iteration 1 to e = 0; the first M are the candidates, all of
    // weight 0, so member 0 is chosen.
    for (int w = lane; w < nw; w += 32) out_corr[w] = 0u;
    if (a.logical)
      for (int w = lane; w < kw; w += 32) a.logical[(size_t)shot * a.log_stride + w] = 0u;
    if (a.obs) {
      uint32_t f = 0;
      for (int w = lane; w < kw; w += 32) f |= a.obs[(size_t)shot * a.log_stride + w];
      if (__any_sync(kFull, f) && lane == 0) ++my_fail;
    }
    if (a.stats && lane == 0) {
      vibe_shot_stats st;
      st.status = VIBE_STATUS_OK; st.lsd_invoked = 0; st.n_converged = (uint8_t)M; st.chosen_member = 0;
      st.iters = 1; st.largest_cluster = 0; st.n_clusters = 0;
      a.stats[shot] = st;
    }
    return;
  }

  // candidate list, lane j holds entry j (sorted by iteration, then member)
  int ncand = 0;
  int c_t = 0, c_i = 0, c_slot = 0;
  float c_W = 0.0f;

  for (int i = 0; i < K; ++i) {
    const int budget = ncand < M ? T : __shfl_sync(kFull, c_t, M - 1) - 1;
    if (budget <= 0) break;
    ImageRun R{budget, a.want_soft != 0, ncand == 0, nullptr, lpost, st, 0};
    const int conv = run_member<MT, DP, NCH>(t, i, smem_off, R);
    my_iters += (unsigned long long)R.ran;
    if (conv) {
      // insert (conv, i); i exceeds every member already listed, so it goes after equal iterations
      const int p = __popc(__ballot_sync(kFull, lane < ncand && c_t <= conv));
      const int slot = ncand < M ? ncand : __shfl_sync(kFull, c_slot, M - 1);
      const float W = member_bits(t, i, base, st, cand + (size_t)slot * nw, lane);
      if (a.want_soft) {
        float* dst = cand_post + (size_t)slot * n;
        for (int v = lane; v < n; v += 32) dst[v] = lpost[v];
      }
      const float uW = __shfl_up_sync(kFull, c_W, 1);
      const int ut = __shfl_up_sync(kFull, c_t, 1), ui = __shfl_up_sync(kFull, c_i, 1);
      const int us = __shfl_up_sync(kFull, c_slot, 1);
      const int last = min(ncand, M - 1);
      if (lane > p && lane <= last) { c_W = uW; c_t = ut; c_i = ui; c_slot = us; }
      if (lane == p) { c_W = W; c_t = conv; c_i = i; c_slot = slot; }
      ncand = min(ncand + 1, M);
      __syncwarp();
    } else if (ncand == 0) {
      // not converged after T sweeps and no candidate yet: add LLR^i / ||LLR^i|| (finite entries)
      float part = 0.0f;
      for (int v = lane; v < n; v += 32) {
        const float x = lpost[v];
        part = __fadd_rn(part, is_finite_bits(x) ? __fmul_rn(x, x) : 0.0f);
      }
#pragma unroll
      for (int off = 16; off >= 1; off >>= 1) part = __fadd_rn(part, __shfl_xor_sync(kFull, part, off));
      const float nrm = __fsqrt_rn(part);
      for (int v = lane; v < n; v += 32) {
        const float x = lpost[v];
        const float term = is_finite_bits(x) ? (nrm == 0.0f ? 0.0f : __fdiv_rn(x, nrm)) : x;
        acc[v] = __fadd_rn(i == 0 ? 0.0f : acc[v], term);
      }
    }
    __syncwarp();
  }

  if (ncand > 0) {
    // first minimum of W over the candidate list
    float bw = lane < ncand ? c_W : __int_as_float(0x7f800000);
    int bi = lane;
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) {
      const float ow = __shfl_xor_sync(kFull, bw, off);
      const int oi = __shfl_xor_sync(kFull, bi, off);
      if (ow < bw || (ow == bw && oi < bi)) { bw = ow; bi = oi; }
    }
    const int slot = __shfl_sync(kFull, c_slot, bi);
    const int member = __shfl_sync(kFull, c_i, bi);
    const int iters = ncand == M ? __shfl_sync(kFull, c_t, M - 1) : T;
    const uint32_t* bits = cand + (size_t)slot * nw;
    for (int w = lane; w < nw; w += 32) out_corr[w] = bits[w];
    if (a.want_soft) {
      const float* src = cand_post + (size_t)slot * n;
      float* dst = a.soft + (size_t)shot * a.soft_stride;
      for (int v = lane; v < n; v += 32) dst[v] = src[v];
    }
    uint32_t fail = 0;
    for (int rb = 0; rb < kw; ++rb) {
      const int r = 32 * rb + lane;
      uint32_t par = 0;
      if (r < t.k)
        for (int e = __ldg(t.lrowptr + r); e < __ldg(t.lrowptr + r + 1); ++e) {
          const int j = __ldg(t.lcolidx + e);
          par ^= (bits[j >> 5] >> (j & 31)) & 1u;
        }
      const uint32_t word = __ballot_sync(kFull, par != 0);
      if (a.logical && lane == 0) a.logical[(size_t)shot * a.log_stride + rb] = word;
      if (a.obs) fail |= word ^ a.obs[(size_t)shot * a.log_stride + rb];
    }
    if (fail && lane == 0) ++my_fail;
    if (a.stats && lane == 0) {
      vibe_shot_stats st;
      st.status = VIBE_STATUS_OK; st.lsd_invoked = 0; st.n_converged = (uint8_t)ncand;
      st.chosen_member = (uint8_t)member; st.iters = (uint16_t)iters; st.largest_cluster = 0; st.n_clusters = 0;
      a.stats[shot] = st;
    }
  } else {
    // hand the averaged soft vector to the LSD kernel
    uint32_t q = 0;
    if (lane == 0) q = atomicAdd(a.lsd_count, 1u);
    q = __shfl_sync(kFull, q, 0);
    if (lane == 0) a.lsd_shots[q] = a.lsd_shot_base + shot;
    float* dst = a.lsd_soft + (size_t)q * a.bnd.n;
    const float kf = (float)K;
    for (int v = lane; v < n; v += 32) dst[v] = __fdiv_rn(acc[v], kf);
  }
  __syncwarp();
}

// Pair mode: member i of shot `shot` (slot `slot` of the chunk) with one warp; the last member of the
// shot to finish writes the shot's outcome (pair_epilogue, vibe_internal.cuh).
template <typename MT, int DP, int NCH>
__device__ __forceinline__ void decode_pair(const BpArgs& a, const Tables& t, uint32_t shot, int slot, int i,
                                            unsigned char* base, int smem_off, float* lpost, uint32_t* gst, int lane,
                                            unsigned long long& my_iters, unsigned long long& my_shots,
                                            unsigned long long& my_fail) {
  const int K = t.K, M = t.M, T = t.T, n = t.n, nw = t.nw, kw = t.kw;
  if (i >= K) return;
  uint32_t* st = t.off_st >= 0 ? reinterpret_cast<uint32_t*>(base + t.off_st) : gst;
  const bool any = load_syndrome(t, a.syn + (size_t)shot * a.syn_stride, reinterpret_cast<uint32_t*>(base + t.off_s), lane);
  if (!any && !a.want_soft) {
    // s = 0: every member converges in iteration 1 to e = 0; member 0 is chosen -- written by member 0
    if (i != 0) return;
    ++my_shots;
    for (int w = lane; w < nw; w += 32) a.corr[(size_t)shot * a.corr_stride + w] = 0u;
    if (a.logical)
      for (int w = lane; w < kw; w += 32) a.logical[(size_t)shot * a.log_stride + w] = 0u;
    if (a.obs) {
      uint32_t f = 0;
      for (int w = lane; w < kw; w += 32) f |= a.obs[(size_t)shot * a.log_stride + w];
      if (__any_sync(kFull, f) && lane == 0) ++my_fail;
    }
    if (a.stats && lane == 0) {
      vibe_shot_stats st;
      st.status = VIBE_STATUS_OK; st.lsd_invoked = 0; st.n_converged = (uint8_t)M; st.chosen_member = 0;
      st.iters = 1; st.largest_cluster = 0; st.n_clusters = 0;
      a.stats[shot] = st;
    }
    return;
  }
  if (i == 0) ++my_shots;
  int* conv = a.pconv + (size_t)slot * a.pair_K;
  ImageRun R{T, a.want_soft != 0, true, conv, lpost, st, 0};
  const int cv = run_member<MT, DP, NCH>(t, i, smem_off, R);
  my_iters += (unsigned long long)R.ran;
  const size_t rec = (size_t)slot * a.pair_K + i;
  if (cv) {
    // the correction's bits and W(e)
    uint32_t* bits = reinterpret_cast<uint32_t*>(base + t.off_cand);
    const float W = member_bits(t, i, base, st, bits, lane);
    for (int w = lane; w < nw; w += 32) a.pbits[rec * a.bnd.nw + w] = bits[w];
    if (lane == 0) a.pW[rec] = W;
    if (a.want_soft)
      for (int v = lane; v < n; v += 32) a.ppost[rec * a.bnd.n + v] = lpost[v];
    __threadfence();
    __syncwarp();
    if (lane == 0) *reinterpret_cast<volatile int*>(conv + i) = cv;
  } else if (R.ran == T) {
    llr_term_add(lpost, a.pterms + rec * a.bnd.n, n, true, lane);
  }
  __syncwarp();
  if (pair_finish(a.pdone + slot, K, lane) && pair_epilogue(a, t, shot, slot, lane) && lane == 0) ++my_fail;
  __syncwarp();
}

// MIXED: the shots of the launch name their problems (dem_of_shot); the problems' descriptors are
// copied to shared memory after the warps' regions. Otherwise every shot decodes a.one, which the
// kernel reads from its parameter space.
template <typename MT, int DP, int NCH, bool MIXED>
__global__ void __launch_bounds__(kBpWarpsPerCta * 32, MinBlocks<MT, DP>::value) k_bp(const __grid_constant__ BpArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31;
  const int wcta = threadIdx.x >> 5;
  const long long gw = (long long)blockIdx.x * kBpWarpsPerCta + wcta;
  Tables* sdem = reinterpret_cast<Tables*>(smem + (size_t)kBpWarpsPerCta * a.bnd.warp_smem);
  if (MIXED) {
    const uint32_t* src = reinterpret_cast<const uint32_t*>(a.dems);
    uint32_t* dst = reinterpret_cast<uint32_t*>(sdem);
    const int words = a.ndem * (int)(sizeof(Tables) / 4);
    for (int q = threadIdx.x; q < words; q += blockDim.x) dst[q] = __ldg(src + q);
    __syncthreads();
  }
  const int smem_off = wcta * a.bnd.warp_smem;
  unsigned char* base = smem + smem_off;
  float* acc = a.scratch + gw * a.scratch_pitch;  // n floats: LLR average accumulator
  float* lpost = acc + a.bnd.n;                    // n floats: the member's posterior when needed
  uint32_t* gst = reinterpret_cast<uint32_t*>(lpost + a.bnd.n);   // n words with bnd.global_st: decision words
  float* cand_post = lpost + (a.bnd.global_st ? 2 : 1) * (size_t)a.bnd.n;   // M * n floats (only with want_soft)
  unsigned long long my_iters = 0, my_shots = 0, my_fail = 0;

  if (a.pair_mode) {
    const unsigned long long npairs = (unsigned long long)a.nshots * (unsigned long long)a.pair_K;
    for (;;) {
      unsigned long long q = 0;
      if (lane == 0) q = atomicAdd(a.next_pair, 1u);
      q = __shfl_sync(kFull, q, 0);
      if (q >= npairs) break;
      const uint32_t shot = (uint32_t)(q / a.pair_K);
      const int i = (int)(q % a.pair_K);
      if (MIXED) {
        const int di = __ldg(a.dem_of_shot + shot);
        if ((unsigned)di >= (unsigned)a.ndem) {
          if (i != 0 || !a.flag_bad) continue;
          for (int w = lane; w < a.corr_stride; w += 32) a.corr[(size_t)shot * a.corr_stride + w] = 0u;
          if (a.logical)
            for (int w = lane; w < a.log_stride; w += 32) a.logical[(size_t)shot * a.log_stride + w] = 0u;
          if (a.stats && lane == 0) {
            vibe_shot_stats st;
            st.status = VIBE_STATUS_BAD_PROBLEM; st.lsd_invoked = 0; st.n_converged = 0; st.chosen_member = 0;
            st.iters = 0; st.largest_cluster = 0; st.n_clusters = 0;
            a.stats[shot] = st;
          }
          if (a.counters && lane == 0) atomicAdd(a.counters + VIBE_CNT_BAD_PROBLEM, 1ull);
          continue;
        }
        if (sdem[di].engine != VIBE_ENGINE_IMAGE) continue;   // left to the summary engine
        decode_pair<MT, DP, NCH>(a, sdem[di], shot, (int)shot, i, base, smem_off, lpost, gst, lane, my_iters, my_shots, my_fail);
      } else {
        decode_pair<MT, DP, NCH>(a, a.one, shot, (int)shot, i, base, smem_off, lpost, gst, lane, my_iters, my_shots, my_fail);
      }
    }
  }
  for (;;) {
    if (a.pair_mode) break;
    uint32_t shot = 0;
    if (lane == 0) shot = atomicAdd(a.next_shot, 1u);
    shot = __shfl_sync(kFull, shot, 0);
    if (shot >= a.nshots) break;
    if (MIXED) {
      const int di = __ldg(a.dem_of_shot + shot);
      if ((unsigned)di >= (unsigned)a.ndem) {
        if (!a.flag_bad) continue;
        // problem index outside the launch's table: zero outputs, status BAD_PROBLEM, no decoding
        for (int w = lane; w < a.corr_stride; w += 32) a.corr[(size_t)shot * a.corr_stride + w] = 0u;
        if (a.logical)
          for (int w = lane; w < a.log_stride; w += 32) a.logical[(size_t)shot * a.log_stride + w] = 0u;
        if (a.soft)
          for (int j = lane; j < a.soft_stride; j += 32) a.soft[(size_t)shot * a.soft_stride + j] = 0.0f;
        if (a.stats && lane == 0) {
          vibe_shot_stats st;
          st.status = VIBE_STATUS_BAD_PROBLEM; st.lsd_invoked = 0; st.n_converged = 0; st.chosen_member = 0;
          st.iters = 0; st.largest_cluster = 0; st.n_clusters = 0;
          a.stats[shot] = st;
        }
        if (a.counters && lane == 0) atomicAdd(a.counters + VIBE_CNT_BAD_PROBLEM, 1ull);
        continue;
      }
      if (sdem[di].engine != VIBE_ENGINE_IMAGE) continue;   // left to the summary engine
      decode_shot<MT, DP, NCH>(a, sdem[di], shot, base, smem_off, acc, lpost, cand_post, gst, lane, my_iters, my_shots,
                                     my_fail);
    } else {
      decode_shot<MT, DP, NCH>(a, a.one, shot, base, smem_off, acc, lpost, cand_post, gst, lane, my_iters, my_shots,
                                      my_fail);
    }
  }
  if (lane == 0 && a.counters) {
    atomicAdd(a.counters + VIBE_CNT_SHOTS, my_shots);
    atomicAdd(a.counters + VIBE_CNT_PAIR_ITERS, my_iters);
    if (my_fail) atomicAdd(a.counters + VIBE_CNT_FAILURES, my_fail);
  }
}

// 16-byte chunks of a row when every problem of the launch has the same 1 to 4, else 0 (read per problem).
inline int nch_of(const Bounds& b, int spc) {
  const int c = b.RP / spc;
  return b.RP > 0 && c <= 4 ? c : 0;
}

inline size_t align16(size_t x) { return (x + 15) & ~(size_t)15; }

template <typename MT, int DP, int NCH, bool MIXED>
cudaError_t launch_one(const BpArgs& a, int grid, size_t smem, cudaStream_t s) {
  cudaError_t err = ensure_dyn_smem<k_bp<MT, DP, NCH, MIXED>>(smem);
  if (err != cudaSuccess) return err;
  k_bp<MT, DP, NCH, MIXED><<<grid, kBpWarpsPerCta * 32, smem, s>>>(a);
  return cudaGetLastError();
}

template <typename MT, int DP, int NCH, bool MIXED>
cudaError_t occupancy_one(size_t smem, int* out) {
  cudaError_t err = ensure_dyn_smem<k_bp<MT, DP, NCH, MIXED>>(smem);
  if (err != cudaSuccess) return err;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, k_bp<MT, DP, NCH, MIXED>, kBpWarpsPerCta * 32, smem);
}

template <typename Fn>
cudaError_t by_nch(int nch, Fn&& f) {
  switch (nch) {
    case 1: return f(std::integral_constant<int, 1>{});
    case 2: return f(std::integral_constant<int, 2>{});
    case 3: return f(std::integral_constant<int, 3>{});
    case 4: return f(std::integral_constant<int, 4>{});
    default: return f(std::integral_constant<int, 0>{});
  }
}

template <typename Fn>
cudaError_t by_dp(int DP, Fn&& f) {
  switch (DP) {
    case 3: return f(std::integral_constant<int, 3>{});
    case 4: return f(std::integral_constant<int, 4>{});
    case 8: return f(std::integral_constant<int, 8>{});
    case 16: return f(std::integral_constant<int, 16>{});
    case 32: return f(std::integral_constant<int, 32>{});
    default: return cudaErrorInvalidValue;
  }
}

// Mixed launches use the generic row scan (NCH 0) only, which keeps the number of instantiations down.
template <typename MT>
cudaError_t launch_mt(const BpArgs& a, int grid, cudaStream_t s) {
  const bool mixed = a.dem_of_shot != nullptr;
  const size_t smem = bp_cta_smem_bytes(a.bnd, mixed ? a.ndem : 0);
  return by_dp(a.bnd.CD, [&](auto dp) {
    if (mixed) return launch_one<MT, decltype(dp)::value, 0, true>(a, grid, smem, s);
    return by_nch(nch_of(a.bnd, Msg<MT>::kSpc), [&](auto nch) {
      return launch_one<MT, decltype(dp)::value, decltype(nch)::value, false>(a, grid, smem, s);
    });
  });
}

template <typename MT>
cudaError_t occupancy_mt(const Bounds& b, int ndem, int* out) {
  const size_t smem = bp_cta_smem_bytes(b, ndem);
  return by_dp(b.CD, [&](auto dp) {
    if (ndem > 0) return occupancy_one<MT, decltype(dp)::value, 0, true>(smem, out);
    return by_nch(nch_of(b, Msg<MT>::kSpc), [&](auto nch) {
      return occupancy_one<MT, decltype(dp)::value, decltype(nch)::value, false>(smem, out);
    });
  });
}

}  // namespace

size_t bp_warp_smem_bytes(Tables* t, int msg_fp16) {
  const size_t words = 4 * (size_t)t->mw, dec = ((size_t)t->n + 3) / 4 * 4, steps = 4 * (size_t)t->nstep;
  const bool bytes = t->n_flood > 0 || t->n_layered > 0;   // these members keep a byte per decision
  size_t o = 0;
  t->off_msg = (int)o;
  o = align16(o + (size_t)t->m * t->RP * (msg_fp16 ? 2 : 4));
  t->off_s = (int)o;
  o = align16(o + words);
  t->off_par = (int)o;
  o = align16(o + words);
  // decision bytes and step words share their place: a member uses one of them. The words of a graph of
  // long chains (few columns per step) go to global scratch where they would take the state beyond that of a
  // byte per decision, per syndrome bit and per parity (which bounds the problems the engine takes).
  t->off_dec = t->off_st = (int)o;
  const size_t bytes3 = align16(dec) + 2 * align16(((size_t)t->m + 3) / 4 * 4);
  size_t d = bytes ? dec : 0;
  if (steps <= bytes3 - 2 * align16(words)) d = std::max(d, steps);
  else t->off_st = -1;
  o = align16(o + d);
  t->off_cand = (int)o;
  o = align16(o + (size_t)t->M * t->nw * 4);
  t->off_cv = -1;
  if (t->n_layered > 0 || (t->n_flood > 0 && msg_fp16)) {
    t->off_cv = (int)o;
    o = align16(o + (size_t)t->m * t->RP * 4);
  }
  t->warp_smem = (int)o;
  return o;
}

size_t bp_cta_smem_bytes(const Bounds& b, int ndem) {
  return (size_t)kBpWarpsPerCta * b.warp_smem + align16((size_t)ndem * sizeof(Tables));
}

cudaError_t launch_bp(const BpArgs& a, int msg_fp16, int grid, cudaStream_t s) {
  return msg_fp16 ? launch_mt<__half>(a, grid, s) : launch_mt<float>(a, grid, s);
}

cudaError_t bp_occupancy(const Bounds& b, int ndem, int msg_fp16, int* blocks_per_sm) {
  return msg_fp16 ? occupancy_mt<__half>(b, ndem, blocks_per_sm) : occupancy_mt<float>(b, ndem, blocks_per_sm);
}

}  // namespace vibe

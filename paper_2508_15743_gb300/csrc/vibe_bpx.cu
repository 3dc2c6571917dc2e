// K1' -- the BP ensemble for problems whose message image does not fit in shared memory (circuit-level
// detector error models: rows of 100-200 entries, E up to ~4e5): the summary engine. Same method, same
// results as the image engine (vibe_bp.cu), which keeps a member's whole message image in shared
// memory; a different layout.
//
// Mapping: one warp, or for wide graphs in batches that do not fill the GPU a team of 8 (a CTA either way), per
// (shot, member), one lane per edge. A sweep runs the member's steps (k_steps in vibe_graph.cu): up to 32 edges per
// warp of columns that share no check, packed in the member's order. A lane asks its check's summary for the
// check-to-variable message of its edge,
// the lanes of a column pass each other these messages with shuffles, and every lane forms its own
// exclusion sum and updates its own check. A team takes a unit of as many steps as it has warps at a
// time, no two of which share a check, with a barrier after each unit. In shot mode each team decodes one
// shot at a time (persistent, shots from a global counter), running the members one after another with
// the iteration budget of the correction limit (Sec. III.D.2); in pair mode each team takes one (shot,
// member) pair at a time, and the last member of a shot to finish runs the shot's selection and
// epilogue. The first warp of a team runs that control flow and calls the others for each member.
//
// Check-node state: a summary per check in shared memory.
//   m1 <= m2  the magnitudes of up to two "holder" edges of the row, with their positions p1, p2 inside
//             the check's CSR row; an empty holder is position 255 with +inf
//   F         a floor: every entry of the row that is not a holder has magnitude >= F, and the holders'
//             magnitudes are <= F (after a rescan, F is the third smallest magnitude, or +inf)
//   flags     the parity of the sign bits of the row's messages XOR the syndrome bit (bit 31 of the flag
//             word), and the check's parity (H e)_c XOR s_c (bit 30).
// The minimum over the row without the edge at position p is m2 if p == p1, else m1 -- unless that
// value exceeds F, which only an empty holder's +inf above a finite floor does: then the row is
// rescanned first -- lazily, only when a column actually needs the answer. The sign product without p,
// syndrome included, is the flag XOR the sign of p's own message. Together these are exactly the
// minimum and sign product that Algorithm 1's check update takes over N(c) \ v.
//
// Keeping the summary exact after the edge at position p gets the new magnitude x: p leaves the
// holders if it is one; then, if x <= F, (x, p) is inserted into the sorted pair of holders and the value
// that falls out, if any, becomes the floor (it is <= F). With the floor most holders that grow stay
// answerable; on circuit-level colour codes this needs ~2.5x fewer row rescans per sweep than two
// holders without a floor (117 vs 296 at d=11).
//
// Messages. A member's variable-to-check messages live in the warp's global scratch in step order: a
// step's messages are contiguous, so its stores coalesce. A step never reads its old messages: it needs
// only their signs, kept with the columns' previous decisions as two 32-bit words per step (bit l: lane
// l's edge; the decision on the lane of the column's last edge). Messages are read only by rescans,
// through a per-member map from each CSR entry of H to its message slot.
//
// What bounds it and what the mapping bought. A sweep is a dependent chain of steps (summary, shuffles, sums,
// update, next step); in a member's first sweeps, which rescan most, the rescans' message rows come on top: on
// circuit-level d=11 (1672 members of 10 sweeps in flight, 565 rescans a sweep) issue is active 22 % of the time, the
// long scoreboard is the main stall and DRAM runs at 39 % of its peak, 10.2 MB a sweep for 1.1 MB of messages. The
// mapping it replaces gave each lane a whole column and unrolled its checks: on levels of 4-30 columns most
// lanes idled (88.4 G warp instructions for that launch, 52.2 G now: 191 a step, rescans included); a step of 32
// edges has nearly every lane at work (31.2 lanes an instruction).
// Measured (GB300), column / edge per lane, one warp per shot: circuit-level d=5, K=8, T=20, 100,000 shots FP32 1898
// / 491 ms, FP16 2313 / 512; d=9, 6000 shots 1087 / 619 and 1235 / 603. As pairs: d=11, FP32, K=64, T=50, 32 shots 223 / 153.
//
// Arithmetic equals the oracle's bit for bit: same per-node operation order (__fadd_rn/__fmul_rn), min
// and sign exact, FP16 storage with -0 stored as +0.
#include <cstddef>
#include <type_traits>

#include "vibe_internal.cuh"

namespace vibe {
namespace {

// Stored messages as bits: the rounding of a sum, its sign bit at bit 31, loads and stores.
template <typename MT>
struct XMsg;

template <>
struct XMsg<float> {
  __device__ __forceinline__ static uint32_t round(float x) { return __float_as_uint(x); }
  __device__ __forceinline__ static uint32_t sign31(uint32_t b) { return b; }
  __device__ __forceinline__ static uint32_t load(const float* p) { return __float_as_uint(__ldcg(p)); }
  __device__ __forceinline__ static void store(float* p, uint32_t b) { __stcs(p, __uint_as_float(b)); }
};

template <>
struct XMsg<__half> {
  __device__ __forceinline__ static uint32_t round(float x) {   // -0 as +0
    const uint32_t h = (uint32_t)__half_as_ushort(__float2half_rn(x));
    return h == 0x8000u ? 0u : h;
  }
  __device__ __forceinline__ static uint32_t sign31(uint32_t b) { return b << 16; }
  __device__ __forceinline__ static uint32_t load(const __half* p) {
    return (uint32_t)__ldcg(reinterpret_cast<const unsigned short*>(p));
  }
  __device__ __forceinline__ static void store(__half* p, uint32_t b) {
    __stcs(reinterpret_cast<unsigned short*>(p), (unsigned short)b);
  }
};


constexpr uint32_t kSgnBit = 1u << 31, kParBit = 1u << 30;   // flags of a summary

// What a lane sees of its check: `ans`, the minimum magnitude of the row without the lane's edge;
// `ok`, whether the summary holds it; `flags`. A check is addressed by its summary's shared address, an
// edge by its record word (position in the row in bits 0-7).
// Sum<float>: 16 bytes per check {m1, m2, F, p1 | p2 << 8 | flags}.
// Sum<__half>: 8 bytes. Magnitudes are binary16 (exact: those of stored binary16 messages) and a holder
// is one 23-bit key, magnitude << 8 | position, so that an integer comparison orders holders by
// magnitude, then position. x: key 1 | low 9 bits of F << 23; y: high 6 bits of F | key 2 << 6 | flags.
template <typename MT>
struct Sum;

template <>
struct Sum<float> {
  static constexpr int kBytes = 16;
  float m1, m2, F;
  uint32_t w;
  bool is1;
  __device__ __forceinline__ void load(uint32_t addr, uint32_t rec) {
    const uint4 q = lds128(addr);
    m1 = __uint_as_float(q.x);
    m2 = __uint_as_float(q.y);
    F = __uint_as_float(q.z);
    w = q.w;
    is1 = ((w ^ rec) & 0xffu) == 0u;
  }
  __device__ __forceinline__ float ans() const { return is1 ? m2 : m1; }
  __device__ __forceinline__ bool ok() const { return ans() <= F; }
  __device__ __forceinline__ uint32_t flags() const { return w; }
  // the edge takes the message with bits b; `toggle` flips flag bits. Stores only what changed.
  __device__ __forceinline__ void update(uint32_t addr, uint32_t rec, uint32_t b, uint32_t toggle, bool act) const {
    const float inf = __uint_as_float(kInfBits);
    const float x = fabsf(__uint_as_float(b));
    const uint32_t p1 = w & 0xffu, p2 = (w >> 8) & 0xffu;
    const bool was = is1 || ((p2 ^ rec) & 0xffu) == 0u, ins = x <= F;
    const float b1 = ans(), b2 = was ? inf : m2;
    const uint32_t c1 = is1 ? p2 : p1, c2 = was ? 255u : p2;
    const float y = ins ? x : inf;
    const uint32_t py = ins ? (rec & 0xffu) : 255u;
    const bool lt1 = y < b1;
    const float n1 = fminf(y, b1), t = fmaxf(y, b1);
    const uint32_t r1 = lt1 ? py : c1, tp = lt1 ? c1 : py;
    const bool lt2 = t < b2;
    const float n2 = fminf(t, b2), h = fmaxf(t, b2);
    const uint32_t r2 = lt2 ? tp : c2;
    if (act && (was || ins || toggle))
      sts128(addr, make_uint4(__float_as_uint(n1), __float_as_uint(n2), __float_as_uint(fminf(F, h)),
                              ((w ^ toggle) & 0xffff0000u) | r1 | (r2 << 8)));
  }
  __device__ __forceinline__ static void init(uint32_t addr, float4 s, uint32_t flip) {
    sts128(addr, make_uint4(__float_as_uint(s.x), __float_as_uint(s.y), __float_as_uint(s.z), __float_as_uint(s.w) ^ flip));
  }
  // a message as the rescan orders it: the bits of its magnitude (unsigned order of non-negative floats)
  __device__ __forceinline__ static uint32_t key(uint32_t b, uint32_t) { return b & 0x7fffffffu; }
  static constexpr uint32_t kNone = kInfBits;
  __device__ __forceinline__ static void rescanned(uint32_t addr, uint32_t k1, uint32_t k2, uint32_t k3, uint32_t p1,
                                                   uint32_t p2) {
    sts128(addr, make_uint4(k1, k2, k3, (lds32(addr + 12) & 0xffff0000u) | p1 | (p2 << 8)));
  }
};

template <>
struct Sum<__half> {
  static constexpr int kBytes = 8;
  static constexpr uint32_t kEmpty = 0x7c00ffu;   // +inf at position 255
  static constexpr uint32_t kKey = 0x7fffffu;
  uint2 q;
  uint32_t k1, k2, F;
  bool is1;
  __device__ __forceinline__ void load(uint32_t addr, uint32_t rec) {
    q = lds64(addr);
    k1 = q.x & kKey;
    k2 = (q.y >> 6) & kKey;
    F = __funnelshift_r(q.x, q.y, 23) & 0x7fffu;
    is1 = ((q.x ^ rec) & 0xffu) == 0u;
  }
  __device__ __forceinline__ uint32_t akey() const { return is1 ? k2 : k1; }
  __device__ __forceinline__ float ans() const { return __half2float(__ushort_as_half((unsigned short)(akey() >> 8))); }
  __device__ __forceinline__ bool ok() const { return (akey() >> 8) <= F; }
  __device__ __forceinline__ uint32_t flags() const { return q.y; }
  __device__ __forceinline__ static uint2 pack(uint32_t k1, uint32_t k2, uint32_t F, uint32_t flags) {
    return make_uint2(k1 | (F << 23), (F >> 9) | (k2 << 6) | flags);
  }
  __device__ __forceinline__ void update(uint32_t addr, uint32_t rec, uint32_t b, uint32_t toggle, bool act) const {
    const uint32_t xh = b & 0x7fffu;
    const bool was = is1 || ((k2 ^ rec) & 0xffu) == 0u, ins = xh <= F;
    const uint32_t b1 = akey(), b2 = was ? kEmpty : k2;
    const uint32_t y = ins ? __byte_perm(xh, rec, 0x3104) : kEmpty;   // magnitude << 8 | position
    const uint32_t t = max(y, b1), h = max(t, b2);
    if (act && (was || ins || toggle))
      sts64(addr, pack(min(y, b1), min(t, b2), min(F, h >> 8), (q.y ^ toggle) & (kSgnBit | kParBit)));
  }
  __device__ __forceinline__ static void init(uint32_t addr, float4 s, uint32_t flip) {
    const uint32_t w = __float_as_uint(s.w);
    sts64(addr, pack(((uint32_t)__half_as_ushort(__float2half_rn(s.x)) << 8) | (w & 0xffu),
                     ((uint32_t)__half_as_ushort(__float2half_rn(s.y)) << 8) | ((w >> 8) & 0xffu),
                     (uint32_t)__half_as_ushort(__float2half_rn(s.z)), (w & kSgnBit) ^ flip));
  }
  __device__ __forceinline__ static uint32_t key(uint32_t b, uint32_t pos) { return ((b & 0x7fffu) << 8) | pos; }
  static constexpr uint32_t kNone = kEmpty;
  __device__ __forceinline__ static void rescanned(uint32_t addr, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t,
                                                   uint32_t) {
    sts64(addr, pack(a1, a2, a3 >> 8, lds32(addr + 4) & (kSgnBit | kParBit)));
  }
};

// Warp-cooperative rescan of the check with summary `addr`, whose CSR row is b .. b + d: the two smallest magnitudes with
// their positions and the third smallest as the floor; the flags are kept. Each lane keeps the three
// smallest of its entries; the warp minimum is then taken three times, its owner dropping its entry.
// NaN messages (sums of +inf and -inf) are no candidates.
template <typename MT>
__device__ __forceinline__ void rescan_row(uint32_t addr, int b, int d, const uint32_t* rmap, const MT* msg, int lane) {
  uint32_t loc[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int q = lane + 32 * u;
    loc[u] = q < d ? __ldg(rmap + b + q) : 0u;
  }
  uint32_t a1 = Sum<MT>::kNone, a2 = a1, a3 = a1, p1 = 255u, p2 = 255u;
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int q = lane + 32 * u;
    if (32 * u < d) {
      const uint32_t k = q < d ? Sum<MT>::key(XMsg<MT>::load(msg + loc[u]), (uint32_t)q) : 0xffffffffu;
      const bool b1 = k < a1, b2 = k < a2;
      a3 = b2 ? a2 : min(a3, k);
      a2 = b1 ? a1 : (b2 ? k : a2);
      p2 = b1 ? p1 : (b2 ? (uint32_t)q : p2);
      a1 = b1 ? k : a1;
      p1 = b1 ? (uint32_t)q : p1;
    }
  }
  const uint32_t r1 = __reduce_min_sync(kFull, a1);
  const int o1 = __ffs(__ballot_sync(kFull, a1 == r1)) - 1;
  const uint32_t f1 = __shfl_sync(kFull, p1, o1);
  if (lane == o1) { a1 = a2; p1 = p2; a2 = a3; p2 = 255u; }
  const uint32_t r2 = __reduce_min_sync(kFull, a1);
  const int o2 = __ffs(__ballot_sync(kFull, a1 == r2)) - 1;
  const uint32_t f2 = __shfl_sync(kFull, p1, o2);
  if (lane == o2) a1 = a2;
  const uint32_t r3 = __reduce_min_sync(kFull, a1);
  if (lane == 0) Sum<MT>::rescanned(addr, r1, r2, r3, f1, f2);
}

// What a warp's steps near the current one need: a window in shared memory. Its first 32 entries of 16
// bytes are (signs, decisions, first slot of the step, end of its slots) of the warp's current block of
// 32 steps, read by all lanes of a step at once. Then two buffers of edge records, which come in chunks of
// four steps by cp.async, one chunk ahead, and two of their links. (Two steps per chunk cost 6 % and are
// taken only where the window would not fit beside the summaries.) A chunk is copied in groups of four
// slots.
constexpr int kChunk = kStepChunk;

__host__ __device__ constexpr uint32_t chunk_slots(int chunk) { return (uint32_t)chunk * 32u + 8u; }
__host__ __device__ constexpr uint32_t rec_at(int chunk, int buf) { return 512u + (uint32_t)buf * chunk_slots(chunk) * 8u; }
__host__ __device__ constexpr uint32_t lnk_at(int chunk, int buf) {
  return 512u + 2u * chunk_slots(chunk) * 8u + (uint32_t)buf * chunk_slots(chunk) * 4u;
}
__host__ __device__ constexpr uint32_t window_bytes(int chunk) { return lnk_at(chunk, 2); }
static_assert(window_bytes(4) % 16 == 0 && window_bytes(2) % 16 == 0, "cp.async blocks are 16 bytes");

// What the first warp of a team tells the others, and their common sums. It precedes the windows of the
// team's warps in shared memory; the check summaries follow them.
struct alignas(16) TeamCmd {
  const Tables* t;
  const uint32_t* syn;
  const int* conv;
  int go, i, nsyn, budget, soft, keep_last, K, M;
  int stop;
  int sum[kTeam];
};

__device__ __forceinline__ void team_sync(int W) {
  if (W == 1) __syncwarp();
  else __syncthreads();
}

__device__ __forceinline__ void cp_async_cg16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Copies the records of slots [sb, se) of a member into buffer `buf` (one commit group; none if empty).
// win: shared address of the warp's window; first: the member's first slot in the tables.
__device__ __forceinline__ void fetch_chunk(uint32_t win, int chunk, int buf, uint32_t sb, uint32_t se, const uint2* rec,
                                            const uint32_t* lnk, size_t first, int lane) {
  const size_t b = (first + sb) & ~(size_t)3, e = first + se;
  const uint32_t dr = win + rec_at(chunk, buf), dl = win + lnk_at(chunk, buf);
  const int quads = se > sb ? (int)((e - b + 3) >> 2) : 0;
  for (int q = lane; q < quads; q += 32) {
    cp_async_cg16(dr + 32 * q, rec + b + 4 * q);
    cp_async_cg16(dr + 32 * q + 16, rec + b + 4 * q + 2);
    cp_async_cg16(dl + 16 * q, lnk + b + 4 * q);
  }
  cp_async_commit();
}

// One sweep of a member over its ns steps by warp w of a team of W. Of every kChunk * W consecutive steps
// the warp has the kChunk from kChunk * w on; the j-th steps of all warps form a unit. win: shared address of the
// warp's window; sums: of the summaries; stg: (signs, decisions) of every step in global scratch; LP: the
// posteriors go to lp. Returns the lane's change of the number of unsatisfied checks.
template <typename MT, int DP, bool LP, int chunk>
__device__ __forceinline__ int sweep_x(const Tables& t, const uint32_t* soff, const int ns, const size_t first,
                                       const uint32_t* rmap, const float alpha, const uint32_t win, const uint32_t sums,
                                       MT* msg, uint2* stg, float* lp, uint32_t& rescans, const int lane, const int W,
                                       const int w) {
  const uint2* trec = t.xrec;
  const uint32_t* tlnk = t.xlnk;
  const int32_t* rowptr = t.rowptr;
  const int J = ns / W;   // the warp's steps (with W > 1 ns is a multiple of kChunk * W)
  int dpar = 0;
  auto place = [&](int j) { return j / kChunk * kChunk * W + kChunk * w + j % kChunk; };
  auto entry = [&](int j) {
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (j < J) {
      const int q = place(j);
      const uint2 x = stg[q];
      v = make_uint4(x.x, x.y, __ldg(soff + q), __ldg(soff + q + 1));
    }
    return v;
  };
  uint4 cur = entry(lane), nxt = cur;
  int buf = 0;
  for (int j0 = 0; j0 < J; j0 += 32) {
    // block of 32 of the warp's steps
    sts128(win + 16 * lane, cur);
    __syncwarp();
    if (j0 == 0) fetch_chunk(win, chunk, 0, lds32(win + 8), lds32(win + 16 * (min(chunk, J) - 1) + 12), trec, tlnk, first, lane);
    if (j0 + 32 < J) nxt = entry(j0 + 32 + lane);
    const int jb = min(32, J - j0);
    uint32_t wst = win;   // the step's window entry
    for (int j1 = 0; j1 < jb; j1 += chunk) {
      // this chunk's records are here, the last one's buffer is free
      cp_async_wait<0>();
      __syncwarp();
      {
        const int jn = j1 + chunk, left = J - j0 - jn;   // the next chunk and the steps from it on
        const int le = min(chunk, left) - 1;
        uint32_t sb = 0u, se = 0u;
        if (left > 0) {
          if (jn < 32) {
            sb = lds32(win + 16 * jn + 8);
            se = lds32(win + 16 * (jn + le) + 12);
          } else {
            sb = __shfl_sync(kFull, nxt.z, 0);
            se = __shfl_sync(kFull, nxt.w, le);
          }
        }
        fetch_chunk(win, chunk, buf ^ 1, sb, se, trec, tlnk, first, lane);
      }
      // addresses of slot 0's records if the buffer reached back that far
      const uint32_t o0 = lds32(wst + 8), sh = (((uint32_t)first + o0) & 3u) - o0;
      const uint32_t ra = win + rec_at(chunk, buf) + 8u * sh, la = win + lnk_at(chunk, buf) + 4u * sh;
      buf ^= 1;
#pragma unroll 1
      for (int u = 0; u < chunk; ++u) {   // steps past the last one have no edges
        const uint4 st = lds128(wst);
        const uint32_t ol = st.z + (uint32_t)lane;   // slot of the lane's edge
        uint2 r = make_uint2(0u, 0u);
        uint32_t ln = 0u;
        if (ol < st.w) {
          r = lds64(ra + 8u * ol);
          ln = lds32(la + 4u * ol);
        }
        const bool act = (int)ln < 0;
        // lanes without an edge read their own window (a check could be another warp's in this unit)
        const uint32_t sa = act ? sums + (r.x >> 18) * (uint32_t)Sum<MT>::kBytes : win;
        const uint32_t osg = st.x << (31 - lane);   // bit 31: sign of the edge's own old message
        Sum<MT> S;
        S.load(sa, r.x);
        uint32_t bal = __ballot_sync(kFull, act && !S.ok());
        if (bal) {
          // rescan every check whose summary could not answer (the checks of a step are distinct), ask again
          int rb = 0, rd = 0;
          if ((bal >> lane) & 1u) {
            rb = __ldg(rowptr + (r.x >> 18));
            rd = __ldg(rowptr + (r.x >> 18) + 1) - rb;
          }
          while (bal) {
            const int src = __ffs(bal) - 1;
            bal &= bal - 1u;
            rescan_row<MT>(__shfl_sync(kFull, sa, src), __shfl_sync(kFull, rb, src), __shfl_sync(kFull, rd, src), rmap,
                           msg, lane);
            ++rescans;
          }
          __syncwarp();
          S.load(sa, r.x);
        }
        // check-to-variable message (Algorithm 1's check update over N(c) \ v): sign parity, syndrome, own
        // sign; then the exclusion sum: lambda and the column's other messages in ascending check order
        const uint32_t mcv = __float_as_uint(__fmul_rn(alpha, S.ans())) ^ ((S.flags() ^ osg) & kSgnBit);
        float acc = __uint_as_float(r.y);
#pragma unroll
        for (int j = 0; j < DP; ++j)
          acc = add_if(acc, __uint_as_float(__shfl_sync(kFull, mcv, (int)ln + j)), ln & (32u << j));
        const float L = __fadd_rn(acc, __uint_as_float(mcv));   // on the last edge's lane: the posterior
        const uint32_t dec = __ballot_sync(kFull, (ln & kLnkLast) && L <= 0.0f);
        const uint32_t xb = XMsg<MT>::round(acc), xs = XMsg<MT>::sign31(xb);
        const uint32_t sg = __ballot_sync(kFull, (int)(xs & ln) < 0);
        if (act) XMsg<MT>::store(msg + ol, xb);   // streamed: read again only by rescans
        uint32_t toggle = (xs ^ osg) & kSgnBit;
        const uint32_t ch = dec ^ st.y;
        if (ch) {   // some column of the step changed its decision
          if (act && ((ch >> ((ln >> kLnkLastLane) & 31u)) & 1u)) {
            toggle |= kParBit;
            dpar += (S.flags() & kParBit) ? -1 : 1;
          }
        }
        S.update(sa, r.x, xb, toggle, act);
        if (lane == 0) sts64(wst, make_uint2(sg, dec));
        if (LP) {
          if (ln & kLnkLast) lp[__ldg(t.xcolid + first + ol)] = L;
          else if (ln == 0u && ol < st.w) lp[__ldg(t.xcolid + first + ol)] = __uint_as_float(r.y);   // no checks
        }
        wst += 16u;
        team_sync(W);
      }
    }
    if (j0 + lane < J) stg[place(j0 + lane)] = lds64(win + 16 * lane);
    __syncwarp();
    cur = nxt;
  }
  cp_async_wait<0>();
  return dpar;
}

// What a member's run is told and what it reports.
struct MemberRun {
  const uint32_t* syn;   // the shot's syndrome words
  int nsyn;              // its flipped checks
  int budget;            // sweeps at most
  bool soft, keep_last;  // the posterior after every sweep / after sweep T
  const int* conv;       // pair mode: the shot's converged members (pair_should_stop), else NULL
  int K, M;
  int chunk;             // steps per chunk of records
  // results
  int ran;               // sweeps run
  uint32_t rescans;
};

// One member (index i) on one shot: initialises the member's state and runs up to `budget` sweeps,
// stopping at the first that leaves H e = s, or in pair mode before a sweep that no longer counts.
// Returns the converging sweep (0 if none; its decisions are then in the warp's scratch, column order);
// leaves the posterior of the last sweep in the scratch when soft output is on or `keep_last` is set
// and the member reached sweep T. Called by all warps of the team (the block); gs: its global scratch.
// Not inlined: the sweep gets its own registers, whatever the caller keeps between members.
template <typename MT, int DP>
__device__ __noinline__ int run_member_x(const Tables& t, int i, MemberRun& R, unsigned char* gs) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = __shfl_sync(kFull, (int)(threadIdx.x & 31), (int)(threadIdx.x & 31));
  const int W = (int)(blockDim.x >> 5), w = __shfl_sync(kFull, (int)(threadIdx.x >> 5), lane);
  const int tid = 32 * w + lane, nt = 32 * W;
  TeamCmd* cmd = reinterpret_cast<TeamCmd*>(smem);
  const uint32_t wins = __shfl_sync(kFull, (uint32_t)__cvta_generic_to_shared(smem) + (uint32_t)sizeof(TeamCmd), lane);
  const uint32_t win = wins + (uint32_t)w * window_bytes(R.chunk);
  const uint32_t sums = wins + (uint32_t)W * window_bytes(R.chunk);
  const int m = t.m, T = t.T, nw = t.nw;
  MT* msg = reinterpret_cast<MT*>(gs + t.xg_msg);
  uint2* stg = reinterpret_cast<uint2*>(gs + t.xg_st);   // (signs, decisions) of every step
  const uint32_t* syn = R.syn;
  uint32_t rescans = 0;
  const size_t first = (size_t)i * t.SP;
  const uint32_t* colid = t.xcolid + first;
  const uint32_t* rmap = t.xrmap + (size_t)i * t.E;
  const uint32_t* soff = t.soff + (size_t)i * t.soff_pitch;
  const int ns = __ldg(t.stepcnt + i);
  // member init: prior summaries with this shot's syndrome (parity = s), prior messages in step order,
  // signs and decisions 0
  for (int c = tid; c < m; c += nt)
    Sum<MT>::init(sums + c * Sum<MT>::kBytes, __ldg(t.xsum + c),
                  ((__ldg(syn + (c >> 5)) >> (c & 31)) & 1u) ? (kSgnBit | kParBit) : 0u);
  for (int j = tid; j < t.SP; j += nt)
    XMsg<MT>::store(msg + j, XMsg<MT>::round(__uint_as_float(__ldg(&t.xrec[first + j].y))));
  for (int s = tid; s < ns; s += nt) stg[s] = make_uint2(0u, 0u);
  team_sync(W);
  const float alpha = __ldg(t.alpha_m + i);   // member i's scaling factor
  const int budget = R.budget;
  int unsat = R.nsyn;
  int conv = 0, ran = 0;
  for (int it = 1; it <= budget; ++it) {
    if (R.conv) {   // one answer for the team: other members converge meanwhile
      bool stop;
      if (W == 1) {
        stop = pair_should_stop(R.conv, R.K, R.M, i, it, lane);
      } else {
        if (w == 0) {
          stop = pair_should_stop(R.conv, R.K, R.M, i, it, lane);
          if (lane == 0) cmd->stop = stop;
        }
        __syncthreads();
        stop = cmd->stop != 0;
      }
      if (stop) break;
    }
    // the posterior is needed after the last possible sweep of a member that may end without
    // converging (LLR average) and, for soft output, after every sweep
    int dpar;
    float* lp = reinterpret_cast<float*>(gs + t.xg_lpost);
    auto sweep = [&](auto with_lp, auto chunk) {
      return sweep_x<MT, DP, decltype(with_lp)::value, decltype(chunk)::value>(t, soff, ns, first, rmap, alpha, win, sums,
                                                                              msg, stg, lp, rescans, lane, W, w);
    };
    const bool with_lp = R.soft || (it == T && R.keep_last);
    if (R.chunk == kChunk)
      dpar = with_lp ? sweep(std::true_type{}, std::integral_constant<int, kChunk>{})
                     : sweep(std::false_type{}, std::integral_constant<int, kChunk>{});
    else
      dpar = with_lp ? sweep(std::true_type{}, std::integral_constant<int, 2>{})
                     : sweep(std::false_type{}, std::integral_constant<int, 2>{});
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) dpar += __shfl_xor_sync(kFull, dpar, off);
    if (W > 1) {
      if (lane == 0) cmd->sum[w] = dpar;
      __syncthreads();
      dpar = 0;
      for (int q = 0; q < W; ++q) dpar += cmd->sum[q];
    }
    unsat += dpar;
    ran = it;
    if (unsat == 0) { conv = it; break; }
  }
  R.ran = ran;
  R.rescans = rescans;
  if (conv) {   // decisions in column order
    uint32_t* bits = reinterpret_cast<uint32_t*>(gs + t.xg_dec);
    for (int q = tid; q < nw; q += nt) __stcg(bits + q, 0u);
    team_sync(W);
    for (int s = tid; s < ns; s += nt) {
      uint32_t d = stg[s].y;
      const uint32_t o = __ldg(soff + s);
      while (d) {
        const uint32_t v = __ldg(colid + o + (uint32_t)__ffs(d) - 1u);
        atomicOr(bits + (v >> 5), 1u << (v & 31));
        d &= d - 1u;
      }
    }
  }
  team_sync(W);
  return conv;
}

// run_member_x by the team's first warp: hands the call to the others first.
template <typename MT, int DP>
__device__ __forceinline__ int team_member(const Tables& t, int i, MemberRun& R, unsigned char* gs) {
  extern __shared__ __align__(16) unsigned char smem[];
  if (blockDim.x > 32) {
    if (threadIdx.x == 0) {
      TeamCmd* c = reinterpret_cast<TeamCmd*>(smem);
      c->t = &t; c->syn = R.syn; c->conv = R.conv; c->go = 1; c->i = i; c->nsyn = R.nsyn; c->budget = R.budget;
      c->soft = R.soft; c->keep_last = R.keep_last; c->K = R.K; c->M = R.M;
    }
    __syncthreads();
  }
  return run_member_x<MT, DP>(t, i, R, gs);
}

// The other warps of a team: run members until the first warp is done. Returns the rescans they made.
template <typename MT, int DP>
__device__ __forceinline__ uint32_t team_serve(unsigned char* gs) {
  extern __shared__ __align__(16) unsigned char smem[];
  const TeamCmd* c = reinterpret_cast<const TeamCmd*>(smem);
  uint32_t rescans = 0;
  for (;;) {
    __syncthreads();
    if (!c->go) return rescans;
    MemberRun R{c->syn, c->nsyn, c->budget, c->soft != 0, c->keep_last != 0, c->conv, c->K, c->M, kChunk, 0, 0u};
    run_member_x<MT, DP>(*c->t, c->i, R, gs);
    rescans += R.rescans;
  }
}

// W(e) = sum of lambda_j over e_j = 1, ascending j, of the decisions in dec (every lane folds the same
// sequence); with bits != NULL the decision words are copied there.
__device__ __forceinline__ float decision_weight(const Tables& t, const uint32_t* dec, uint32_t* bits, int lane) {
  const int nw = t.nw;
  if (bits)
    for (int w = lane; w < nw; w += 32) bits[w] = __ldcg(dec + w);
  float W = 0.0f;
  for (int w = 0; w < nw; ++w) {
    uint32_t x = __ldcg(dec + w);
    while (x) {
      const int bpos = __ffs(x) - 1;
      W = __fadd_rn(W, __ldg(t.lam + 32 * w + bpos));
      x &= x - 1;
    }
  }
  return W;
}

// Decodes shot `shot` of problem t with the team, driven by its first warp. gs: the team's global
// scratch (messages, state words, decisions, posterior, LLR accumulator, candidate records).
template <typename MT, int DP>
__device__ __forceinline__ void decode_shot_x(const BpArgs& a, const Tables& t, uint32_t shot, unsigned char* gs, int lane,
                                              uint32_t& my_iters,
                                              uint32_t& my_shots, uint32_t& my_fail, uint32_t& my_rescans) {
  const int n = t.n, m = t.m, K = t.K, M = t.M, T = t.T, nw = t.nw, kw = t.kw, mw = t.mw;
  const uint32_t* dec = reinterpret_cast<const uint32_t*>(gs + t.xg_dec);
  float* lpost = reinterpret_cast<float*>(gs + t.xg_lpost);
  float* acc = reinterpret_cast<float*>(gs + t.xg_acc);
  uint32_t* cand = reinterpret_cast<uint32_t*>(gs + t.xg_cand);
  float* cpost = reinterpret_cast<float*>(gs + t.xg_cpost);

  const uint32_t* syn = a.syn + (size_t)shot * a.syn_stride;
  int nsyn = 0;
  for (int w = lane; w < mw; w += 32) {
    const int rem = m - 32 * w;
    nsyn += __popc(__ldg(syn + w) & (rem >= 32 ? 0xffffffffu : ((1u << rem) - 1u)));
  }
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) nsyn += __shfl_xor_sync(kFull, nsyn, off);
  ++my_shots;
  uint32_t* out_corr = a.corr + (size_t)shot * a.corr_stride;

  if (nsyn == 0 && !a.want_soft) {
    // s = 0: every member converges in iteration 1 to e = 0; member 0 is chosen
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
    MemberRun R{syn, nsyn, budget, a.want_soft != 0, ncand == 0, nullptr, K, M, a.x_chunk, 0, 0u};
    const int conv = team_member<MT, DP>(t, i, R, gs);
    my_iters += (uint32_t)R.ran;
    my_rescans += R.rescans;
    if (conv) {
      // insert (conv, i); i exceeds every member already listed, so it goes after equal iterations
      const int p = __popc(__ballot_sync(kFull, lane < ncand && c_t <= conv));
      const int slot = ncand < M ? ncand : __shfl_sync(kFull, c_slot, M - 1);
      const float W = decision_weight(t, dec, cand + (size_t)slot * nw, lane);
      if (a.want_soft) {
        float* dst = cpost + (size_t)slot * n;
        for (int v = lane; v < n; v += 32) dst[v] = lpost[v];
      }
      const float uW = __shfl_up_sync(kFull, c_W, 1);
      const int ut = __shfl_up_sync(kFull, c_t, 1), ui = __shfl_up_sync(kFull, c_i, 1);
      const int us = __shfl_up_sync(kFull, c_slot, 1);
      const int last = min(ncand, M - 1);
      if (lane > p && lane <= last) { c_W = uW; c_t = ut; c_i = ui; c_slot = us; }
      if (lane == p) { c_W = W; c_t = conv; c_i = i; c_slot = slot; }
      ncand = min(ncand + 1, M);
    } else if (ncand == 0) {
      // not converged after T sweeps and no candidate yet: add LLR^i / ||LLR^i|| (finite entries)
      llr_term_add(lpost, acc, n, i == 0, lane);
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
      const float* src = cpost + (size_t)slot * n;
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

// Pair mode: member i of shot `shot` (slot `slot` of the chunk) with the team; the last member of the
// shot to finish writes the shot's outcome (pair_epilogue, vibe_internal.cuh).
template <typename MT, int DP>
__device__ __forceinline__ void decode_pair_x(const BpArgs& a, const Tables& t, uint32_t shot, int slot, int i,
                                              unsigned char* gs, int lane, uint32_t& my_iters,
                                              uint32_t& my_shots, uint32_t& my_fail, uint32_t& my_rescans) {
  const int K = t.K, M = t.M, T = t.T, n = t.n, m = t.m, mw = t.mw, nw = t.nw, kw = t.kw;
  if (i >= K) return;
  const uint32_t* syn = a.syn + (size_t)shot * a.syn_stride;
  int nsyn = 0;
  for (int w = lane; w < mw; w += 32) {
    const int rem = m - 32 * w;
    nsyn += __popc(__ldg(syn + w) & (rem >= 32 ? 0xffffffffu : ((1u << rem) - 1u)));
  }
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) nsyn += __shfl_xor_sync(kFull, nsyn, off);
  if (nsyn == 0 && !a.want_soft) {
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
  const uint32_t* dec = reinterpret_cast<const uint32_t*>(gs + t.xg_dec);
  float* lpost = reinterpret_cast<float*>(gs + t.xg_lpost);
  int* conv = a.pconv + (size_t)slot * a.pair_K;
  MemberRun R{syn, nsyn, T, a.want_soft != 0, true, conv, K, M, a.x_chunk, 0, 0u};
  const int cv = team_member<MT, DP>(t, i, R, gs);
  my_iters += (uint32_t)R.ran;
  my_rescans += R.rescans;
  const size_t rec = (size_t)slot * a.pair_K + i;
  if (cv) {
    const float W = decision_weight(t, dec, a.pbits + rec * a.bnd.nw, lane);
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

// MIXED: shots name their problems (dem_of_shot); the descriptors are copied to shared memory after
// the team's region, and shots of image-engine problems or of another team size are left to their
// launches. Otherwise every shot decodes a.one from the parameter space. The register budget is 128, with
// which the sweep spills nothing. (80 registers spill inside it and are no faster: the engine waits on
// latencies.)
template <typename MT, int DP, bool MIXED>
__global__ void __launch_bounds__(kTeam * 32, 2) k_bpx(const __grid_constant__ BpArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31;
  const int W = (int)(blockDim.x >> 5);
  Tables* sdem = reinterpret_cast<Tables*>(smem + (size_t)a.x_team_smem);
  if (MIXED) {
    const uint32_t* src = reinterpret_cast<const uint32_t*>(a.dems);
    uint32_t* dst = reinterpret_cast<uint32_t*>(sdem);
    const int words = a.ndem * (int)(sizeof(Tables) / 4);
    for (int q = threadIdx.x; q < words; q += blockDim.x) dst[q] = __ldg(src + q);
    __syncthreads();
  }
  unsigned char* gs = a.xscratch + (long long)blockIdx.x * a.xscratch_pitch;
  uint32_t my_iters = 0, my_shots = 0, my_fail = 0, my_rescans = 0;   // flushed before they could wrap
  if (threadIdx.x >= 32) {
    my_rescans = team_serve<MT, DP>(gs);
    if (lane == 0 && a.counters && my_rescans) atomicAdd(a.counters + VIBE_CNT_RESCANS, (unsigned long long)my_rescans);
    return;
  }

  if (a.pair_mode) {
    const unsigned long long npairs = (unsigned long long)a.nshots * (unsigned long long)a.pair_K;
    for (;;) {
      unsigned long long q = 0;
      if (lane == 0) q = atomicAdd(a.next_pair_x, 1u);
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
          if (lane == 0) {
            if (a.stats) {
              vibe_shot_stats st;
              st.status = VIBE_STATUS_BAD_PROBLEM; st.lsd_invoked = 0; st.n_converged = 0; st.chosen_member = 0;
              st.iters = 0; st.largest_cluster = 0; st.n_clusters = 0;
              a.stats[shot] = st;
            }
            if (a.counters) atomicAdd(a.counters + VIBE_CNT_BAD_PROBLEM, 1ull);
          }
          continue;
        }
        if (sdem[di].engine != VIBE_ENGINE_SUMMARY || sdem[di].team != W) continue;   // left to another launch
        decode_pair_x<MT, DP>(a, sdem[di], shot, (int)shot, i, gs, lane, my_iters, my_shots, my_fail, my_rescans);
      } else {
        decode_pair_x<MT, DP>(a, a.one, shot, (int)shot, i, gs, lane, my_iters, my_shots, my_fail, my_rescans);
      }
    }
  }
  for (;;) {
    if (a.pair_mode) break;
    if (my_iters > 0x70000000u || my_rescans > 0x70000000u) {
      if (lane == 0 && a.counters) {
        atomicAdd(a.counters + VIBE_CNT_PAIR_ITERS, (unsigned long long)my_iters);
        atomicAdd(a.counters + VIBE_CNT_RESCANS, (unsigned long long)my_rescans);
      }
      my_iters = 0;
      my_rescans = 0;
    }
    uint32_t shot = 0;
    if (lane == 0) shot = atomicAdd(a.next_shot_x, 1u);
    shot = __shfl_sync(kFull, shot, 0);
    if (shot >= a.nshots) break;
    if (MIXED) {
      const int di = __ldg(a.dem_of_shot + shot);
      if ((unsigned)di >= (unsigned)a.ndem) {
        if (!a.flag_bad) continue;
        for (int w = lane; w < a.corr_stride; w += 32) a.corr[(size_t)shot * a.corr_stride + w] = 0u;
        if (a.logical)
          for (int w = lane; w < a.log_stride; w += 32) a.logical[(size_t)shot * a.log_stride + w] = 0u;
        if (a.soft)
          for (int j = lane; j < a.soft_stride; j += 32) a.soft[(size_t)shot * a.soft_stride + j] = 0.0f;
        if (lane == 0) {
          if (a.stats) {
            vibe_shot_stats st;
            st.status = VIBE_STATUS_BAD_PROBLEM; st.lsd_invoked = 0; st.n_converged = 0; st.chosen_member = 0;
            st.iters = 0; st.largest_cluster = 0; st.n_clusters = 0;
            a.stats[shot] = st;
          }
          if (a.counters) atomicAdd(a.counters + VIBE_CNT_BAD_PROBLEM, 1ull);
        }
        continue;
      }
      if (sdem[di].engine != VIBE_ENGINE_SUMMARY || sdem[di].team != W) continue;   // left to another launch
      decode_shot_x<MT, DP>(a, sdem[di], shot, gs, lane, my_iters, my_shots, my_fail, my_rescans);
    } else {
      decode_shot_x<MT, DP>(a, a.one, shot, gs, lane, my_iters, my_shots, my_fail, my_rescans);
    }
  }
  if (W > 1) {
    if (lane == 0) reinterpret_cast<TeamCmd*>(smem)->go = 0;
    __syncthreads();
  }
  if (lane == 0 && a.counters) {
    atomicAdd(a.counters + VIBE_CNT_SHOTS, (unsigned long long)my_shots);
    atomicAdd(a.counters + VIBE_CNT_PAIR_ITERS, (unsigned long long)my_iters);
    if (my_fail) atomicAdd(a.counters + VIBE_CNT_FAILURES, (unsigned long long)my_fail);
    if (my_rescans) atomicAdd(a.counters + VIBE_CNT_RESCANS, (unsigned long long)my_rescans);
  }
}

inline size_t a16(size_t x) { return (x + 15) & ~(size_t)15; }

template <typename MT, int DP, bool MIXED>
cudaError_t prefer_shared() {
  // the summaries and the ring are the working set; L1 caches little here
  static bool done[kMaxDevices] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return cudaSuccess;
  if (done[dev]) return cudaSuccess;
  cudaError_t err = cudaFuncSetAttribute(k_bpx<MT, DP, MIXED>, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  if (err == cudaSuccess) done[dev] = true;
  return err;
}

template <typename MT, int DP, bool MIXED>
cudaError_t launch_x(const BpArgs& a, int grid, int team, size_t smem, cudaStream_t s) {
  cudaError_t err = prefer_shared<MT, DP, MIXED>();
  if (err != cudaSuccess) return err;
  err = ensure_dyn_smem<k_bpx<MT, DP, MIXED>>(smem);
  if (err != cudaSuccess) return err;
  k_bpx<MT, DP, MIXED><<<grid, team * 32, smem, s>>>(a);
  return cudaGetLastError();
}

template <typename MT, int DP, bool MIXED>
cudaError_t occupancy_x(size_t smem, int team, int* out) {
  cudaError_t err = prefer_shared<MT, DP, MIXED>();
  if (err != cudaSuccess) return err;
  err = ensure_dyn_smem<k_bpx<MT, DP, MIXED>>(smem);
  if (err != cudaSuccess) return err;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, k_bpx<MT, DP, MIXED>, team * 32, smem);
}

template <typename Fn>
cudaError_t by_xd(int XD, Fn&& f) {
  switch (XD) {
    case 4: return f(std::integral_constant<int, 4>{});
    case 6: return f(std::integral_constant<int, 6>{});
    case 8: return f(std::integral_constant<int, 8>{});
    case 16: return f(std::integral_constant<int, 16>{});
    default: return cudaErrorInvalidValue;
  }
}

template <typename MT>
cudaError_t launch_x_mt(const BpArgs& a, int grid, int team, cudaStream_t s) {
  const bool mixed = a.dem_of_shot != nullptr;
  const size_t smem = bpx_cta_smem_bytes(a.bnd, team, mixed ? a.ndem : 0);
  return by_xd(a.bnd.XD, [&](auto dp) {
    if (mixed) return launch_x<MT, decltype(dp)::value, true>(a, grid, team, smem, s);
    return launch_x<MT, decltype(dp)::value, false>(a, grid, team, smem, s);
  });
}

template <typename MT>
cudaError_t occupancy_x_mt(const Bounds& b, int team, int ndem, int* out) {
  const size_t smem = bpx_cta_smem_bytes(b, team, ndem);
  return by_xd(b.XD, [&](auto dp) {
    if (ndem > 0) return occupancy_x<MT, decltype(dp)::value, true>(smem, team, out);
    return occupancy_x<MT, decltype(dp)::value, false>(smem, team, out);
  });
}

}  // namespace

int bpx_degree_bucket(int maxcol) {
  return maxcol <= 4 ? 4 : maxcol <= 6 ? 6 : maxcol <= 8 ? 8 : maxcol <= 16 ? 16 : 0;
}

int bpx_summary_bytes(int m, int msg_fp16) { return (int)a16((msg_fp16 ? 8 : 16) * (size_t)m); }

void bpx_layout(Tables* t, int msg_fp16) {
  long long g = 0;
  t->xg_msg = g;   g += (long long)a16((size_t)t->SP * (msg_fp16 ? 2 : 4));
  t->xg_st = g;    g += (long long)a16(8 * (size_t)t->nstep);
  t->xg_dec = g;   g += (long long)a16(4 * (size_t)t->nw);
  t->xg_lpost = g; g += (long long)a16(4 * (size_t)t->n);
  t->xg_acc = g;   g += (long long)a16(4 * (size_t)t->n);
  t->xg_cand = g;  g += (long long)a16(4 * (size_t)t->M * t->nw);
  t->xg_cpost = g;
  t->x_warp_scratch = g;
}

static size_t team_smem(const Bounds& b, int team, int chunk) {
  return sizeof(TeamCmd) + (size_t)team * window_bytes(chunk) + (size_t)b.x_sums[team_class(team)];
}

// Steps per chunk: kChunk, or for single warps 2 where only that fits beside the summaries and descriptors. That
// takes m above 10,000, and LSD's shared memory ends at m = 4300, so 2 is not chosen at present. The choice
// stays because the kernel without it measured slower with FP32 messages: XYZ d=7 49.9 -> 53.2 ms, circuit d=11 150 ->
// 161 ms, the same in five forms of the code around the sweep.
static int bpx_chunk(const Bounds& b, int team, int ndem) {
  const size_t limit = 227u * 1024u;   // shared memory of a CTA on sm_103a
  return team == 1 && team_smem(b, team, kChunk) + a16((size_t)ndem * sizeof(Tables)) > limit ? 2 : kChunk;
}

size_t bpx_cta_smem_bytes(const Bounds& b, int team, int ndem) {
  return team_smem(b, team, bpx_chunk(b, team, ndem)) + a16((size_t)ndem * sizeof(Tables));
}

cudaError_t launch_bpx(const BpArgs& a0, int team, int msg_fp16, int grid, cudaStream_t s) {
  BpArgs a = a0;
  a.x_chunk = bpx_chunk(a.bnd, team, a.dem_of_shot ? a.ndem : 0);
  a.x_team_smem = (int)team_smem(a.bnd, team, a.x_chunk);
  return msg_fp16 ? launch_x_mt<__half>(a, grid, team, s) : launch_x_mt<float>(a, grid, team, s);
}

cudaError_t bpx_occupancy(const Bounds& b, int team, int ndem, int msg_fp16, int* blocks_per_sm) {
  return msg_fp16 ? occupancy_x_mt<__half>(b, team, ndem, blocks_per_sm) : occupancy_x_mt<float>(b, team, ndem, blocks_per_sm);
}

}  // namespace vibe

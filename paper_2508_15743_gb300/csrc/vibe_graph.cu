// K0 -- Tanner-graph builder (offline setup, Sec. III.D.1).
//
// From the CSR of H it builds, on the device: the CSC of H (checks ascending per column), the packed
// per-column edge table csc_ent of the flooding and layered sweeps, the padded message image (prior LLR of
// each edge's column, +inf padding), and for every ensemble member its serial schedule packed into steps
// of 32 edges (k_steps): columns of one step touch disjoint checks and columns that share a check keep
// their order, so the steps give the same floats as the serial order of Algorithm 1 (serial branch).
#include "vibe_internal.cuh"

namespace vibe {
namespace {

__global__ void k_col_count(const int32_t* __restrict__ colidx, int E, int32_t* __restrict__ cnt) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < E; e += gridDim.x * blockDim.x)
    atomicAdd(&cnt[colidx[e]], 1);
}

// Exclusive scan of cnt[0..n) into out[0..n], one CTA (used once per handle).
__global__ void k_scan_single(const int32_t* __restrict__ cnt, int n, int32_t* __restrict__ out) {
  __shared__ int32_t part[1024];
  __shared__ int32_t carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int base = 0; base < n; base += 1024) {
    int i = base + threadIdx.x;
    int v = i < n ? cnt[i] : 0;
    part[threadIdx.x] = v;
    __syncthreads();
    for (int off = 1; off < 1024; off <<= 1) {
      int add = threadIdx.x >= off ? part[threadIdx.x - off] : 0;
      __syncthreads();
      part[threadIdx.x] += add;
      __syncthreads();
    }
    if (i < n) out[i] = carry + part[threadIdx.x] - v;
    __syncthreads();
    if (threadIdx.x == 1023) carry += part[1023];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[n] = carry;
}

// Scatter every edge into its column as (check << 8) | slot, slot = position inside the check row.
__global__ void k_csc_fill(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ colidx, int m,
                           const int32_t* __restrict__ colptr, int32_t* __restrict__ fill,
                           uint32_t* __restrict__ packed) {
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < m; c += gridDim.x * blockDim.x) {
    for (int e = rowptr[c]; e < rowptr[c + 1]; ++e) {
      int v = colidx[e];
      int pos = atomicAdd(&fill[v], 1);
      packed[colptr[v] + pos] = ((uint32_t)c << 8) | (uint32_t)(e - rowptr[c]);
    }
  }
}

// Sort each column's entries by check (insertion sort, degree <= 32) in place and emit rowidx and
// csc_ent.
__global__ void k_csc_finish(int n, int DP, int RP, int spc, const int32_t* __restrict__ colptr,
                             uint32_t* __restrict__ packed, int32_t* __restrict__ rowidx,
                             uint32_t* __restrict__ csc_ent) {
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
    int b = colptr[v], d = colptr[v + 1] - b;
    for (int i = 1; i < d; ++i) {
      uint32_t x = packed[b + i];
      int j = i - 1;
      while (j >= 0 && packed[b + j] > x) { packed[b + j + 1] = packed[b + j]; --j; }
      packed[b + j + 1] = x;
    }
    for (int k = 0; k < DP; ++k) {
      uint32_t x = k < d ? packed[b + k] : 0u;
      csc_ent[(size_t)v * DP + k] = k < d ? csc_entry(x >> 8, x & 0xffu, RP, spc) : 0u;
      if (k < d) rowidx[b + k] = (int32_t)(x >> 8);
    }
  }
}

template <typename MT>
__device__ __forceinline__ MT to_msg(float x);
template <>
__device__ __forceinline__ float to_msg<float>(float x) { return x; }
template <>
__device__ __forceinline__ __half to_msg<__half>(float x) { return __float2half_rn(x); }

template <typename MT>
__global__ void k_msg_init(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ colidx, int m, int RP,
                           const float* __restrict__ lam, MT* __restrict__ out) {
  const int spc = 16 / (int)sizeof(MT);
  long long total = (long long)m * RP;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(t / RP), pos = (int)(t % RP);
    const int slot = (int)row_position((uint32_t)c, (uint32_t)pos, RP, spc);   // the XOR swizzle is its own inverse
    const int deg = rowptr[c + 1] - rowptr[c];
    float x = slot < deg ? lam[colidx[rowptr[c] + slot]] : __int_as_float(0x7f800000);
    out[t] = to_msg<MT>(x);
  }
}

template <typename MT>
__device__ __forceinline__ float msg_magnitude(MT x);
template <>
__device__ __forceinline__ float msg_magnitude<float>(float x) { return fabsf(x); }
template <>
__device__ __forceinline__ float msg_magnitude<__half>(__half x) { return fabsf(__half2float(x)); }

// Summary engine: the summary of each check's prior messages -- the two smallest magnitudes (ordered by
// value, then row position) with their positions, the third smallest as the floor (+inf when the row
// is shorter; a missing second holder is position 255 with +inf), and the parity of the messages' sign
// bits (bit 31). The syndrome enters per shot in the kernel.
template <typename MT>
__global__ void k_xsum(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ colidx, int m,
                       const float* __restrict__ lam, float4* __restrict__ out) {
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < m; c += gridDim.x * blockDim.x) {
    const float inf = __int_as_float(0x7f800000);
    float a1 = inf, a2 = inf, a3 = inf;
    uint32_t q1 = 255u, q2 = 255u, sg = 0u;
    for (int q = rowptr[c]; q < rowptr[c + 1]; ++q) {
      const MT x = to_msg<MT>(lam[colidx[q]]);
      const float a = msg_magnitude<MT>(x);
      const uint32_t p = (uint32_t)(q - rowptr[c]);
      sg ^= (float)x < 0.0f ? 1u : 0u;
      if (a < a1 || (a == a1 && p < q1)) { a3 = a2; a2 = a1; q2 = q1; a1 = a; q1 = p; }
      else if (a < a2 || (a == a2 && p < q2)) { a3 = a2; a2 = a; q2 = p; }
      else if (a < a3) a3 = a;
    }
    out[c] = make_float4(a1, a2, a3, __uint_as_float(q1 | (q2 << 8) | (sg << 31)));
  }
}

// The steps of every member's sweep (one warp per member): its columns, taken in the member's order,
// are packed into steps of at most 32 edges, each column into the first step that (1) comes after the
// steps of all earlier columns it shares a check with and (2) still has a lane for each of its checks
// (one lane for a column without checks). Columns of one step therefore share no check, and two
// columns that do keep their order, so a sweep that takes the steps one after another, one lane per
// edge, computes the floats of the serial order.
// Why steps and not the wavefront levels: a level is cut where the next column conflicts, whatever
// its size, and rounding each level up to whole warps leaves lanes idle. On random orders of the d=9
// phenomenological problem the levels make 79 warps of edges and the steps 62 (E / 32 = 60.8); on
// circuit-level d=11 4887 and 4407 (4371).
// With a team of W > 1 warps (summary engine) W consecutive steps form a unit that shares no check, and
// the steps are numbered so that a warp's steps of kStepChunk consecutive units are neighbours: their
// records are copied together. Step u of the packing is number team_place(u); the count is rounded up to
// whole groups of kStepChunk * W.
// slot[v] = step << 5 | first lane, nstep = number of steps, off[s] = edges before step s (s <= nstep).
// The search looks at 64 windows of 32 steps; past them it opens a new step at the end, which bounds the
// work per column. lo (lane d - 1: degree d) skips the steps known to have no room for that degree.
constexpr int kStepWindows = 64;

__device__ __forceinline__ uint32_t team_place(uint32_t x, uint32_t W) {
  if (W == 1u) return x;
  const uint32_t unit = x / W;
  return unit / kStepChunk * kStepChunk * W + (x % W) * kStepChunk + unit % kStepChunk;
}
__device__ __forceinline__ uint32_t team_unplace(uint32_t s, uint32_t W) {
  if (W == 1u) return s;
  const uint32_t group = kStepChunk * W, q = s % group;
  return (s / group * kStepChunk + q % kStepChunk) * W + q / kStepChunk;
}

__global__ void k_steps(const uint32_t* __restrict__ perm, int n, int m, const int32_t* __restrict__ colptr,
                        const uint32_t* __restrict__ cpos, int room_in_smem, uint32_t* __restrict__ slot,
                        uint32_t* __restrict__ off, int32_t* __restrict__ nstep, uint8_t* __restrict__ room_g, int cap,
                        int off_pitch, uint32_t W) {
  extern __shared__ uint32_t sh[];
  uint32_t* nxt = sh;                       // m: first step allowed at each check
  uint32_t* stage = sh + m;                 // 32 x kMaxColDeg: checks of the 32 columns in work
  uint8_t* room = room_in_smem ? reinterpret_cast<uint8_t*>(stage + 32 * kMaxColDeg)
                               : room_g + (size_t)blockIdx.x * cap;   // free lanes of each step
  const int lane = threadIdx.x;
  perm += (size_t)blockIdx.x * n;
  slot += (size_t)blockIdx.x * n;
  off += (size_t)blockIdx.x * off_pitch;
  for (int c = lane; c < m; c += 32) nxt[c] = 0u;
  uint32_t lo = 0u;
  uint32_t ns = 0u;
  for (int t0 = 0; t0 < n; t0 += 32) {
    const int cnt = min(32, n - t0);
    uint32_t v = 0u;
    int d = 0;
    __syncwarp();
    if (lane < cnt) {
      v = perm[t0 + lane];
      const int b = colptr[v];
      d = colptr[v + 1] - b;
      for (int k = 0; k < d; ++k) stage[lane * kMaxColDeg + k] = cpos[b + k] >> 8;
    }
    __syncwarp();
    uint32_t mine = 0u;
    for (int j = 0; j < cnt; ++j) {
      const int dj = __shfl_sync(kFull, d, j);
      const uint32_t need = (uint32_t)max(dj, 1);
      const uint32_t c = lane < dj ? stage[j * kMaxColDeg + lane] : 0u;
      const uint32_t s0 = __reduce_max_sync(kFull, lane < dj ? nxt[c] : 0u);
      const uint32_t lod = __shfl_sync(kFull, lo, (int)need - 1);
      uint32_t s = max(s0, lod);
      bool found = false;
      for (int w = 0; w < kStepWindows && !found; ++w) {
        const uint32_t x = s + lane;
        const uint32_t bal = __ballot_sync(kFull, x >= ns || room[x] >= need);
        if (bal) {
          s += (uint32_t)__ffs(bal) - 1u;
          found = true;
        } else {
          s += 32u;
        }
      }
      if (!found) s = max(ns, s0);
      else if (s0 <= lod && lane == (int)need - 1) lo = s;
      const uint32_t r = s < ns ? room[s] : 32u;
      if (lane == j) mine = (team_place(s, W) << 5) | (32u - r);
      __syncwarp();
      if (lane == 0) {
        for (uint32_t x = ns; x < s; ++x) room[x] = 32u;   // the rest of a unit may stay empty
        room[s] = (uint8_t)(r - need);
      }
      ns = max(ns, s + 1u);
      if (lane < dj) nxt[c] = (s / W + 1u) * W;
      __syncwarp();
    }
    if (lane < cnt) slot[v] = mine;
  }
  uint32_t run = 0u;
  const uint32_t group = kStepChunk * W, total = W == 1u ? ns : (ns + group - 1u) / group * group;
  for (uint32_t s0 = 0; s0 <= total; s0 += 32) {
    const uint32_t x = s0 + lane, px = team_unplace(x, W);
    const uint32_t u = x < total && px < ns ? 32u - room[px] : 0u;
    uint32_t inc = u;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(kFull, inc, o);
      if (lane >= o) inc += y;
    }
    if (x <= total) off[x] = run + inc - u;
    run += __shfl_sync(kFull, inc, 31);
  }
  if (lane == 0) nstep[blockIdx.x] = (int32_t)total;
}

// Column of each edge slot (only the slots of first edges are written, and read).
__global__ void k_step_columns(const uint32_t* __restrict__ slot, const uint32_t* __restrict__ off, int off_pitch, int n,
                               long long total, int SP, uint32_t* __restrict__ at) {
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < total;
       q += (long long)gridDim.x * blockDim.x) {
    const long long i = q / n;
    const uint32_t sl = slot[q];
    at[i * SP + off[i * off_pitch + (sl >> 5)] + (sl & 31u)] = (uint32_t)(q % n);
  }
}

// Order of a step's columns over its lanes (one warp per step). A 16-byte row load is served in four
// phases of eight lanes, and rows fall on the eight bank groups by their index mod 8 (row_position): a
// phase takes as many wavefronts as its most frequent residue. The columns are placed one after another,
// each time the one that adds least to its phases (ties: more checks first). On the d=9 phenomenological
// problem a row load of a step takes 8.0 wavefronts so ordered instead of 9.5 (ideal 4).
// cnt packs the current phase's counts, four bits per residue.
__global__ void k_step_order(const uint32_t* __restrict__ off, int off_pitch, const int32_t* __restrict__ nstep, int K,
                             int n, int SP, int per_member, const uint32_t* __restrict__ at,
                             const int32_t* __restrict__ colptr, const uint32_t* __restrict__ cpos,
                             uint32_t* __restrict__ slot) {
  const int lane = threadIdx.x & 31;
  const long long w = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  const int i = (int)(w / per_member), s = (int)(w % per_member);
  if (i >= K || s >= nstep[i]) return;
  const uint32_t b = off[(size_t)i * off_pitch + s];
  const int used = (int)(off[(size_t)i * off_pitch + s + 1] - b);
  slot += (size_t)i * n;
  // the step's columns, one per lane
  uint32_t v = 0u;
  int d = 0, cols = 0;
  for (int p = 0; p < used;) {
    const uint32_t u = at[(size_t)i * SP + b + p];
    const int du = colptr[u + 1] - colptr[u];
    if (lane == cols) { v = u; d = du; }
    ++cols;
    p += max(du, 1);
  }
  const int e0 = lane < cols ? colptr[v] : 0;
  bool left = lane < cols;
  int pos = 0;
  uint32_t cnt = 0u, top = 0u;   // the current phase's counts and their maximum
  for (int k = 0; k < cols; ++k) {
    uint32_t cost = 0u, c = cnt, t = top, t0 = top;
    if (left) {
      for (int j = 0; j < d; ++j) {
        if (((pos + j) & 7) == 0) { cost += t - t0; c = 0u; t = t0 = 0u; }
        const uint32_t r = 4u * ((cpos[e0 + j] >> 8) & 7u);
        c += 1u << r;
        t = max(t, (c >> r) & 15u);
      }
      cost += t - t0;
    }
    // least added cost, then most checks, then the lowest lane
    const uint32_t key = left ? (cost << 16) | ((uint32_t)(32 - d) << 8) | (uint32_t)lane : 0xffffffffu;
    const int pick = (int)(__reduce_min_sync(kFull, key) & 31u);
    if (lane == pick) {
      slot[v] = ((uint32_t)s << 5) | (uint32_t)pos;
      left = false;
    }
    const int dp = max(__shfl_sync(kFull, d, pick), 1);
    cnt = __shfl_sync(kFull, c, pick);
    top = __shfl_sync(kFull, t, pick);
    pos += dp;
    if ((pos & 7) == 0) cnt = top = 0u;
  }
}

// The step offsets with the common pitch of the resident table; the entries past a member's last step
// repeat its total.
__global__ void k_step_offsets(const uint32_t* __restrict__ tmp, int tmp_pitch, const int32_t* __restrict__ nstep, int K,
                               int pitch, uint32_t* __restrict__ soff) {
  const long long total = (long long)K * pitch;
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < total;
       q += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(q / pitch), s = (int)(q % pitch);
    soff[q] = tmp[(size_t)i * tmp_pitch + min(s, nstep[i])];
  }
}

// The edge records of every member's steps, one thread per (member, column); see Tables::xrec. xcolid
// names each slot's column, xrmap the message slot of each CSR entry of H.
__global__ void k_step_fill(const uint32_t* __restrict__ slot, const uint32_t* __restrict__ off, int off_pitch, int n,
                            long long total, int E, int SP, const int32_t* __restrict__ rowptr, const int32_t* __restrict__ colptr,
                            const uint32_t* __restrict__ cpos, const float* __restrict__ lam, uint2* __restrict__ xrec,
                            uint32_t* __restrict__ xlnk, uint32_t* __restrict__ xcolid, uint32_t* __restrict__ xrmap,
                            bool wide) {
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < total;
       q += (long long)gridDim.x * blockDim.x) {
    const long long i = q / n;
    const uint32_t v = (uint32_t)(q % n);
    const uint32_t sl = slot[q];
    const uint32_t o = off[i * off_pitch + (sl >> 5)] + (sl & 31u);
    const int b = colptr[v], d = colptr[v + 1] - b;
    const uint32_t lv = __float_as_uint(lam[v]);
    if (d == 0) {
      xrec[i * SP + o] = make_uint2(0u, lv);
      xlnk[i * SP + o] = 0u;
      xcolid[i * SP + o] = v;
    }
    for (int k = 0; k < d; ++k) {
      const uint32_t x = cpos[b + k];
      const uint32_t others = ((2u << (d - 1)) - 1u) & ~(1u << k);
      const uint32_t links = wide ? ((uint32_t)k << 5) | ((uint32_t)(d - 1) << 10)
                                  : (others << 5) | (((sl & 31u) + (uint32_t)(d - 1)) << kLnkLastLane);
      xrec[i * SP + o + k] = make_uint2(((x >> 8) << 18) | (x & 0xffu), lv);
      xlnk[i * SP + o + k] = (sl & 31u) | links | (k == d - 1 ? kLnkLast : 0u) | kLnkEdge;
      xcolid[i * SP + o + k] = v;
      if (xrmap) xrmap[(size_t)i * E + rowptr[x >> 8] + (x & 0xffu)] = o + (uint32_t)k;
    }
  }
}

__device__ __forceinline__ uint64_t splitmix64_next(uint64_t& st) {
  uint64_t z = (st += 0x9E3779B97F4A7C15ull);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

__global__ void k_seeded_schedules(uint32_t* __restrict__ perm, int n, int K, uint64_t seed) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= K) return;
  uint32_t* p = perm + (size_t)i * n;
  uint64_t st = seed + (uint64_t)(i + 1) * 0xD1B54A32D192ED03ull;
  for (int j = 0; j < n; ++j) p[j] = (uint32_t)j;
  for (int k = n - 1; k >= 1; --k) {
    uint64_t r = splitmix64_next(st);
    uint64_t j = __umul64hi(r, (uint64_t)(k + 1));
    uint32_t t = p[k]; p[k] = p[j]; p[j] = t;
  }
}

inline int grid_for(long long work, int threads) {
  long long g = (work + threads - 1) / threads;
  if (g < 1) g = 1;
  if (g > 65535) g = 65535;
  return (int)g;
}

}  // namespace

cudaError_t seeded_schedules(uint32_t* d_perm, int n, int K, uint64_t seed, cudaStream_t s) {
  k_seeded_schedules<<<(K + 63) / 64, 64, 0, s>>>(d_perm, n, K, seed);
  return cudaGetLastError();
}

// Check layers of the layered schedule (the oracle's reading R10): check c, in ascending order,
// joins the smallest layer that holds no earlier check sharing a column with it. One CTA: the checks
// are placed one after another (each placement depends on all earlier ones), the threads mark the
// layers of c's earlier neighbours with the stamp c and find the smallest unmarked one.
// scratch: layer_of[m] | stamp[m + 1]
__global__ void k_layers(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ colidx,
                         const int32_t* __restrict__ colptr, const int32_t* __restrict__ rowidx, int m,
                         int32_t* layer_ptr, int32_t* layer_chk, int32_t* layer_vptr, int32_t* layer_var,
                         int32_t* nlayer_out, int32_t* scratch) {
  int32_t* layer_of = scratch;
  int32_t* stamp = scratch + m;   // stamp[l] == c: layer l is taken for check c
  __shared__ int s_nl, s_best;
  for (int l = threadIdx.x; l <= m; l += blockDim.x) stamp[l] = -1;
  if (threadIdx.x == 0) { s_nl = 0; s_best = 0x7fffffff; }
  __syncthreads();
  for (int c = 0; c < m; ++c) {
    for (int e = rowptr[c] + threadIdx.x; e < rowptr[c + 1]; e += blockDim.x) {
      const int v = colidx[e];
      for (int k = colptr[v]; k < colptr[v + 1]; ++k) {
        const int c2 = rowidx[k];   // ascending in the column
        if (c2 >= c) break;
        stamp[layer_of[c2]] = c;
      }
    }
    __syncthreads();
    const int nl = s_nl;
    for (int l = threadIdx.x; l <= nl; l += blockDim.x)   // layer nl is always free
      if (stamp[l] != c) atomicMin(&s_best, l);
    __syncthreads();
    if (threadIdx.x == 0) {
      layer_of[c] = s_best;
      if (s_best == nl) s_nl = nl + 1;
      s_best = 0x7fffffff;
    }
    __syncthreads();
  }
  const int nl = s_nl;
  // group: counts, offsets, checks ascending within a layer, then each layer's columns
  if (threadIdx.x == 0) {
    for (int l = 0; l <= nl; ++l) { layer_ptr[l] = 0; layer_vptr[l] = 0; }
    for (int c = 0; c < m; ++c) {
      layer_ptr[layer_of[c] + 1] += 1;
      layer_vptr[layer_of[c] + 1] += rowptr[c + 1] - rowptr[c];
    }
    for (int l = 0; l < nl; ++l) { layer_ptr[l + 1] += layer_ptr[l]; layer_vptr[l + 1] += layer_vptr[l]; }
    for (int l = 0; l < nl; ++l) stamp[l] = 0;   // fill counters per layer
    for (int c = 0; c < m; ++c) {
      const int l = layer_of[c];
      layer_chk[layer_ptr[l] + stamp[l]++] = c;
    }
    // column offset of each check inside layer_var, kept in layer_of (no longer needed as a layer id)
    for (int l = 0; l < nl; ++l) {
      int o = layer_vptr[l];
      for (int q = layer_ptr[l]; q < layer_ptr[l + 1]; ++q) {
        const int c = layer_chk[q];
        layer_of[c] = o;
        o += rowptr[c + 1] - rowptr[c];
      }
    }
    *nlayer_out = nl;
  }
  __syncthreads();
  for (int c = 0; c < m; ++c) {
    const int o = layer_of[c], b = rowptr[c], d = rowptr[c + 1] - b;
    for (int j = threadIdx.x; j < d; j += blockDim.x) layer_var[o + j] = colidx[b + j];
  }
}

cudaError_t build_tables(const int32_t* d_rowptr, const int32_t* d_colidx, int m, int n, int E, int K,
                         const uint32_t* d_perm, int RP, int DP, int msg_fp16, const float* d_lam, int32_t* d_colptr,
                         int32_t* d_rowidx, uint32_t* d_cpos, uint32_t* d_csc_ent, void* d_msg_init, float4* d_xsum,
                         int32_t* d_scratch, cudaStream_t s) {
  // scratch layout: cnt[n] | fill[n]
  cudaError_t err;
  int32_t* cnt = d_scratch;
  int32_t* fill = cnt + n;
  if ((err = cudaMemsetAsync(cnt, 0, sizeof(int32_t) * 2 * (size_t)n, s)) != cudaSuccess) return err;
  k_col_count<<<grid_for(E, 256), 256, 0, s>>>(d_colidx, E, cnt);
  k_scan_single<<<1, 1024, 0, s>>>(cnt, n, d_colptr);
  k_csc_fill<<<grid_for(m, 128), 128, 0, s>>>(d_rowptr, d_colidx, m, d_colptr, fill, d_cpos);
  k_csc_finish<<<grid_for(n, 128), 128, 0, s>>>(n, DP, RP, msg_fp16 ? 8 : 4, d_colptr, d_cpos, d_rowidx, d_csc_ent);
  if (msg_fp16) {
    k_xsum<__half><<<grid_for(m, 128), 128, 0, s>>>(d_rowptr, d_colidx, m, d_lam, d_xsum);
    k_msg_init<__half><<<grid_for((long long)m * RP, 256), 256, 0, s>>>(d_rowptr, d_colidx, m, RP, d_lam,
                                                                       static_cast<__half*>(d_msg_init));
  } else {
    k_xsum<float><<<grid_for(m, 128), 128, 0, s>>>(d_rowptr, d_colidx, m, d_lam, d_xsum);
    k_msg_init<float><<<grid_for((long long)m * RP, 256), 256, 0, s>>>(d_rowptr, d_colidx, m, RP, d_lam,
                                                                      static_cast<float*>(d_msg_init));
  }
  return cudaGetLastError();
}

// Steps a member can have: one per column, in units of `team`, rounded up to whole groups.
static int step_cap(int n, int team) {
  const int group = kStepChunk * team;
  return team == 1 ? n : (n * team + group - 1) / group * group;
}

cudaError_t build_steps(int m, int n, int K, int team, const uint32_t* d_perm, const int32_t* d_colptr,
                        const uint32_t* d_cpos, int32_t* d_nstep, int32_t* d_scratch, cudaStream_t s) {
  const int cap = step_cap(n, team);
  uint32_t* slot = reinterpret_cast<uint32_t*>(d_scratch);
  uint32_t* off = slot + (size_t)K * n;
  uint8_t* room = reinterpret_cast<uint8_t*>(off + (size_t)K * (cap + 1));
  // m <= 16384 checks take 64 KB at most; the free-lane bytes follow when they fit too
  const size_t fixed = 4 * ((size_t)m + 32 * kMaxColDeg);
  const bool room_in_smem = fixed + (size_t)cap <= 160u * 1024u;
  const size_t smem = fixed + (room_in_smem ? (size_t)cap : 0);
  cudaError_t err = ensure_dyn_smem<k_steps>(smem);
  if (err != cudaSuccess) return err;
  k_steps<<<K, 32, smem, s>>>(d_perm, n, m, d_colptr, d_cpos, room_in_smem ? 1 : 0, slot, off, d_nstep, room, cap, cap + 1,
                              (uint32_t)team);
  return cudaGetLastError();
}

size_t step_scratch_ints(int n, int K, int team) {
  const size_t cap = step_cap(n, team);
  return (size_t)K * (n + cap + 1) + ((size_t)K * cap + 3) / 4;
}

cudaError_t order_steps(int n, int SP, int K, int nstep, const int32_t* d_colptr, const uint32_t* d_cpos,
                        const int32_t* d_nstep, int32_t* d_scratch, uint32_t* d_tmp, cudaStream_t s) {
  uint32_t* slot = reinterpret_cast<uint32_t*>(d_scratch);
  const uint32_t* off = slot + (size_t)K * n;
  k_step_columns<<<grid_for((long long)K * n, 256), 256, 0, s>>>(slot, off, n + 1, n, (long long)K * n, SP, d_tmp);
  const long long blocks = ((long long)K * nstep + 3) / 4;   // four warps each
  k_step_order<<<(unsigned)blocks, 128, 0, s>>>(off, n + 1, d_nstep, K, n, SP, nstep, d_tmp, d_colptr, d_cpos, slot);
  return cudaGetLastError();
}

cudaError_t fill_steps(int n, int E, int SP, int K, int DP, int team, int pitch, const int32_t* d_rowptr, const int32_t* d_colptr,
                       const uint32_t* d_cpos, const float* d_lam, const int32_t* d_nstep, const int32_t* d_scratch,
                       uint32_t* d_soff, uint2* d_xrec, uint32_t* d_xlnk, uint32_t* d_xcolid, uint32_t* d_xrmap,
                       cudaStream_t s) {
  const uint32_t* slot = reinterpret_cast<const uint32_t*>(d_scratch);
  const uint32_t* off = slot + (size_t)K * n;
  const int off_pitch = step_cap(n, team) + 1;
  k_step_offsets<<<grid_for((long long)K * pitch, 256), 256, 0, s>>>(off, off_pitch, d_nstep, K, pitch, d_soff);
  k_step_fill<<<grid_for((long long)K * n, 256), 256, 0, s>>>(slot, off, off_pitch, n, (long long)K * n, E, SP, d_rowptr,
                                                              d_colptr, d_cpos, d_lam, d_xrec, d_xlnk, d_xcolid, d_xrmap, DP > 16);
  return cudaGetLastError();
}

cudaError_t build_layers(const int32_t* d_rowptr, const int32_t* d_colidx, const int32_t* d_colptr,
                         const int32_t* d_rowidx, int m, int32_t* d_layer_ptr, int32_t* d_layer_chk,
                         int32_t* d_layer_vptr, int32_t* d_layer_var, int32_t* d_nlayer, int32_t* d_scratch,
                         cudaStream_t s) {
  k_layers<<<1, 256, 0, s>>>(d_rowptr, d_colidx, d_colptr, d_rowidx, m, d_layer_ptr, d_layer_chk, d_layer_vptr,
                             d_layer_var, d_nlayer, d_scratch);
  return cudaGetLastError();
}

}  // namespace vibe

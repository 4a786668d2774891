// decode.cu -- decode-phase update of the retained caches, one generated token
// per call, for every layer of a route in one launch (the decode step of the
// rules Sec. 2.1 cites: H2O accumulates the new token's attention, TOVA keeps
// only the current step's attention, StreamingLLM keeps sinks + a rolling
// window, and a layer without a decode-phase rule appends).
//
// Decode arena (caller-owned device memory, layout from the plan): layer l
// holds B*H_kv*cap_l slots, slot (s, h, j) at row row_off(l) + (s*H_kv + h) *
// cap_l + j of dec_K / dec_V.  The state buffer holds lens[B], and per unit u
// = unit_off(l) + s*H_kv + h: count[u], evicted[u], and per slot pos (the
// position it holds, -1 = empty) and acc (H2O: accumulated attention; TOVA:
// the last step's attention).  Slot order carries no meaning: an evicted
// slot is overwritten by the new token.
//
// One CTA per H2O / TOVA unit, or a cluster of up to eight when there are few
// units (each CTA takes a run of 16-slot tiles; the softmax normalisers and the
// eviction candidates cross the cluster through distributed shared memory),
// and one warp per StreamingLLM or append-only unit (eight per CTA).  H2O /
// TOVA: the G query rows of the new token attend to every retained slot and to
// the new token, p_j = (1/G) sum_g softmax_j(q_g . k_j / sqrt(d)); acc += p (H2O) or acc = p (TOVA).  When the unit already
// holds b slots, the slot with the smallest acc among positions older than
// the protected recent window (r = h2o_recent for H2O, 0 for TOVA) is
// evicted, ties to the higher position, and the new token takes its place
// (unless the new token itself is the one evicted).  The retained K rows are
// streamed once, as 16-byte loads feeding m16n8k16 tensor-core products of
// the G query rows; logits stay in shared memory.
#include "kvev_internal.cuh"

namespace kvev {

namespace {

constexpr int kDecodeThreads = 256;

// Unit index -> layer: the last layer whose first unit is <= u (layers
// without slots own no units and share their unit_off with the next layer).
__device__ __forceinline__ int find_dec_layer(const DecodeParams& p, int u) {
  int lo = 0, hi = p.L - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (p.layer[mid].unit_off <= u) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// A warp's or CTA's eviction candidate (DecChoice) and, from the CTA that holds
// the new token's index, the new token's key.
struct __align__(16) DecCandidate {
  uint32_t hi, lo;
  int aux;
  float new_key;
};

constexpr int kDecodeWarps = kDecodeThreads / 32;

// Every array is written once per step and read after one barrier.
template <bool kSplit>
struct DecShared {
  static constexpr int kC = kSplit ? kMaxDecCluster : 1;
  DecCandidate cand[kC];        // of every CTA of the cluster
  float cm[kC][8], cz[kC][8];   // their per-head (max, sum)
  __align__(16) float wmax[8][kDecodeWarps];  // per-head maxima of this CTA's warps (G <= 8 heads)
  __align__(16) float wsum[8][kDecodeWarps];  // and sums
  DecCandidate wcand[kDecodeWarps];           // their eviction candidates
};
static_assert(sizeof(DecShared<false>) <= 1024, "the host leaves 1 KiB beside the logits");

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

// Every thread of the cluster: what was stored to shared memory (its own or
// another CTA's) before is visible after.
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// A CTA may store into another one only once that one has started: every
// thread arrives when its unit's step begins and waits before the first store.
__device__ __forceinline__ void cluster_started_arrive() {
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_started_wait() {
  asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
}

// The address of this CTA's shared-memory object in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t cluster_addr(const void* p, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
  return a;
}

__device__ __forceinline__ void st_cluster(uint32_t addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}

__device__ __forceinline__ void st_cluster(uint32_t addr, const DecCandidate& c) {
  asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(c.hi), "r"(c.lo),
               "r"(c.aux), "r"(__float_as_int(c.new_key))
               : "memory");
}

// The maximum (kMax) or sum, over the warps, of one head's per-warp values.
template <bool kMax>
__device__ __forceinline__ float over_warps(const float (&w)[kDecodeWarps]) {
  static_assert(kDecodeWarps == 8, "two 16-byte loads");
  const float4 a = lds4(w), b = lds4(w + 4);
  return kMax ? fmaxf(fmaxf(fmaxf(a.x, a.y), fmaxf(a.z, a.w)), fmaxf(fmaxf(b.x, b.y), fmaxf(b.z, b.w)))
              : ((((((a.x + a.y) + a.z) + a.w) + b.x) + b.y) + b.z) + b.w;
}

// Eviction order: smaller key first, then higher position first; NaN after every
// number, the lower slot first.  As two words whose lexicographic minimum is the
// slot to evict the order is total, so that every lane, warp and CTA that merges
// candidates ends with the same one: each thread writes its part of the new row
// to the slot it found.
struct DecChoice {
  static constexpr uint32_t kNaN = 0xFFFFFFFEu;  // past +inf's
  uint32_t hi, lo;  // all ones: no candidate
  int aux;          // the slot, or with a NaN key, whose slot is lo, the position
  __device__ __forceinline__ int slot() const { return hi == kNaN ? static_cast<int>(lo) : aux; }
  __device__ __forceinline__ int pos() const { return hi == kNaN ? aux : static_cast<int>(0x7FFFFFFFu - lo); }
  __device__ __forceinline__ bool before(const DecChoice& o) const { return hi < o.hi || (hi == o.hi && lo < o.lo); }
};
constexpr DecChoice kNoChoice = {0xFFFFFFFFu, 0xFFFFFFFFu, -1};

__device__ __forceinline__ DecChoice candidate(float key, int pos, int slot) {
  const uint32_t u = __float_as_uint(key + 0.f);  // -0 as 0
  if (key != key) return DecChoice{DecChoice::kNaN, static_cast<uint32_t>(slot), pos};
  return DecChoice{u ^ (static_cast<uint32_t>(static_cast<int>(u) >> 31) | 0x80000000u),
                   0x7FFFFFFFu - static_cast<uint32_t>(pos), slot};
}

// The first candidate of the warp's lanes, in every lane.
__device__ __forceinline__ DecChoice warp_evict_choice(const DecChoice& d) {
  DecChoice r;
  r.hi = __reduce_min_sync(0xffffffffu, d.hi);
  r.lo = __reduce_min_sync(0xffffffffu, d.hi == r.hi ? d.lo : 0xFFFFFFFFu);
  const uint32_t who = __ballot_sync(0xffffffffu, d.hi == r.hi && d.lo == r.lo);
  r.aux = __shfl_sync(0xffffffffu, d.aux, __ffs(who) - 1);
  return r;
}

// Block-wide first candidate, in every thread; slot -1 if there is none.
__device__ __forceinline__ DecChoice block_evict_choice(const DecChoice& d, DecCandidate (&wcand)[kDecodeWarps]) {
  const int lane = threadIdx.x & 31;
  const DecChoice w = warp_evict_choice(d);
  if (lane == 0) wcand[threadIdx.x >> 5] = DecCandidate{w.hi, w.lo, w.aux, 0.f};
  __syncthreads();
  const DecCandidate e = wcand[lane & (kDecodeWarps - 1)];
  return warp_evict_choice(DecChoice{e.hi, e.lo, e.aux});
}

// Copy one d-wide bf16 row (16-byte vectors) with the whole block.
__device__ __forceinline__ void copy_row(uint16_t* dst, const uint16_t* src, int d) {
  for (int i = threadIdx.x; i < d / 8; i += blockDim.x)
    reinterpret_cast<uint4*>(dst)[i] = reinterpret_cast<const uint4*>(src)[i];
}

struct UnitRef {
  int l, s, h, u;
  size_t rows0;  // first slot row of the unit
};

// Put the new token into slot dst: its K/V row, position n and key.  Called by
// the whole block.
__device__ __forceinline__ void place_new(const DecodeParams& p, const DecLayer& ly, const UnitRef& r, int D, int dst,
                                          int n, float new_key) {
  const size_t src = static_cast<size_t>(r.s) * p.H_kv + r.h;
  copy_row(static_cast<uint16_t*>(p.K) + (r.rows0 + dst) * D, static_cast<const uint16_t*>(ly.k_new) + src * D, D);
  copy_row(static_cast<uint16_t*>(p.V) + (r.rows0 + dst) * D, static_cast<const uint16_t*>(ly.v_new) + src * D, D);
  if (threadIdx.x == 0) {
    p.pos[r.rows0 + dst] = n;
    p.acc[r.rows0 + dst] = new_key;
  }
}

// One m16n8k16 bf16 tensor-core product with fp32 accumulation (per warp):
// d[16 x 8] += a[16 x 16] * b[16 x 8].
__device__ __forceinline__ void mma_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Logits (base 2) of the G query rows against slots 0..c-1 and the new token
// (index c), tiles [tile0, tile1) of 16 indices, into lg[head][index - 16 tile0],
// and each warp's maximum per head into wmax.
template <int D, int G>
__device__ __forceinline__ void unit_logits(const DecodeParams& p, const uint16_t* Kb, const uint16_t* qn,
                                            const uint16_t* kn, int c, int tile0, int tile1, int ld, float* lg,
                                            float (&wmax)[8][kDecodeWarps]) {
  constexpr int KP = D / 32;  // k-step pairs
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int gid = lane >> 2, tig = lane & 3;
  // B fragments: head gid (column), dims kp*32 + tig*8 + 4w + [0, 4) of k-step 2kp + w
  uint32_t bq[2 * KP][2];
#pragma unroll
  for (int kp = 0; kp < KP; ++kp) {
#pragma unroll
    for (int w = 0; w < 2; ++w) {
      uint2 v = make_uint2(0, 0);
      if (gid < G) v = *reinterpret_cast<const uint2*>(qn + gid * D + kp * 32 + tig * 8 + 4 * w);
      bq[2 * kp + w][0] = v.x;
      bq[2 * kp + w][1] = v.y;
    }
  }
  // Slots 0..c-1 from the arena and the new token (index c) from its own k
  // row, 16 per tile; tiles are dealt to the warps in turn.
  const int cnt = c + 1;
  lg -= 16 * tile0;
  float mx0 = -INFINITY, mx1 = -INFINITY;  // this lane's heads 2tig, 2tig + 1
  for (int t = tile0 + warp; t < tile1; t += kDecodeThreads / 32) {
    const int j0 = t * 16 + gid, j1 = j0 + 8;  // this lane's two slot rows
    uint4 X[KP], Y[KP];
#pragma unroll
    for (int kp = 0; kp < KP; ++kp) {
      const int off = kp * 32 + tig * 8;
      X[kp] = make_uint4(0, 0, 0, 0);
      Y[kp] = make_uint4(0, 0, 0, 0);
      if (j0 < c) X[kp] = __ldcs(reinterpret_cast<const uint4*>(Kb + static_cast<size_t>(j0) * D + off));
      else if (j0 == c) X[kp] = *reinterpret_cast<const uint4*>(kn + off);
      if (j1 < c) Y[kp] = __ldcs(reinterpret_cast<const uint4*>(Kb + static_cast<size_t>(j1) * D + off));
      else if (j1 == c) Y[kp] = *reinterpret_cast<const uint4*>(kn + off);
    }
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int kp = 0; kp < KP; ++kp) {
      const uint32_t a0[4] = {X[kp].x, Y[kp].x, X[kp].y, Y[kp].y};
      const uint32_t a1[4] = {X[kp].z, Y[kp].z, X[kp].w, Y[kp].w};
      mma_16816(acc, a0, bq[2 * kp][0], bq[2 * kp][1]);
      mma_16816(acc, a1, bq[2 * kp + 1][0], bq[2 * kp + 1][1]);
    }
    // acc: (slot j0, heads 2tig, 2tig+1) and (slot j1, same heads)
    const int h0 = 2 * tig;
    if (h0 < G) {
      if (j0 < cnt) { lg[h0 * ld + j0] = acc[0] * p.scale_log2; mx0 = fmaxf(mx0, acc[0]); }
      if (j1 < cnt) { lg[h0 * ld + j1] = acc[2] * p.scale_log2; mx0 = fmaxf(mx0, acc[2]); }
    }
    if (h0 + 1 < G) {
      if (j0 < cnt) { lg[(h0 + 1) * ld + j0] = acc[1] * p.scale_log2; mx1 = fmaxf(mx1, acc[1]); }
      if (j1 < cnt) { lg[(h0 + 1) * ld + j1] = acc[3] * p.scale_log2; mx1 = fmaxf(mx1, acc[3]); }
    }
  }
  mx0 *= p.scale_log2;
  mx1 *= p.scale_log2;
#pragma unroll
  for (int o = 4; o < 32; o <<= 1) {
    mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, o));
    mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, o));
  }
  if (gid == 0) {
    if (2 * tig < G) wmax[2 * tig][warp] = mx0;
    if (2 * tig + 1 < G) wmax[2 * tig + 1][warp] = mx1;
  }
}

// H2O / TOVA unit.  lg: [G][cap + 1] floats of shared memory.
//
// Logits: a warp takes 16 slots at a time and forms S[16 slots][8 heads] =
// K Q^T on the tensor core (m16n8k16, heads past G are zero columns).  The
// dot product runs over d in a permuted order that lets every lane fill its
// A fragment from 16-byte loads of whole K rows: in the k-step pair kp, lane
// quadrant t (= lane % 4) holds dims kp*32 + t*8 + [0, 8) of its two slot
// rows; k-step 2kp + w takes elements 4w .. 4w + 3 of that slice (the low two
// as fragment columns 2t, 2t+1, the high two as 2t+8, 2t+9), and Q's B
// fragment is loaded in the same order.
//
// The CTA of rank `rank` of the unit's `p.cluster` CTAs takes a run of the
// tiles (kSplit; without it the one CTA takes all).  Each CTA softmaxes its
// run against its own maximum; the (max, sum) pairs of all CTAs give the scale
// of each, and their best eviction candidates the slot to evict.
template <int D, int G, bool kSplit>
__device__ void attend_unit(const DecodeParams& p, const DecLayer& ly, const UnitRef& r, int n, int c,
                            float* lg, DecShared<kSplit>& sh) {
  if (kSplit) cluster_started_arrive();
  const int C = kSplit ? p.cluster : 1;
  const uint32_t rank = kSplit ? cluster_rank() : 0;
  const int cnt = c + 1;                          // indices: slots 0..c-1, then the new token
  const int ntiles = (cnt + 15) / 16;
  const int per = kSplit ? (ntiles + C - 1) / C : ntiles;
  const int tile0 = kSplit ? min(static_cast<int>(rank) * per, ntiles) : 0;
  const int tile1 = kSplit ? min(tile0 + per, ntiles) : ntiles;
  const int base = 16 * tile0;                    // first index of this CTA
  const int m = kSplit ? max(0, min(cnt, 16 * tile1) - base) : cnt;  // and how many it has
  const int ld = kSplit ? 16 * ((ly.cap + 16) / 16 / C + 1) : ly.cap + 1;  // row stride of lg, >= 16 per
  const uint16_t* Kb = static_cast<const uint16_t*>(p.K) + r.rows0 * D;
  const uint16_t* kn = static_cast<const uint16_t*>(ly.k_new) + (static_cast<size_t>(r.s) * p.H_kv + r.h) * D;
  const uint16_t* qn = ly.q_new == nullptr
                           ? nullptr
                           : static_cast<const uint16_t*>(ly.q_new) + (static_cast<size_t>(r.s) * p.H_q + r.h * G) * D;

  // attention supplied by the caller's own decode attention: slots 0..c-1, then the new token
  // (never with a split unit)
  const float* at = kSplit || ly.attn == nullptr
                        ? nullptr
                        : ly.attn + (static_cast<size_t>(r.s) * p.H_kv + r.h) * static_cast<size_t>(ly.cap + 1);
  float zg[G];  // 1 / (G z) of every head's softmax (not needed when the attention is supplied)
#pragma unroll
  for (int g = 0; g < G; ++g) zg[g] = 1.f;
  if (at == nullptr) {
    unit_logits<D, G>(p, Kb, qn, kn, c, tile0, tile1, ld, lg, sh.wmax);
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float mg[G], z[G];
#pragma unroll
    for (int g = 0; g < G; ++g) {
      mg[g] = over_warps<true>(sh.wmax[g]);
      // another CTA may hold a finite logit: -inf here then weighs 0, not NaN
      if (kSplit && mg[g] == -INFINITY) mg[g] = 0.f;
      z[g] = 0.f;
    }
    for (int j = threadIdx.x; j < m; j += blockDim.x) {  // each thread keeps its own exponentials
#pragma unroll
      for (int g = 0; g < G; ++g) {
        const float e = exp2f(lg[g * ld + j] - mg[g]);
        lg[g * ld + j] = e;
        z[g] += e;
      }
    }
#pragma unroll
    for (int g = 0; g < G; ++g) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) z[g] += __shfl_xor_sync(0xffffffffu, z[g], o);
      if (lane == 0) sh.wsum[g][warp] = z[g];
    }
    __syncthreads();
    if (kSplit) {
      cluster_started_wait();
      for (int i = threadIdx.x; i < C * G; i += kDecodeThreads) {  // head g's pair to CTA k
        const int k = i / G, g = i - k * G;
        st_cluster(cluster_addr(&sh.cm[rank][g], k), over_warps<true>(sh.wmax[g]));
        st_cluster(cluster_addr(&sh.cz[rank][g], k), over_warps<false>(sh.wsum[g]));
      }
      __syncwarp();
      cluster_sync();
#pragma unroll
      for (int g0 = 0; g0 < G; g0 += 4) {  // lanes: four heads x the pairs of up to eight CTAs
        const int g = min(g0 + (lane >> 3), G - 1), k = lane & 7;
        const float mk = k < C ? sh.cm[k][g] : -INFINITY, zk = k < C ? sh.cz[k][g] : 0.f;
        float M = mk;
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
        float Z = zk * exp2f(mk - M);
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) Z += __shfl_xor_sync(0xffffffffu, Z, o);
        const float scale = exp2f(sh.cm[rank][g] - M) / (static_cast<float>(G) * Z);
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (g0 + q < G) zg[g0 + q] = __shfl_sync(0xffffffffu, scale, 8 * q);
      }
    } else {
#pragma unroll
      for (int g = 0; g < G; ++g) zg[g] = 1.0f / (static_cast<float>(G) * over_warps<false>(sh.wsum[g]));
    }
  }
  // group-mean attention -> new keys (each thread overwrites row 0 at its own j only)
  const float* accr = p.acc + r.rows0 + base;
  const int32_t* posr = p.pos + r.rows0 + base;
  if (at != nullptr) at += base;
  const int limit = n + 1 - ly.r;  // positions >= limit are protected
  const int mc = c - base;         // the new token's local index
  DecChoice ev = kNoChoice;        // the slot to evict: of the thread's slots, then of all
  constexpr int kU = 4;  // slots per thread whose global loads are issued together
  for (int j0 = threadIdx.x; j0 < m; j0 += kU * kDecodeThreads) {
    float accv[kU], atv[kU];
    int posv[kU];
#pragma unroll
    for (int q = 0; q < kU; ++q) {
      const int j = j0 + q * kDecodeThreads;
      const bool slot = j < m && j < mc;
      accv[q] = (ly.method == KVEV_H2O && slot) ? accr[j] : 0.f;
      posv[q] = slot ? posr[j] : n;
      atv[q] = (at != nullptr && j < m) ? at[j] : 0.f;
    }
#pragma unroll
    for (int q = 0; q < kU; ++q) {
      const int j = j0 + q * kDecodeThreads;
      if (j >= m) break;
      float pj = atv[q];
      if (at == nullptr) {  // group mean of the kept exponentials times 1 / (G z_g)
        pj = 0.f;
#pragma unroll
        for (int g = 0; g < G; ++g) pj += lg[g * ld + j] * zg[g];
      }
      const float a = accv[q] + pj;
      lg[j] = a;
      const int pos = posv[q];
      if (pos >= 0 && pos < limit) {
        const DecChoice x = candidate(a, pos, base + j);
        if (x.before(ev)) ev = x;
      }
    }
  }
  const bool full = c >= ly.b;
  float new_key = 0.f;
  if (full) {
    ev = block_evict_choice(ev, sh.wcand);  // slot c: the new token; ends past a barrier: lg is complete
    if (kSplit) {
      if (static_cast<int>(threadIdx.x) < C)
        st_cluster(cluster_addr(&sh.cand[rank], threadIdx.x),
                   DecCandidate{ev.hi, ev.lo, ev.aux, mc >= 0 && mc < m ? lg[mc] : 0.f});
      __syncwarp();
      cluster_sync();
      const int k = threadIdx.x & 7;
      ev = warp_evict_choice(k < C ? DecChoice{sh.cand[k].hi, sh.cand[k].lo, sh.cand[k].aux} : kNoChoice);
      new_key = sh.cand[(c / 16) / per].new_key;
    } else {
      new_key = lg[c];
    }
  } else {
    ev = kNoChoice;
    __syncthreads();
    if (mc >= 0 && mc < m) new_key = lg[mc];
  }
  const int bs = ev.slot();
  for (int j = threadIdx.x; j < m; j += blockDim.x)
    if (j < mc && base + j != bs) p.acc[r.rows0 + base + j] = lg[j];
  const bool lead = rank == 0 && threadIdx.x == 0;
  if (!full) {
    if (c >= ly.cap) {  // never for a consistent state: slots of an evicting layer stay <= b
      if (lead) atomicOr(p.status, kStatusDevice);
      return;
    }
    if (mc >= 0 && mc < m) place_new(p, ly, r, D, c, n, new_key);
    if (lead) {
      p.count[r.u] = c + 1;
      p.evicted[r.u] = -1;
    }
  } else if (bs < 0) {  // no evictable slot (protected window covers the cache)
    if (lead) atomicOr(p.status, kStatusDevice);
  } else {
    if (bs < c && bs >= base && bs < base + m) place_new(p, ly, r, D, bs, n, new_key);
    if (lead) {
      p.count[r.u] = c;
      p.evicted[r.u] = ev.pos();  // the new token's own position when it is the one evicted
    }
  }
}

__device__ __forceinline__ UnitRef unit_ref(const DecodeParams& p, int l, int rem) {
  const DecLayer& ly = p.layer[l];
  UnitRef r;
  r.l = l;
  r.s = rem / p.H_kv;
  r.h = rem - r.s * p.H_kv;
  r.u = ly.unit_off + rem;
  r.rows0 = static_cast<size_t>(ly.row_off) + static_cast<size_t>(rem) * ly.cap;
  return r;
}

// The step of the a-th H2O / TOVA unit (called by the whole block; returns
// early on an inconsistent state, which it records in the status word).
template <int D, int G, bool kSplit>
__device__ __forceinline__ void step_attend(const DecodeParams& p, int a, float* lg, DecShared<kSplit>& sh) {
  const int per_layer = p.B * p.H_kv;
  const int l = p.att_layer[a / per_layer];
  const DecLayer& ly = p.layer[l];
  const UnitRef r = unit_ref(p, l, a % per_layer);
  const int n = p.lens[r.s];
  const int c = p.count[r.u];
  if (c < 0 || c > ly.cap) {  // the same for every CTA of the unit
    if (threadIdx.x == 0) atomicOr(p.status, kStatusDevice);
    return;
  }
  attend_unit<D, G, kSplit>(p, ly, r, n, c, lg, sh);
}

// place_new by one warp: the new token's K/V row (16-byte vectors over the
// lanes), then its bookkeeping by lane 0.
__device__ __forceinline__ void place_new_warp(const DecodeParams& p, const UnitRef& r, int D, int dst, int n,
                                               float acc_new, int new_count, int evicted_pos) {
  const int lane = threadIdx.x & 31;
  if (dst >= 0) {
    const int vec = D / 8;
    const size_t src = static_cast<size_t>(r.s) * p.H_kv + r.h;
    for (int i = lane; i < 2 * vec; i += 32) {
      const bool isv = i >= vec;
      const int e = isv ? i - vec : i;
      uint4* drow = reinterpret_cast<uint4*>(isv ? p.V : p.K) + (r.rows0 + dst) * vec + e;
      const uint4* srow = reinterpret_cast<const uint4*>(isv ? p.layer[r.l].v_new : p.layer[r.l].k_new) + src * vec + e;
      *drow = *srow;
    }
  }
  if (lane == 0) {
    if (dst >= 0) {
      p.pos[r.rows0 + dst] = n;
      p.acc[r.rows0 + dst] = acc_new;
    }
    p.count[r.u] = new_count;
    p.evicted[r.u] = evicted_pos;
  }
}

// The step of the i-th StreamingLLM or append-only unit, by one warp (no
// block barrier): StreamingLLM evicts the smallest position >= sink once
// sink + recent slots are held; an append-only unit takes the next slot.
__device__ void step_cheap_warp(const DecodeParams& p, int i, int D) {
  const int lane = threadIdx.x & 31;
  const int per_layer = p.B * p.H_kv;
  const int l = p.cheap_layer[i / per_layer];
  const DecLayer& ly = p.layer[l];
  const UnitRef r = unit_ref(p, l, i % per_layer);
  const int n = p.lens[r.s];
  const int c = p.count[r.u];
  const bool streaming = ly.method == KVEV_STREAMING;
  if (c < 0 || c > ly.cap || (!streaming && c >= ly.cap) ||
      (streaming && c + 1 <= ly.sink + ly.recent && c >= ly.cap)) {
    if (lane == 0) atomicOr(p.status, kStatusDevice);
    return;
  }
  if (!streaming || c + 1 <= ly.sink + ly.recent) {  // append
    place_new_warp(p, r, D, c, n, 0.f, c + 1, -1);
    return;
  }
  // smallest position >= sink among the slots and the new token (positions are
  // distinct); 16 loads in flight per lane, as one warp scans the whole unit
  int bp = 0x7FFFFFFF, bs = -1;
  const int32_t* posr = p.pos + r.rows0;
  if (lane == 0 && n >= ly.sink) {
    bp = n;
    bs = c;
  }
  constexpr int kU = 16;
  for (int j0 = lane; j0 < c; j0 += 32 * kU) {
    int v[kU];
#pragma unroll
    for (int q = 0; q < kU; ++q) v[q] = j0 + 32 * q < c ? posr[j0 + 32 * q] : -1;
#pragma unroll
    for (int q = 0; q < kU; ++q) {
      if (v[q] >= ly.sink && v[q] < bp) {
        bp = v[q];
        bs = j0 + 32 * q;
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const int bp2 = __shfl_xor_sync(0xffffffffu, bp, o);
    const int bs2 = __shfl_xor_sync(0xffffffffu, bs, o);
    if (bp2 < bp) {
      bp = bp2;
      bs = bs2;
    }
  }
  __syncwarp();  // every lane has read the positions before slot bs is rewritten
  if (bs < 0) {
    if (lane == 0) atomicOr(p.status, kStatusDevice);
    return;
  }
  place_new_warp(p, r, D, bs < c ? bs : -1, n, 0.f, c, bp);
}

// What a unit (`rem` of its layer) reads of the caller's tensors, on its way to
// L2 before the wait for the step before: thread t of n.  The new token's rows
// are read at the end of the step's chain of round trips, and from HBM when the
// caller wrote them some time ago.  Measured with 32 steps' tokens laid out
// beforehand, 2,048 slots: batch 1 13.4 and 13.0 us a step, batch 16 91.6 and
// 90.6; with the attention supplied, batch 8: 8.2 and 7.5.
__device__ __forceinline__ void prefetch_l2(const void* base, size_t bytes, size_t at) {
  if (at < bytes) asm volatile("prefetch.global.L2 [%0];" ::"l"(static_cast<const char*>(base) + at));
}
template <int D, int G>
__device__ __forceinline__ void prefetch_token(const DecLayer& ly, int rem, bool attends, int t, int n) {
  constexpr size_t kRow = D * sizeof(uint16_t);
  const size_t at = 128 * static_cast<size_t>(t);
  prefetch_l2(static_cast<const char*>(ly.k_new) + rem * kRow, kRow, at);
  prefetch_l2(static_cast<const char*>(ly.v_new) + rem * kRow, kRow, at);
  if (!attends) return;
  if (ly.attn == nullptr) {
    prefetch_l2(static_cast<const char*>(ly.q_new) + rem * (G * kRow), G * kRow, at);
  } else {
    const size_t row = sizeof(float) * (static_cast<size_t>(ly.cap) + 1);
    for (size_t a = at; a < row; a += 128 * static_cast<size_t>(n))
      prefetch_l2(reinterpret_cast<const char*>(ly.attn) + rem * row, row, a);
  }
}

template <int D, int G, bool kSplit>
__global__ void __launch_bounds__(kDecodeThreads, kDecCtasPerSm) decode_step_kernel(const __grid_constant__ DecodeParams p) {
  extern __shared__ float lg[];
  __shared__ DecShared<kSplit> sh;
  // the H2O / TOVA units, and eight cheap units per CTA: after the others, or,
  // split, before them (those end first and leave their places; as a rule all
  // CTAs are resident at once, nothing depends on it)
  const int n_cheap_ctas = kSplit ? static_cast<int>(gridDim.x) - p.n_att * p.cluster : 0;
  const int n_att_ctas = kSplit ? 0 : p.n_att;
  const int b = static_cast<int>(blockIdx.x);
  const int per_layer = p.B * p.H_kv;
  if (kSplit ? b >= n_cheap_ctas : b < n_att_ctas) {
    const int a = kSplit ? (b - n_cheap_ctas) / p.cluster : b;
    prefetch_token<D, G>(p.layer[p.att_layer[a / per_layer]], a % per_layer, true, threadIdx.x, kDecodeThreads);
    pdl_wait();
    step_attend<D, G, kSplit>(p, a, lg, sh);
  } else {
    const int i = (b - n_att_ctas) * kDecodeWarps + (threadIdx.x >> 5);
    if (i < p.n_cheap)
      prefetch_token<D, G>(p.layer[p.cheap_layer[i / per_layer]], i % per_layer, false, threadIdx.x & 31, 32);
    pdl_wait();
    if (i < p.n_cheap) step_cheap_warp(p, i, D);
  }
  // The next kernel's CTAs come in as this one's finish.  Let in at the start of
  // the step they were placed beside CTAs with most of their work ahead, and
  // stayed there: 16 steps of 256 units of 256 slots 166 us, from here 147; 168
  // units of 512 slots in clusters of two 263 and 247; 256 units of 64 slots 99
  // and 105.
  pdl_trigger();
  // The last CTA of the step to finish advances every sequence by one token:
  // every other CTA has read lens before it counted itself done.
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(p.done, 1) == static_cast<int>(gridDim.x) - 1) {
      for (int s = 0; s < p.B; ++s) p.lens[s] += 1;
      *p.done = 0;
      __threadfence();
    }
  }
}

// A step of a route without decode units: the sequences are one token longer.
__global__ void decode_advance_kernel(int32_t* lens, int B) {
  for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < B; s += gridDim.x * blockDim.x) lens[s] += 1;
}

// Decode arena from the packed prefill output: slot j < kept count of unit
// (l, s, h) takes prefill row j (its position and, for H2O prefill layers,
// its score as the initial acc); the remaining slots are marked empty.  A
// unit's slots are split over init_split CTAs, and a thread has four vectors
// of K and four of V in flight: HBM-bound (rows read and written).  Measured,
// 32 layers x 8 heads x 2,048 slots, one CTA per unit and one vector of each
// at a time before: batch 1 169 and 83 us (6.4 TB/s), batch 16 1.32 and 1.28 ms (6.7 TB/s).
__global__ void __launch_bounds__(kDecodeThreads) decode_init_kernel(const __grid_constant__ DecodeParams p) {
  pdl_wait();
  pdl_trigger();
  const int u = blockIdx.x / p.init_split, part = blockIdx.x - u * p.init_split;
  const int l = find_dec_layer(p, u);
  const DecLayer& ly = p.layer[l];
  const int rem = u - ly.unit_off;
  const size_t rows0 = static_cast<size_t>(ly.row_off) + static_cast<size_t>(rem) * ly.cap;
  const size_t pre0 = static_cast<size_t>(ly.pre_row_off) + static_cast<size_t>(rem) * ly.pre_slots;
  int c = p.pre_count[static_cast<size_t>(l) * p.B * p.H_kv + rem];
  if (c < 0 || c > ly.pre_slots) {
    if (threadIdx.x == 0) atomicOr(p.status, kStatusDevice);
    c = 0;
  }
  const int per = (ly.cap + p.init_split - 1) / p.init_split;  // slots [j0, j1) are this CTA's
  const int j0 = min(part * per, ly.cap), j1 = min(j0 + per, ly.cap);
  const int vec = p.d / 8;  // 16-byte vectors per row
  const int nv = max(min(c, j1) - j0, 0) * vec;  // vectors to copy: contiguous in both
  const uint4* Ks = reinterpret_cast<const uint4*>(p.pre_K) + (pre0 + j0) * vec;
  const uint4* Vs = reinterpret_cast<const uint4*>(p.pre_V) + (pre0 + j0) * vec;
  uint4* Kd = reinterpret_cast<uint4*>(p.K) + (rows0 + j0) * vec;
  uint4* Vd = reinterpret_cast<uint4*>(p.V) + (rows0 + j0) * vec;
  constexpr int kU = 4;
  for (int i0 = threadIdx.x; i0 < nv; i0 += kU * kDecodeThreads) {
    uint4 kv[kU], vv[kU];
#pragma unroll
    for (int q = 0; q < kU; ++q) {
      const int i = i0 + q * kDecodeThreads;
      if (i < nv) {
        kv[q] = Ks[i];
        vv[q] = Vs[i];
      }
    }
#pragma unroll
    for (int q = 0; q < kU; ++q) {
      const int i = i0 + q * kDecodeThreads;
      if (i < nv) {
        Kd[i] = kv[q];
        Vd[i] = vv[q];
      }
    }
  }
  const bool seed_acc = ly.pre_method == KVEV_H2O && p.h2o_state != nullptr;
  for (int j = j0 + threadIdx.x; j < j1; j += blockDim.x) {
    p.pos[rows0 + j] = j < c ? p.pre_idx[pre0 + j] : -1;
    p.acc[rows0 + j] = (j < c && seed_acc) ? p.h2o_state[pre0 + j] : 0.f;
  }
  if (threadIdx.x == 0 && part == 0) {
    p.count[u] = c;
    p.evicted[u] = -1;
    if (u == 0) *p.done = 0;
  }
  if (u == 0 && part == 0)  // the first unit also copies the sequence lengths
    for (int i = threadIdx.x; i < p.B; i += blockDim.x) p.lens[i] = p.lens_in[i];
}

template <int D, int G, bool kSplit>
cudaError_t launch_step_dgs(const DecodeParams& p, size_t smem, int smem_optin, cudaStream_t st) {
  if (smem > 48 * 1024) {
    // one value for every call (all a block may have beside the static part):
    // the limit is the kernel's, and other plans and threads launch it too
    constexpr int kStatic = sizeof(DecShared<kSplit>) <= 1024 ? 1024 : 2048;
    static_assert(sizeof(DecShared<kSplit>) <= kStatic, "the limit leaves room for the static part");
    const cudaError_t e = cudaFuncSetAttribute(decode_step_kernel<D, G, kSplit>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, smem_optin - kStatic);
    if (e != cudaSuccess) return e;
  }
  const int cheap = (p.n_cheap + kDecodeWarps - 1) / kDecodeWarps;
  const int grid = p.n_att * p.cluster + (cheap + p.cluster - 1) / p.cluster * p.cluster;  // whole clusters
  return launch_overlapped(decode_step_kernel<D, G, kSplit>, p, grid, kDecodeThreads, smem, st, p.cluster);
}

template <int D, int G>
cudaError_t launch_step_dg(const DecodeParams& p, size_t smem, int smem_optin, cudaStream_t st) {
  return p.cluster > 1 ? launch_step_dgs<D, G, true>(p, smem, smem_optin, st) : launch_step_dgs<D, G, false>(p, smem, smem_optin, st);
}

template <int D>
cudaError_t launch_step_d(const DecodeParams& p, size_t smem, int smem_optin, cudaStream_t st) {
  switch (p.G) {
    case 1: return launch_step_dg<D, 1>(p, smem, smem_optin, st);
    case 2: return launch_step_dg<D, 2>(p, smem, smem_optin, st);
    case 4: return launch_step_dg<D, 4>(p, smem, smem_optin, st);
    case 8: return launch_step_dg<D, 8>(p, smem, smem_optin, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

bool decode_supported(int d, int G) {
  return (d == 64 || d == 128) && (G == 1 || G == 2 || G == 4 || G == 8);
}

// Dynamic shared memory of a step: `rows` rows of logits over a CTA's share of
// the unit's cap + 1 indices (cap slots and the new token).
size_t decode_logit_bytes(int cap, int rows, int cluster) {
  const size_t ld = cluster > 1 ? 16 * static_cast<size_t>((cap + 16) / 16 / cluster + 1) : static_cast<size_t>(cap) + 1;
  return sizeof(float) * rows * ld;
}

cudaError_t launch_decode_init(const DecodeParams& p, cudaStream_t st) {
  if (p.units == 0) return cudaSuccess;
  return launch_overlapped(decode_init_kernel, p, p.units * p.init_split, kDecodeThreads, 0, st);
}

cudaError_t launch_decode_step(const DecodeParams& p, size_t smem, int smem_optin, cudaStream_t st) {
  if (p.units > 0)  // the step kernel advances lens itself
    return p.d == 64 ? launch_step_d<64>(p, smem, smem_optin, st) : launch_step_d<128>(p, smem, smem_optin, st);
  decode_advance_kernel<<<1, 256, 0, st>>>(p.lens, p.B);
  return cudaGetLastError();
}

}  // namespace kvev

// Prompt-phase DMC compression (Algorithm 1 over a prompt, without attention).
//
// With binary alpha, Eq. partial-accumulation makes every slot the
// omega-weighted mean of one segment of consecutive tokens: a segment opens at
// a token with alpha = 0 (k[0] < 0) or at the first token of an empty head, and
// runs up to the next opening token; z of the slot is the segment's summed
// omega. Two kernels, no host synchronisation:
//
//  plan: one block per (sequence, KV head). Reads k[t, h, 0] of the prompt,
//        records which tokens open a slot (128 bits per chunk and head: a byte
//        per token and head, strided, cost plan + scan of a 7B layer 281 us
//        instead of 272, of one 2048-token prompt 28.7 instead of 24.6), counts
//        openings per 128-token chunk, takes pages for the head's new slots from
//        the pool (one atomic per head), and stores each chunk's first slot index.
//  scan: one block per (128-token chunk, KV head, sequence). The block owns the
//        segments that open inside its chunk (and chunk 0 also owns the tokens
//        that continue the head's existing last slot); a segment that runs past
//        the chunk end is followed to its end. Lanes split a row into 16-byte
//        pieces and accumulate sum(omega k), sum(omega v), sum(omega) in fp32;
//        the slot is the quotient, rounded once to the cache dtype. The chunk's
//        tokens are walked in row groups (see the kernel). When asked for
//        (prompt attention), the block also records, at every chunk start a
//        segment runs across, the segment's sums up to that point (the
//        "carry"), so that each chunk can rebuild the running state of its
//        tokens without reading back to the segment's start.
//  ring: window grouping only, after the scan: stores each head's open
//        segment's last W - 1 tokens and its length.
#include "dmc_internal.cuh"

namespace dmc {

constexpr int kPlanThreads = 256;
// Chunks of a warp of the plan in flight, four k[t, h, 0] a lane each. Every one
// costs its 128-byte line of DRAM (the floor: 40 us of a 7B layer's 47), but a
// head's block used to wait for each 256 tokens in turn: one 16384-token prompt,
// plan of 4096 tokens 16 us, now 9.
constexpr int kPlanChunks = 2;  // 4: the same
constexpr int kScanThreads = 128;

struct PrefillArgs {
  Layout lay;
  int layer, first_seq, num_seqs;
  const char* q;
  long long q_tok, q_head;  // element strides of the queries' first components
  const char* k;
  const char* v;
  const int* cu;
  int total_tokens, max_seqlen;
  float* carry;    // [chunk id][Hkv][2D + 1] (sum w k, sum w v, sum w), or null
  float* weights;  // with carry: [chunk id][Hkv][128], omega, its sign bit set where the token opens a slot
};

__device__ __forceinline__ bool seq_bounds(const PrefillArgs& a, int s, int& t0, int& t1) {
  t0 = a.cu[s];
  t1 = a.cu[s + 1];
  return t0 >= 0 && t0 <= t1 && t1 <= a.total_tokens && (t1 - t0) <= a.max_seqlen;
}

__device__ __forceinline__ int chunk_id(int t0, int c, int s) { return (t0 + c * kPrefillChunk) / kPrefillChunk + s; }

template <typename T, int D>
__global__ void __launch_bounds__(kPlanThreads) dmc_prefill_plan_kernel(const PrefillArgs a) {
  extern __shared__ int cnt[];  // [ceil(max_seqlen / 128)]
  __shared__ int s_fail, s_first_page, s_nan, s_wsum[kPlanThreads / 32 + 1];
  const Layout& L = a.lay;
  const int s = blockIdx.x, h = blockIdx.y;
  const int bh = (a.first_seq + s) * L.Hkv + h;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  griddep_launch_dependents();  // the scan may start its copies of k and v
  if (a.weights != nullptr && (blockIdx.x | blockIdx.y | tid) == 0) *L.unbounded = 0;
  const int parity = *reinterpret_cast<volatile int*>(&L.ctl[a.layer * 4]);
  int* len = L.lengths + ((size_t)a.layer * 2 + parity) * L.NH;
  int t0, t1;
  if (!seq_bounds(a, s, t0, t1)) {
    if (tid == 0) atomicOr(L.error, DMC_FAULT_BAD_SEQLENS);
    return;
  }
  const int ntok = t1 - t0;
  const int nch = ceil_div(ntok, kPrefillChunk);
  const int len_old = len[bh];
  if (tid == 0) { s_fail = 0; s_nan = 0; }
  __syncthreads();
  const T* kk = reinterpret_cast<const T*>(a.k);
  uint4* opens = L.opens + (size_t)h * L.plan_stride + chunk_id(t0, 0, s);  // chunk c: opens[c]
  bool nan = false;
  for (int cb = warp; cb < nch; cb += kPlanThreads / 32 * kPlanChunks) {  // a chunk is a warp's
    T x0[kPlanChunks][4];
#pragma unroll
    for (int u = 0; u < kPlanChunks; ++u)
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const int i = (cb + u * (kPlanThreads / 32)) * kPrefillChunk + v * 32 + lane;
        if (i < ntok) x0[u][v] = kk[((size_t)(t0 + i) * L.Hkv + h) * D];
      }
#pragma unroll
    for (int u = 0; u < kPlanChunks; ++u) {
      const int c = cb + u * (kPlanThreads / 32);
      if (c >= nch) break;  // the whole warp
      unsigned bits[4];
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const int i = c * kPrefillChunk + v * 32 + lane;
        bool op = false;
        if (i < ntok) {
          const float x = Elt<T>::to_f(x0[u][v]);
          nan |= x != x;
          // alpha = round(sigmoid(k[0])) = [k[0] >= 0]; alpha = 0 opens a slot,
          // and so does the first token of an empty head.
          op = !(x >= 0.f) || (i == 0 && len_old == 0);
        }
        bits[v] = __ballot_sync(0xffffffffu, op);
      }
      if (lane == 0) {
        opens[c] = make_uint4(bits[0], bits[1], bits[2], bits[3]);
        cnt[c] = __popc(bits[0]) + __popc(bits[1]) + __popc(bits[2]) + __popc(bits[3]);
      }
    }
  }
  if (nan) s_nan = 1;
  __syncthreads();
  // exclusive scan of the chunk counts (nch <= max_seqlen / 128 + 1)
  const int per = ceil_div(nch, kPlanThreads);
  const int c0 = min(tid * per, nch), c1 = min(c0 + per, nch);
  int local = 0;
  for (int c = c0; c < c1; ++c) local += cnt[c];
  int incl = local;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int o = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += o;
  }
  if (lane == 31) s_wsum[warp] = incl;
  __syncthreads();
  if (tid == 0) {
    int run = 0;
    for (int w = 0; w < kPlanThreads / 32; ++w) { const int t = s_wsum[w]; s_wsum[w] = run; run += t; }
    s_wsum[kPlanThreads / 32] = run;
  }
  __syncthreads();
  const int new_slots = s_wsum[kPlanThreads / 32];
  const int len_new = len_old + new_slots;
  const int old_pages = ceil_div(len_old, kPage), new_pages = ceil_div(len_new, kPage);
  const int need = new_pages - old_pages;
  if (tid == 0) {
    int fail = 0, first = 0;
    if (len_new > L.max_slots) {
      atomicOr(L.error, DMC_FAULT_SLOT_CAPACITY);
      fail = 1;
    } else if (need > 0) {
      const unsigned long long f = atomicAdd(L.pool_top, (unsigned long long)need);
      if (f + (unsigned long long)need > (unsigned long long)L.num_pages) {
        atomicOr(L.error, DMC_FAULT_PAGES_EXHAUSTED);
        fail = 1;
      } else {
        first = (int)f;
      }
    }
    if (s_nan) atomicOr(L.error, DMC_FAULT_NAN_GATE);
    s_fail = fail;
    s_first_page = first;
  }
  __syncthreads();
  const int fail = s_fail;
  int run = s_wsum[warp] + incl - local;
  for (int c = c0; c < c1; ++c) {
    L.plan[(size_t)h * L.plan_stride + chunk_id(t0, c, s)] = fail ? -1 : len_old + run;
    run += cnt[c];
  }
  if (!fail) {
    int* pt = L.page_table + ((size_t)a.layer * L.NH + bh) * L.MPH;
    for (int i = tid; i < need; i += kPlanThreads) pt[old_pages + i] = s_first_page + i;
    if (tid == 0) len[bh] = len_new;
  }
}

// Carry slot of the chunk of sequence s that starts at token cs (t0 = the
// sequence's first token).
__device__ __forceinline__ float* carry_at(const PrefillArgs& a, int t0, int cs, int s, int h, int D) {
  return a.carry + ((size_t)chunk_id(t0, (cs - t0) / kPrefillChunk, s) * a.lay.Hkv + h) * (2 * D + 1);
}

// Window grouping: the head's open segment [tb, te = end of the prompt), which
// had n_old tokens before this prompt, leaves its last W - 1 tokens (k with
// k[0] cleared, v, omega) in the ring and its length in seglen. One warp.
template <typename T, int D>
__device__ __forceinline__ void fill_ring(const PrefillArgs& a, int h, int bh, int tb, int te,
                                          int n_old) {
  constexpr int ROW = D * (int)sizeof(T);
  constexpr int LPR = ROW / 16;
  constexpr int RPI = 32 / LPR;
  const Layout& L = a.lay;
  const int W = L.window;
  const int lane = threadIdx.x & 31, sub = lane / LPR, lr = lane % LPR;
  const int parity = *reinterpret_cast<const volatile int*>(&L.ctl[a.layer * 4]);
  char* ring = L.ring + ((size_t)a.layer * L.NH + bh) * W * 2 * ROW;
  float* ring_w = L.ring_w + ((size_t)a.layer * L.NH + bh) * W;
  const T* qq = reinterpret_cast<const T*>(a.q);
  const size_t hrow = (size_t)L.Hkv * ROW;
  for (int t = max(tb, te - (W - 1)) + sub; t < te; t += RPI) {
    const int pos = (n_old + t - tb) % W;
    uint4 kr = __ldg(reinterpret_cast<const uint4*>(a.k + (size_t)t * hrow + (size_t)h * ROW + lr * 16));
    const uint4 vr = __ldg(reinterpret_cast<const uint4*>(a.v + (size_t)t * hrow + (size_t)h * ROW + lr * 16));
    if (lr == 0) {
      // k[0] <- 0: the first element of this lane's piece
      if (sizeof(T) == 2) kr.x &= 0xffff0000u;
      else kr.x = 0u;
    }
    *reinterpret_cast<uint4*>(ring + (size_t)pos * 2 * ROW + lr * 16) = kr;
    *reinterpret_cast<uint4*>(ring + (size_t)pos * 2 * ROW + ROW + lr * 16) = vr;
    if (lr == 0) {
      float y = 0.f;
      for (int g = 0; g < L.G; ++g)
        y += Elt<T>::to_f(qq[(size_t)t * a.q_tok + (size_t)(h * L.G + g) * a.q_head]);
      ring_w[pos] = sigmoidf_(y / (float)L.G);
    }
  }
  if (lane == 0) L.seglen[((size_t)a.layer * 2 + parity) * L.NH + bh] = n_old + (te - tb);
}

// Exact compression (no window). The chunk's tokens are split evenly among
// row groups of LPR lanes (a lane holds one 16-byte piece of a row); each group
// walks its tokens in order and closes a slot at every opening token. A lane
// streams its pieces of the group's rows through a private ring in shared
// memory (16-byte async copies, kRing rows ahead, issued before anything else
// the block needs), so the copies overlap the block's setup and the walk. What
// a group sums before its first opening is handed, through shared memory, to
// the group that holds the open segment before it. The chunk's last segment is
// followed past the chunk end up to the next opening token (recording the carry
// at each chunk start it runs across), and chunk 0 also finishes the segment
// that continues the head's existing last slot.
constexpr int kRing = 8;        // rows in a lane's ring
// Rows of a segment past its chunk that its group still adds alone (7B at 4x: three
// on average). More are summed by all groups: at CR 32 plan + scan of 32 x 2048
// tokens took 289 us so (270 now), with one group for any tail 477; at 4x the
// exchange costs more than it saves (297 us if every tail was shared, 281 so, 272
// now).
constexpr int kLongTail = 8;
constexpr int kRingBatch = 4;   // rows per async-copy group
constexpr size_t kScanRingBytes = (size_t)kRing * 2 * kScanThreads * 16;

// Window grouping (kWin): a slot counts only its segment's last W tokens, so the
// other tokens' rows are neither copied nor added, and a segment that continues the
// head's last slot takes the old tokens still inside the window from the head's ring
// (token p of the segment at entry p % W). The copies start once the decisions are
// known. Plan + scan of 16 x 1500 tokens in us (with every row of a longer segment read,
// its last W again; and with a warp per segment before that): bf16 d 128, W = 12, CR 4
// 118 (134; 349), CR 32 99 (125; 143), fp32 d 128 CR 32 112 (189; 165); a 7B layer at
// 4x, W = 12 284 (323; 891).
template <typename T, int D, bool kWin>
__global__ void __launch_bounds__(kScanThreads, 6) dmc_prefill_scan_kernel(const PrefillArgs a) {
  using CK = Chunk<T>;
  constexpr int ROW = D * (int)sizeof(T);
  constexpr int LPR = ROW / 16;               // lanes per row
  constexpr int NG = kScanThreads / LPR;      // row groups
  constexpr int TPG = kPrefillChunk / NG;     // tokens per group
  constexpr int NB = (TPG + kRingBatch - 1) / kRingBatch;
  constexpr int EPC = CK::N;
  constexpr int kMaxPages = kPrefillChunk / kPage + 2;
  constexpr int HS = 2 * D + 1;               // floats of one group's head sums
  static_assert(kScanThreads == kPrefillChunk, "one thread per chunk token");
  static_assert(TPG <= 32 && 32 % TPG == 0, "a group's tokens sit in one ballot word");
  static_assert(kRing == 2 * kRingBatch, "two copy groups in flight");
  static_assert((size_t)2 * NG * HS * sizeof(float) <= kScanRingBytes, "heads and tails fit the ring");
  __shared__ __align__(16) unsigned char ring[kScanRingBytes];  // [kRing][K, V][thread] 16 B
  __shared__ float s_w[kPrefillChunk];
  __shared__ unsigned s_bal[2 * kPrefillChunk / 32];  // opening bits: the chunk's, the next one's
  __shared__ int s_page[kMaxPages];
  __shared__ int s_next;
  const Layout& L = a.lay;
  const int c = blockIdx.x, h = blockIdx.y, s = blockIdx.z;
  const int bh = (a.first_seq + s) * L.Hkv + h;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = tid / LPR, lr = tid % LPR;
  int t0, t1;
  // every block waits for the plan before it ends, so that the scan never
  // completes ahead of the plan it was launched after
  if (!seq_bounds(a, s, t0, t1) || t0 + c * kPrefillChunk >= t1) {
    griddep_wait();
    return;
  }
  const int a0 = t0 + c * kPrefillChunk;
  const int a1 = min(a0 + kPrefillChunk, t1);
  const int g0 = a0 + g * TPG, g1 = min(g0 + TPG, a1);  // the group's tokens
  const size_t hrow = (size_t)L.Hkv * ROW;
  const char* kb = a.k + (size_t)h * ROW + lr * 16;
  const char* vb = a.v + (size_t)h * ROW + lr * 16;
  const uint32_t rbase = smem_u32(ring) + tid * 16;
  auto rk = [&](int pos) { return rbase + (uint32_t)(pos * 2) * kScanThreads * 16; };
  unsigned counts = 0;  // window grouping: the group's tokens that are summed
  auto issue = [&](int b) {  // copy group b: the group's rows g0 + 4b ... (always committed)
#pragma unroll
    for (int u = 0; u < kRingBatch; ++u) {
      const int t = g0 + b * kRingBatch + u;
      if (b < NB && t < g1 && (!kWin || (counts >> (t - g0) & 1u))) {
        const uint32_t dk = rk((b % 2) * kRingBatch + u);
        cp_async16(dk, kb + (size_t)t * hrow);
        cp_async16(dk + kScanThreads * 16, vb + (size_t)t * hrow);
      }
    }
    cp_async_commit();
  };
  if constexpr (!kWin) {
    issue(0);
    issue(1);
  }
  // launched as a programmatic dependent of the plan: what follows reads its
  // outputs (the copies above read only the prompt)
  griddep_wait();
  // Prompt attention may set itself up. (Only when it is what comes next: a decode
  // launched as a dependent would read this layer's slots while they are written.)
  if (a.weights != nullptr) griddep_launch_dependents();

  const int base = L.plan[(size_t)h * L.plan_stride + chunk_id(t0, c, s)];
  const int* len_both = L.lengths + (size_t)a.layer * 2 * L.NH + bh;  // as the plan left them
  const int len_0 = len_both[0], len_1 = len_both[L.NH];
  const int len = *reinterpret_cast<const volatile int*>(&L.ctl[a.layer * 4]) ? len_1 : len_0;
  const int nch = ceil_div(t1 - t0, kPrefillChunk);
  const uint4* opens = L.opens + (size_t)h * L.plan_stride + chunk_id(t0, c, s);  // [1]: the next chunk's
  const T* qq = reinterpret_cast<const T*>(a.q);
  // omega = sigmoid(q[0]) (group mean for GQA); the group's loads, up to eight
  // at a time, are in flight together
  auto omega = [&](int t) {
    const T* q0 = qq + (size_t)t * a.q_tok + (size_t)(h * L.G) * a.q_head;
    float y = Elt<T>::to_f(q0[0]);
    for (int g0 = 1; g0 < L.G; g0 += 7) {
      T x[7];
#pragma unroll
      for (int u = 0; u < 7; ++u)
        if (g0 + u < L.G) x[u] = q0[(size_t)(g0 + u) * a.q_head];
#pragma unroll
      for (int u = 0; u < 7; ++u)
        if (g0 + u < L.G) y += Elt<T>::to_f(x[u]);
    }
    return sigmoidf_(y / (float)L.G);
  };
  // pages of the slots the block may write, [base - 1, base + 128): at most
  // kMaxPages entries, all inside the head's row since the plan fitted the slots
  const int pfirst = max(base - 1, 0) / kPage;
  if (base >= 0 && tid < kMaxPages && pfirst + tid < L.MPH)
    s_page[tid] = L.page_table[((size_t)a.layer * L.NH + bh) * L.MPH + pfirst + tid];
  // the chunk's opening bits and the next one's (the first of those ends the
  // chunk's last segment); one thread per token: its omega
  {
    const unsigned* bits = reinterpret_cast<const unsigned*>(opens);
    // (the masks and the bounds below hold the walk inside the prompt, and the slots
    // inside the head, whatever the words and `base` say: sequences of inconsistent
    // cu_seqlens may share a chunk's entry)
    const int left = a1 - a0 - warp * 32;
    const unsigned mine = left >= 32 ? bits[warp] : left > 0 ? bits[warp] & ((1u << left) - 1u) : 0u;
    unsigned other = 0;
    if (lane == 0 && c + 1 < nch) other = bits[4 + warp];
    const float w = a0 + tid < a1 ? omega(a0 + tid) : 0.f;
    s_w[tid] = w;
    if (a.weights != nullptr)  // the sign set as a bit: that of a negated NaN is unspecified
      a.weights[((size_t)chunk_id(t0, c, s) * L.Hkv + h) * kPrefillChunk + tid] =
          __uint_as_float((__float_as_uint(w) & 0x7fffffffu) | ((mine >> lane) & 1u) << 31);
    if (lane == 0) { s_bal[warp] = mine; s_bal[kPrefillChunk / 32 + warp] = other; }
  }
  __syncthreads();
  int nstart = 0, first = -1, next = -1;
#pragma unroll
  for (int w = 0; w < kPrefillChunk / 32; ++w) {
    const unsigned b = s_bal[w], nb = s_bal[kPrefillChunk / 32 + w];
    if (first < 0 && b) first = w * 32 + __ffs(b) - 1;
    if (next < 0 && nb) next = a1 + w * 32 + __ffs(nb) - 1;
    nstart += __popc(b);
  }
  next = min(next, t1);
  const bool pre = c == 0 && base > 0 && !(s_bal[0] & 1u);  // continues the existing last slot
  if (base < 0 || base + nstart > len || (nstart == 0 && !pre)) {
    // the plan failed (or the entry is another sequence's), or every token belongs
    // to an earlier chunk's segment
    cp_async_wait<0>();
    return;
  }
  if constexpr (kWin) {
    // Bit j of x: the token after the group's j-th opens a slot, or the prompt has
    // ended. The j-th counts if one of bits j .. j + W - 1 is set (TPG + W <= 64).
    const int q = g * TPG + 1, w0 = q >> 5;
    unsigned long long x = (unsigned long long)s_bal[w0 + 1] << 32 | s_bal[w0];
    if (q & 31) x = x >> (q & 31) | (unsigned long long)s_bal[w0 + 2] << (64 - (q & 31));
    const int end = t1 - a0 - q;
    if (end >= 0 && end < 64) x |= 1ull << end;
    for (int n = 1; n < L.window;) {
      const int d = min(n, L.window - n);
      x |= x >> d;
      n += d;
    }
    counts = (unsigned)x;
    issue(0);
    issue(1);
  }
  if (next < 0) {  // no opening in the next 128 tokens: search on (uniform)
    if (tid == 0) s_next = t1;
    __syncthreads();
#pragma unroll 1
    for (int cb = 2; c + cb < nch; cb += kScanThreads) {
      bool found = false;
      if (c + cb + tid < nch) {
        const uint4 b = opens[cb + tid];
        const int at = b.x ? __ffs(b.x) : b.y ? 32 + __ffs(b.y) : b.z ? 64 + __ffs(b.z) : b.w ? 96 + __ffs(b.w) : 0;
        found = at != 0;
        if (found) atomicMin(&s_next, a0 + (cb + tid) * kPrefillChunk + at - 1);
      }
      if (__syncthreads_or(found)) break;
    }
    next = s_next;
  }

  float ak[EPC], av[EPC], zs = 0.f;
  auto reset = [&]() {
#pragma unroll
    for (int e = 0; e < EPC; ++e) { ak[e] = 0.f; av[e] = 0.f; }
    zs = 0.f;
  };
  auto add_to = [&](float* xk, float* xv, float& xz, const uint4& kr, const uint4& vr, float w) {
    float kf[EPC], vf[EPC];
    CK::unpack(kr, kf);
    CK::unpack(vr, vf);
    if (lr == 0) kf[0] = 0.f;  // k[0] <- 0 (Algorithm 1)
    const float2 ww = make_float2(w, w);
#pragma unroll
    for (int e = 0; e < EPC; e += 2) {
      const float2 sk = fma2(ww, make_float2(kf[e], kf[e + 1]), make_float2(xk[e], xk[e + 1]));
      const float2 sv = fma2(ww, make_float2(vf[e], vf[e + 1]), make_float2(xv[e], xv[e + 1]));
      xk[e] = sk.x; xk[e + 1] = sk.y;
      xv[e] = sv.x; xv[e + 1] = sv.y;
    }
    xz += w;
  };
  auto add_row = [&](const uint4& kr, const uint4& vr, float w) { add_to(ak, av, zs, kr, vr, w); };
  // The chunk's last segment runs on to `next`, its rows from `tail` on are summed.
  // Few are its group's work; more are summed by all groups, 128 tokens at a time.
  const int tail = kWin ? max(a1, next - L.window) : a1;
  const bool long_tail = next - tail > kLongTail;
  auto slot_ptr = [&](int slot) {
    const int page = s_page[slot / kPage - pfirst];
    return L.pages + (size_t)page * L.page_bytes + (size_t)(slot % kPage) * ROW + lr * 16;
  };
  auto write_slot = [&](int slot) {  // the slot = the segment's omega-weighted mean
    char* kdst = slot_ptr(slot);
    const float iz = 1.f / zs;
    float kn[EPC], vn[EPC];
#pragma unroll
    for (int e = 0; e < EPC; ++e) {
      kn[e] = ak[e] * iz;
      vn[e] = av[e] * iz;
    }
    if (a.weights != nullptr) {  // (a token's infinite or NaN value is its slot's, too)
      float x = 0.f;
#pragma unroll
      for (int e = 0; e < EPC; ++e) x = fmaf(vn[e], 0.f, x);
      if (x != x) *L.unbounded = 1;
    }
    if (lr == 0) kn[0] = 0.f;
    *reinterpret_cast<uint4*>(kdst) = CK::pack(kn);
    *reinterpret_cast<uint4*>(kdst + (size_t)kPage * ROW) = CK::pack(vn);
    if (lr == 0) L.z[(size_t)s_page[slot / kPage - pfirst] * kPage + slot % kPage] = zs;
  };
  auto group_bits = [&](int gg) {  // the opening tokens of group gg's range
    const unsigned b = s_bal[(gg * TPG) >> 5] >> ((gg * TPG) & 31);
    return TPG == 32 ? b : (b & ((1u << TPG) - 1u));
  };

  // walk: tokens [max(g0, wb), g1), wb = the first token the block owns (the
  // token loop stays rolled: one copy of the slot write keeps the code small)
  const int wb = pre ? a0 : a0 + first;
  const unsigned gbits = group_bits(g);
  int slot = base - 1;  // the slot of the segment being summed
  {
    const int wi = (g * TPG) >> 5;
    for (int w = 0; w < wi; ++w) slot += __popc(s_bal[w]);
    slot += __popc(s_bal[wi] & ((1u << ((g * TPG) & 31)) - 1u));
  }
  float hk[EPC], hv[EPC], hz = 0.f;  // the sums before the group's first opening
  bool open = false;                 // summing a segment that opened in this group
  reset();
  for (int b = 0; b < NB; ++b) {
    cp_async_wait<1>();  // copy group b has landed
#pragma unroll 1
    for (int u = 0; u < kRingBatch; ++u) {
      const int t = g0 + b * kRingBatch + u;
      if (t >= wb && t < g1) {
        if ((gbits >> (t - g0)) & 1u) {  // t opens a slot: the segment before it ends
          if (open) {
            write_slot(slot);
          } else {
#pragma unroll
            for (int e = 0; e < EPC; ++e) { hk[e] = ak[e]; hv[e] = av[e]; }
            hz = zs;
          }
          reset();
          open = true;
          ++slot;
        }
        if (kWin && !(counts >> (t - g0) & 1u)) continue;
        const uint32_t sk = rk((b % 2) * kRingBatch + u);
        uint4 kr, vr;
        asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(kr.x), "=r"(kr.y), "=r"(kr.z), "=r"(kr.w) : "r"(sk) : "memory");
        asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(vr.x), "=r"(vr.y), "=r"(vr.z), "=r"(vr.w)
                     : "r"(sk + kScanThreads * 16) : "memory");
        add_row(kr, vr, s_w[t - a0]);
      }
    }
    issue(b + 2);  // into the ring rows just read
  }
  if (!open) {  // no opening in the range: all of it joins an earlier segment
#pragma unroll
    for (int e = 0; e < EPC; ++e) { hk[e] = ak[e]; hv[e] = av[e]; }
    hz = zs;
  }
  // the heads replace the ring (every copy has landed: the last groups are empty)
  cp_async_wait<0>();
  __syncthreads();
  float* heads = reinterpret_cast<float*>(ring);
  float* tails = heads + NG * HS;
  auto put = [&](float* to) {
#pragma unroll
    for (int e = 0; e < EPC; ++e) {
      to[g * HS + lr * EPC + e] = hk[e];
      to[g * HS + D + lr * EPC + e] = hv[e];
    }
    if (lr == 0) to[g * HS + 2 * D] = hz;
  };
  auto add = [&](const float* from) {
#pragma unroll
    for (int e = 0; e < EPC; ++e) {
      ak[e] += from[lr * EPC + e];
      av[e] += from[D + lr * EPC + e];
    }
    zs += from[2 * D];
  };
  // Adds the rows tb, tb + step, ... below te, one at a time: two in flight spill more
  // than they hide (plan + scan of 32 x 2048 tokens at CR 32: 270 us with one, 281 with
  // two; long ragged prompts 596 and 604; windowed prompts 0-7 %).
  auto add_rows = [&](float* xk, float* xv, float& xz, int tb, int step, int te) {
#pragma unroll 1
    for (int t = tb; t < te; t += step) {
      const uint4 kr = __ldg(reinterpret_cast<const uint4*>(kb + (size_t)t * hrow));
      const uint4 vr = __ldg(reinterpret_cast<const uint4*>(vb + (size_t)t * hrow));
      add_to(xk, xv, xz, kr, vr, omega(t));
    }
  };
  auto tail_sums = [&](int pb) {  // this group's rows among [pb, min(next, pb + 128))
#pragma unroll
    for (int e = 0; e < EPC; ++e) { hk[e] = 0.f; hv[e] = 0.f; }
    hz = 0.f;
    add_rows(hk, hv, hz, pb + g, NG, min(next, pb + kPrefillChunk));
  };
  put(heads);
  if (long_tail) {
    tail_sums(tail);
    put(tails);
  }
  __syncthreads();

  const bool carry = a.carry != nullptr;
  auto put_carry = [&](int cs) {  // the sums so far, as the carry of the chunk at cs
    float* cp = carry_at(a, t0, cs, s, h, D);
#pragma unroll
    for (int e = 0; e < EPC; ++e) {
      cp[lr * EPC + e] = ak[e];
      cp[D + lr * EPC + e] = av[e];
    }
    if (lr == 0) cp[2 * D] = zs;
  };
  // adds the heads of the groups after gg up to the first with an opening; if
  // none has one, the segment is the chunk's last and runs on to `next`: true,
  // after its rows in the 128 tokens from a1 have been added
  auto finish = [&](int gg) -> bool {
    for (++gg; gg < NG; ++gg) {
      add(heads + gg * HS);
      if (group_bits(gg)) return false;
    }
    if (next > a1 && carry) put_carry(a1);
    if (long_tail) {
#pragma unroll 1
      for (int i = 0; i < NG; ++i) add(tails + i * HS);
    } else {
      add_rows(ak, av, zs, tail, 1, next);
    }
    return true;
  };
  // where the segment that is open at the end of group gg ends
  auto segment_end = [&](int gg) {
    for (++gg; gg < NG; ++gg)
      if (const unsigned bits = group_bits(gg)) return a0 + gg * TPG + __ffs(bits) - 1;
    return next;
  };
  // The segment that continues the head's last slot is group 0's work (of chunk
  // 0); with an opening in the chunk group 0 may have one of its own besides,
  // whose sums it puts aside.
  const bool both = pre && g == 0 && nstart > 0 && open;
  bool mine = open, past = false;
  if (pre && g == 0) {
    const int own_slot = slot;
    if (both) {
#pragma unroll
      for (int e = 0; e < EPC; ++e) { hk[e] = ak[e]; hv[e] = av[e]; }
      hz = zs;
    }
    slot = base - 1;
    if constexpr (kWin) {
      // the continued segment's tokens still inside the window
      reset();
      const int W = L.window, te = segment_end(-1);
      const int parity = *reinterpret_cast<const volatile int*>(&L.ctl[a.layer * 4]);
      const int n_old = L.seglen[((size_t)a.layer * 2 + parity) * L.NH + bh];
      const int m = min(n_old, W - (te - t0));
      const char* old = L.ring + ((size_t)a.layer * L.NH + bh) * W * 2 * ROW + lr * 16;
      const float* old_w = L.ring_w + ((size_t)a.layer * L.NH + bh) * W;
#pragma unroll 2
      for (int e = 0; e < m; ++e) {
        const int pos = (n_old - 1 - e) % W;
        add_row(*reinterpret_cast<const uint4*>(old + (size_t)pos * 2 * ROW),
                *reinterpret_cast<const uint4*>(old + (size_t)pos * 2 * ROW + ROW), old_w[pos]);
      }
    } else {
      // the old slot's K z_old, V z_old and z_old start the sums
      const char* kold = slot_ptr(slot);
      float ko[EPC], vo[EPC];
      CK::unpack(*reinterpret_cast<const uint4*>(kold), ko);
      CK::unpack(*reinterpret_cast<const uint4*>(kold + (size_t)kPage * ROW), vo);
      const float zo = L.z[(size_t)s_page[slot / kPage - pfirst] * kPage + slot % kPage];
#pragma unroll
      for (int e = 0; e < EPC; ++e) {
        ak[e] = ko[e] * zo;
        av[e] = vo[e] * zo;
      }
      zs = zo;
      if (carry) put_carry(t0);  // the state the prompt's first token continues
    }
    past = finish(-1);
    if (nstart > 0) {
      write_slot(slot);
      past = false;
      slot = own_slot;
      if (both) {
#pragma unroll
        for (int e = 0; e < EPC; ++e) { ak[e] = hk[e]; av[e] = hv[e]; }
        zs = hz;
      }
    } else {
      mine = true;  // the chunk's only segment: below
    }
  }
  if (open) past = finish(g);
  if constexpr (!kWin) {
    // a segment that runs on beyond the 128 tokens from a1
    for (int pb = a1 + kPrefillChunk; pb < next; pb += kPrefillChunk) {
      if (past && carry) put_carry(pb);
      tail_sums(pb);
      __syncthreads();  // the tails before have been read
      put(tails);
      __syncthreads();
      if (past)
        for (int i = 0; i < NG; ++i) add(tails + i * HS);
    }
  }
  if (mine) write_slot(slot);
}

// Window grouping: after the scan (which read the old window of continued
// segments), one block per (sequence, KV head) finds the head's open segment
// (from the prompt's last opening token, or the whole prompt if it continued
// the old one) and stores its last W - 1 tokens and its length.
template <typename T, int D>
__global__ void __launch_bounds__(kPlanThreads) dmc_prefill_ring_kernel(const PrefillArgs a) {
  __shared__ int s_last;
  const Layout& L = a.lay;
  const int s = blockIdx.x, h = blockIdx.y;
  const int bh = (a.first_seq + s) * L.Hkv + h;
  const int tid = threadIdx.x;
  int t0, t1;
  if (!seq_bounds(a, s, t0, t1) || t1 == t0) return;
  if (L.plan[(size_t)h * L.plan_stride + chunk_id(t0, 0, s)] < 0) return;  // the plan failed
  if (tid == 0) s_last = -1;
  __syncthreads();
  const int nch = ceil_div(t1 - t0, kPrefillChunk);
  const uint4* opens = L.opens + (size_t)h * L.plan_stride + chunk_id(t0, 0, s);
  for (int cb = nch - kPlanThreads; cb + kPlanThreads > 0; cb -= kPlanThreads) {
    const int c = cb + tid;
    if (c >= 0) {
      const uint4 b = opens[c];
      const int at = b.w ? 127 - __clz(b.w) : b.z ? 95 - __clz(b.z) : b.y ? 63 - __clz(b.y) : b.x ? 31 - __clz(b.x) : -1;
      if (at >= 0) atomicMax(&s_last, t0 + c * kPrefillChunk + at);
    }
    if (__syncthreads_or(s_last >= 0)) break;
  }
  const int last = min(s_last, t1 - 1);  // inside the prompt whatever the words say
  if (tid >= 32) return;
  const int parity = *reinterpret_cast<const volatile int*>(&L.ctl[a.layer * 4]);
  const int n_old = last >= 0 ? 0 : L.seglen[((size_t)a.layer * 2 + parity) * L.NH + bh];
  fill_ring<T, D>(a, h, bh, last >= 0 ? last : t0, t1, n_old);
}

template <typename T, int D>
static cudaError_t launch_prefill(const PrefillArgs& a, cudaStream_t stream) {
  const int max_chunks = ceil_div(a.max_seqlen, kPrefillChunk);
  const size_t plan_smem = (size_t)max(max_chunks, 1) * sizeof(int);
  if (plan_smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(dmc_prefill_plan_kernel<T, D>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)plan_smem);
    if (e != cudaSuccess) return e;
  }
  dmc_prefill_plan_kernel<T, D><<<dim3(a.num_seqs, a.lay.Hkv), kPlanThreads, plan_smem, stream>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (max_chunks > 0) {
    const dim3 grid(max_chunks, a.lay.Hkv, a.num_seqs);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(kScanThreads);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = a.lay.window > 0 ? cudaLaunchKernelEx(&cfg, dmc_prefill_scan_kernel<T, D, true>, a)
                         : cudaLaunchKernelEx(&cfg, dmc_prefill_scan_kernel<T, D, false>, a);
    if (e != cudaSuccess) return e;
    e = cudaGetLastError();
  }
  if (e == cudaSuccess && a.lay.window > 0) {
    dmc_prefill_ring_kernel<T, D><<<dim3(a.num_seqs, a.lay.Hkv), kPlanThreads, 0, stream>>>(a);
    e = cudaGetLastError();
  }
  return e;
}

cudaError_t prefill_launch(const Layout& L, int layer, int first_seq, int num_seqs, const void* q,
                           long long q_tok, long long q_head, const void* k, const void* v,
                           const int* cu, int total_tokens, int max_seqlen, float* carry,
                           float* weights, cudaStream_t stream) {
  PrefillArgs a;
  a.lay = L;
  a.layer = layer;
  a.first_seq = first_seq;
  a.num_seqs = num_seqs;
  a.q = static_cast<const char*>(q);
  a.q_tok = q_tok;
  a.q_head = q_head;
  a.k = static_cast<const char*>(k);
  a.v = static_cast<const char*>(v);
  a.cu = cu;
  a.total_tokens = total_tokens;
  a.max_seqlen = max_seqlen;
  a.carry = carry;
  a.weights = weights;
  if (L.esize == 4 && L.D == 64) return launch_prefill<float, 64>(a, stream);
  if (L.esize == 4 && L.D == 128) return launch_prefill<float, 128>(a, stream);
  if (L.esize == 2 && L.D == 64) return launch_prefill<__nv_bfloat16, 64>(a, stream);
  if (L.esize == 2 && L.D == 128) return launch_prefill<__nv_bfloat16, 128>(a, stream);
  return cudaErrorInvalidValue;
}

}  // namespace dmc

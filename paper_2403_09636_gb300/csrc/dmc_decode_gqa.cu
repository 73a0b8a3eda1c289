// DMC decode step for grouped-query attention on tensor cores (bf16).
//
// The paper combines DMC with the 8x grouped-query attention of Llama 2 70B
// (one decision and one compressed cache per KV head, shared by the G query
// heads of its group). Here one warp handles all G <= 8 queries of a KV head,
// so every slot page is read once for the whole group and the scores and the
// value sums become small matrix products on the tensor cores
// (mma.sync m16n8k16, bf16 in, fp32 accumulate):
//
//   S  = Q K^T     M = 16 query rows (the G queries, the rest zero),
//                  N = 8 slots, K = 16 dims;
//   O^T += V^T P^T M = 16 dims, N = 8 queries, K = 16 slots.
//
// The score fragment (row = query, cols = 2 slots) is exactly the B operand
// layout of the second product, so P never leaves registers and the output
// accumulator O^T has no padded rows. P enters it twice, rounded to bf16 and what that
// rounding left, with the V fragments of one load: rounded once, the outputs' error
// depended on how many slots were the maximum of a step (their weight is exactly one),
// so that longer steps and fewer workers raised it by 1-4 % (rms against 64 bits, of
// outputs that round to bf16 themselves, 8 x 2000 tokens at 2x, G = 8: relative 2.15e-3
// with 16-slot steps, 2.18e-3 with 32, 1.79e-3 so). It adds 16 products to a page's 48
// (70B batch 64: 89.7 -> 92.2 us per launch; interleaved or in a pass of its own the
// same). K and V move in tiles of 32 slots (a
// page): each lane cp.asyncs 16-byte chunks into a per-warp ring in shared
// memory, chunks XOR-swizzled by row so that ldmatrix (and ldmatrix.trans for
// V) reads without bank conflicts; rows past the head's length are
// zero-filled. The softmax is online in the log2 domain, per query row.
//
// Work split, owner update, split-head combine, double-buffered slot counts,
// programmatic dependent launch and the walk over several layers in one launch
// follow the MHA kernel (dmc_decode.cu): units are a head's pages plus one
// owner unit, split evenly over all warps; the owner applies Algorithm 1 once
// per KV head, and the new row enters the attention as a one-row tile; a head
// cut between warps is merged by the last warp to finish it, in worker order.
#include <math.h>

#include "dmc_internal.cuh"
#include "dmc_split.cuh"

namespace dmc {

constexpr int kGWarps = kGqaWarpsPerBlock;  // workers per block
constexpr int kGThreads = kGWarps * 32;
// Tiles per warp ring (all but one in flight): a cache with so many heads that the
// unit prefixes leave no room for three takes two. A page per softmax step halves
// the shuffles, exponentials of the running maximum and accumulator rescales of the
// 16-slot tiles before (70B batch 64: 93.8 -> 90.2 us per launch). Warps x ring,
// one block per SM: 4 x 3 90.2, 3 x 4 113.1, 5 x 2 91.3, 6 x 2 91.8.
constexpr int kGRing = 3;
constexpr int kGRingMany = 2;
constexpr int kTile = 32;     // slots per tile (a page), worked as two halves of 16
constexpr int kHalf = 16;
constexpr int kGWindow = 64;  // page units per warp window
constexpr int kGMaxBlocks = 256;
constexpr int kGMaxQueries = 8;
constexpr int kGHeadWindow = 32;  // KV heads whose gates a warp holds in its lanes
static_assert(kGMaxBlocks * kGWarps * 2 <= kGqaWorkerStates, "partials hold two states per worker");

enum : int { kGFlagAcc = 1, kGFlagNaN = 2 };

struct GqaArgs {
  Layout lay;
  int layer0, nlayers;  // layers [layer0, layer0 + nlayers), walked in order
  const char* q;        // layer layer0 + i at q + i * q_ls bytes: [B][Hq][D]
  const char* k;        // at k + i * kv_ls: [B][Hkv][D]
  const char* v;
  char* out;            // at out + i * q_ls: [B][Hq][D]
  long long q_ls, kv_ls;
  bool overlap;         // launched as a programmatic dependent
};

template <int D, int RING>
struct GqaGeom {
  static constexpr int ROW = D * 2;               // bf16 row bytes
  static constexpr int CPR = ROW / 16;            // 16-byte chunks per row
  static constexpr int KT = D / 16;               // k-steps of S = m-tiles of O^T
  static constexpr int TILE = 2 * kTile * ROW;    // 32 K rows then 32 V rows
  static constexpr int WRING = RING * TILE;
  static constexpr int WWIN = 2 * kGWindow * 4;   // page ids, rows to copy
  static constexpr int WARP_BYTES = WRING + WWIN;
  static constexpr int MISC = 64;
  // two unit prefixes (by layer parity)
  static size_t smem_bytes(int nh) {
    return (size_t)kGWarps * WARP_BYTES + MISC + (size_t)2 * (nh + 1) * 4;
  }
};

// Byte offset of 16-byte chunk c of a row inside a 16-row block; the chunk
// index is XOR-ed with the row so that 8 consecutive rows hit 8 bank groups.
__device__ __forceinline__ uint32_t swz(int row, int c, int row_bytes) {
  return (uint32_t)(row * row_bytes + ((c ^ (row & 7)) << 4));
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&h);
}
// What pack_bf16x2 rounded off, as bf16 in turn: the pair's sum holds 16 bits or more of
// each value.
__device__ __forceinline__ uint32_t pack_rest(float lo, float hi, uint32_t packed) {
  return pack_bf16x2(lo - __uint_as_float(packed << 16), hi - __uint_as_float(packed & 0xffff0000u));
}

// Workers of a layer of U units over nh heads, on a grid of `warps` warps. A
// worker streams a page unit in about kUnitCost times what the merge of a split
// head spends per contributor, so a head of n units is done soonest with about
// sqrt(kUnitCost n) contributors; more units than that per worker are only taken
// when the grid has no more warps. Measured for 64 query heads over 8 KV heads,
// 2048 tokens at 2x, us per launch at batch 1 / 4: 80.6 / 74.0 with every warp a
// worker and a serial merge; with the merge below and kUnitCost 1, 2, 3, 5: 18.2 /
// 21.9, 17.7 / 20.3, 18.4 / 23.2, 21.0 / 26.0. Below two units per worker it is one: 1.2,
// say, made two of some and one of the others (16 query heads over 8, d 64, batch 16,
// 40-64 slots: 13 us per launch, 8.5-9 with one unit each, 11-12 with every warp a worker
// and the serial merge).
constexpr float kUnitCost = 2.f;
__device__ __forceinline__ int gqa_workers(long long U, int nh, int warps) {
  const float per_head = (float)U / (float)nh;
  const float best = sqrtf(per_head * (1.f / kUnitCost)), per_worker = best < 2.f ? 1.f : best;
  const int want = max(1, (int)((float)U / per_worker));
  return (int)min((long long)min(want, warps), U);
}

// The last contributor of a split head merges the nc workers' states (wf ..
// wf + nc - 1, in worker order) and writes the group's output rows. Lane (g =
// lane / 4, t = lane % 4) sums query g over the dims 8 i + 2 t, + 1 (i = 0 ..
// D / 8 - 1: four lanes read 32 bytes of a row), two contributors' loads in
// flight (four in flight: 18.9 us instead of 20.1 at batch 1, but the registers
// they take spill in the caller, 99.1 against 94.4 us per 70B batch-64 launch).
template <int D>
__device__ __noinline__ void combine_gqa(const float* partials, int wf, int first_off, int nc, int G,
                                         int lane, __nv_bfloat16* ob) {
  constexpr int NB = 2, V2 = D / 8;
  const int g = lane >> 2, t = lane & 3;
  const bool on = g < G;
  const size_t PS = (size_t)G * (D + 2);
  const float* row = partials + (size_t)(on ? g : 0) * (D + 2);
  auto state = [&](int i) { return row + (size_t)(2 * (wf + i) + (i == 0 ? first_off : 0)) * PS; };
  float2 ml[NB], v[NB][V2];
  auto load = [&](int i0) {
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const float2* p = reinterpret_cast<const float2*>(state(min(i0 + b, nc - 1)));
      ml[b] = __ldcg(p);
#pragma unroll
      for (int i = 0; i < V2; ++i) v[b][i] = __ldcg(p + 1 + 4 * i + t);
    }
  };
  float Mc = -INFINITY;
#pragma unroll 4
  for (int i = t; i < nc; i += 4) Mc = fmaxf(Mc, __ldcg(state(i)));
  Mc = fmaxf(Mc, __shfl_xor_sync(0xffffffffu, Mc, 1));
  Mc = fmaxf(Mc, __shfl_xor_sync(0xffffffffu, Mc, 2));
  float Lc = 0.f;
  float2 o[V2];
#pragma unroll
  for (int i = 0; i < V2; ++i) o[i] = make_float2(0.f, 0.f);
  for (int i0 = 0; i0 < nc; i0 += NB) {
    load(i0);
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      if (i0 + b >= nc) break;
      const float w = (ml[b].x == -INFINITY) ? 0.f : exp2f(ml[b].x - Mc);
      Lc = fmaf(ml[b].y, w, Lc);
#pragma unroll
      for (int i = 0; i < V2; ++i) {
        o[i].x = fmaf(v[b][i].x, w, o[i].x);
        o[i].y = fmaf(v[b][i].y, w, o[i].y);
      }
    }
  }
  if (!on) return;
  const float inv = 1.f / Lc;
#pragma unroll
  for (int i = 0; i < V2; ++i)
    *reinterpret_cast<uint32_t*>(ob + (size_t)g * D + 8 * i + 2 * t) = pack_bf16x2(o[i].x * inv, o[i].y * inv);
}

// kWin: the cache uses the window-grouping approximation (L.window > 0)
template <int D, bool kWin, int RING>
__global__ void __launch_bounds__(kGThreads, 1) dmc_decode_gqa_kernel(const GqaArgs a) {
  using G_ = GqaGeom<D, RING>;
  constexpr int ROW = G_::ROW, CPR = G_::CPR, KT = G_::KT;
  using CK = Chunk<__nv_bfloat16>;
  extern __shared__ __align__(128) unsigned char smem[];

  const Layout& L = a.lay;
  const int G = L.G;
  const int NH = L.NH;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, t = lane & 3;  // mma fragment row / column pair
  unsigned char* ring = smem + (size_t)warp * G_::WARP_BYTES;
  int* wpid = reinterpret_cast<int*>(ring + G_::WRING);
  int* wrws = wpid + kGWindow;
  int* misc = reinterpret_cast<int*>(smem + (size_t)kGWarps * G_::WARP_BYTES);
  int* Ubuf = misc + G_::MISC / 4;  // the unit prefixes of layers li (buffer li & 1)
  volatile int* s_done = misc + 8;  // [2]: warps of the block done with the layer in buffer b
  volatile int* s_tag = misc + 10;  // [2]: 1 + the index li of the layer whose prefix buffer b holds

  // Walking several layers, a warp goes on to the next layer as soon as its own
  // part of the current one is done: the block builds the first two layers'
  // unit prefixes here, and the last of its warps to leave layer li builds
  // layer li + 2's into the buffer it frees.
  scan_units(Ubuf, misc, L.ctl + a.layer0 * 4, L.lengths + (size_t)a.layer0 * 2 * NH, NH, NH, 1);
  if (a.nlayers > 1)
    scan_units(Ubuf + NH + 1, misc, L.ctl + (a.layer0 + 1) * 4,
               L.lengths + (size_t)(a.layer0 + 1) * 2 * NH, NH, NH, 1);
  if (tid == 0) {
    s_done[0] = s_done[1] = 0;
    s_tag[0] = 1;
    s_tag[1] = 2;
  }
  __syncthreads();

  for (int li = 0; li < a.nlayers; ++li) {
  const int layer = a.layer0 + li;
  const char* qL = a.q + (size_t)li * a.q_ls;
  const char* kL = a.k + (size_t)li * a.kv_ls;
  const char* vL = a.v + (size_t)li * a.kv_ls;
  char* outL = a.out + (size_t)li * a.q_ls;
  int* ctl = L.ctl + layer * 4;
  const int parity = *reinterpret_cast<volatile int*>(&ctl[0]);
  const int* len_cur = L.lengths + ((size_t)layer * 2 + parity) * NH;
  int* len_nxt = L.lengths + ((size_t)layer * 2 + (parity ^ 1)) * NH;
  int* ptab = L.page_table + (size_t)layer * NH * L.MPH;
  float* partials = L.partials + (size_t)layer * L.partials_layer_stride;
  const int ub = li & 1;
  int* U = Ubuf + ub * (NH + 1);

  // ---------------------------------------------------------------- prologue
  bool have_units = true;
  if (li > 0) {
    // this layer's unit prefix (built by the block's last warp to leave layer
    // li - 2); a warp that gives up waiting does no work in the layer
    const uint64_t w0 = globaltimer_ns();
    while (s_tag[ub] != li + 1) {
      __nanosleep(32);
      if (globaltimer_ns() - w0 > kWaitLimitNs) {
        if (lane == 0) atomicOr(L.error, DMC_FAULT_WAIT_TIMEOUT);
        have_units = false;
        break;
      }
    }
    have_units = __all_sync(0xffffffffu, have_units);
    __threadfence_block();  // the prefix is read after its tag
  }
  const long long Utot = have_units ? U[NH] : 0;
  // The workers of the layer: every warp, or fewer when a head would then be
  // cut into so many parts that merging them takes longer than streaming them
  // (gqa_workers); those are spread over the blocks so that every SM takes part.
  const int NWG = (int)gridDim.x * kGWarps;
  const int NW = have_units ? gqa_workers(Utot, NH, NWG) : NWG;
  const int wid = NW < NWG ? warp * (int)gridDim.x + (int)blockIdx.x : (int)blockIdx.x * kGWarps + warp;
  const bool works = have_units && wid < NW;
  const int u0 = works ? (int)range_start(wid, Utot, NW) : 0;
  const int u1 = works ? (int)range_start(wid + 1, Utot, NW) : 0;
  const int n = u1 - u0;
  const uint32_t ring_s = smem_u32(ring);

  // page window: page id and rows to copy of units [pb, pb + kGWindow)
  int pb = u0;
  auto load_window = [&](int first) {
    pb = first;
    __syncwarp();
    for (int i = lane; i < kGWindow; i += 32) {
      const int u = first + i;
      int pid = 0, rws = 0;
      if (u < u1) {
        const int hv = head_of_unit(U, NH, u);
        const int j = u - U[hv];
        if (j < U[hv + 1] - U[hv] - 1) {
          pid = ptab[(size_t)hv * L.MPH + j];
          rws = min(kPage, len_cur[hv] - j * kPage);
        }
      }
      wpid[i] = pid;
      wrws[i] = rws;
    }
    __syncwarp();
  };

  // issue cursor: tile it of unit u0 + ik; an owner unit reserves one tile
  int ik = 0, it = 0, itn = -1, islot = 0;
  auto issue_next = [&]() {
    while (ik < n) {
      const int iu = u0 + ik;
      if (iu - pb >= kGWindow) load_window(iu);
      if (itn < 0) {
        const int rws = wrws[iu - pb];
        itn = rws > 0 ? ceil_div(rws, kTile) : 1;
      }
      if (it < itn) break;
      ++ik;
      it = 0;
      itn = -1;
    }
    if (ik < n) {
      const int iu = u0 + ik;
      const int rws = wrws[iu - pb];
      if (rws > 0) {
        const char* pg = L.pages + (size_t)wpid[iu - pb] * L.page_bytes;
        const uint32_t dst = ring_s + islot * G_::TILE;
        // the rows past the head's end are zero-filled up to a half's end; a half
        // without a row is neither copied nor worked
        const char* src = pg + (size_t)(lane / CPR) * ROW + (lane % CPR) * 16;
#pragma unroll
        for (int i = 0; i < 2 * kTile * CPR / 32; ++i) {
          constexpr int RPI = 32 / CPR;  // rows per iteration
          const int which = i * RPI / kTile, r0 = i * RPI % kTile;  // 0: K, 1: V
          if (r0 < kHalf || rws > kHalf) {
            const int r = r0 + lane / CPR;
            const bool valid = r < rws;
            cp_async16_zfill(dst + which * kTile * ROW + swz(r, lane % CPR, ROW),
                             valid ? src + (size_t)which * kPage * ROW + (size_t)r0 * ROW : pg, valid);
          }
        }
      }
      ++it;
    }
    cp_async_commit();  // one group per call, possibly empty, on every lane
    islot = (islot + 1 == RING) ? 0 : islot + 1;
  };

  int vh = 0, page0 = -1;  // the current head; the last slot's page if the first unit is an owner
  if (n > 0) {
    load_window(u0);
    for (int s = 0; s < RING - 1; ++s) issue_next();
    vh = head_of_unit(U, NH, u0);
    const int last0 = len_cur[vh] - 1;
    // overlapping the kernel before: an owner unit's old row and z come to L2 before
    // the grid wait is over (64 query heads over 8, us per launch, with the new row
    // and z requested before the reserved tile: batch 1 18.3 -> 17.7, 4 21.8 -> 20.3,
    // 64 90.4 -> 89.7)
    if (a.overlap && U[vh + 1] == u0 + 1 && last0 >= 0) {
      page0 = ptab[(size_t)vh * L.MPH + last0 / kPage];
      const char* row = L.pages + (size_t)page0 * L.page_bytes + (size_t)(last0 % kPage) * ROW;
      constexpr int NL = ROW / 128;
      if (lane < 2 * NL)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(row + (lane < NL ? 0 : kPage * ROW) + lane % NL * 128));
      else if (lane == 2 * NL)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(L.z + (size_t)page0 * kPage + last0 % kPage));
    }
  }

  // q, k, v and the slots this launch writes are touched only after this point
  if (li == 0) {
    griddep_wait();
    griddep_launch_dependents();
  }

  if (n > 0) {
    // lane i holds the gates of KV head hb + i
    int hb = 0, t_len = 0, t_flags = 0;
    float t_omega = 0.f;
    auto load_heads = [&](int first) {
      hb = first;
      const int hv = first + lane;
      t_len = 0;
      t_flags = 0;
      t_omega = 0.f;
      if (hv < NH && U[hv] < u1) {
        const int b = hv / L.Hkv, h = hv % L.Hkv;
        const int len = len_cur[hv];
        const float x = __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(kL)[(size_t)hv * D]);
        float qs = 0.f;
        for (int gg = 0; gg < G; ++gg)
          qs += __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(
              qL)[((size_t)b * L.Hq + (size_t)h * G + gg) * D]);
        t_len = len;
        // alpha = round(sigmoid(k[0])) = [k[0] >= 0]; an empty head always appends
        t_flags = ((x >= 0.f && len > 0) ? kGFlagAcc : 0) | ((x != x) ? kGFlagNaN : 0);
        t_omega = sigmoidf_(qs / (float)G);  // omega = sigmoid(mean of the group's q[0])
      }
    };

    // A fragments of the group's queries: row g = query g (zero for g >= G),
    // q[0] removed. qa[kk][0]: dims kk*16 + 2t, +1; qa[kk][1]: dims + 8.
    auto load_q = [&](int hv, uint32_t (*qa)[2]) {
      const int b = hv / L.Hkv, h = hv % L.Hkv;
      const uint32_t* qrow = reinterpret_cast<const uint32_t*>(
          qL + ((size_t)b * L.Hq + (size_t)h * G + (g < G ? g : 0)) * ROW);
#pragma unroll
      for (int kk = 0; kk < KT; ++kk) {
        qa[kk][0] = g < G ? __ldg(qrow + kk * 8 + t) : 0u;
        qa[kk][1] = g < G ? __ldg(qrow + kk * 8 + 4 + t) : 0u;
      }
    };
    uint32_t qa[KT][2], qn[KT][2];
    load_q(vh, qn);  // with the gates: one round trip to memory after the grid wait
    load_heads(vh);

    const float qscale = 1.4426950408889634f / sqrtf((float)D);  // log2(e) / sqrt(d_h)
    float o[KT][4];
    float m = -INFINITY, lsum = 0.f;
#pragma unroll
    for (int mt = 0; mt < KT; ++mt) o[mt][0] = o[mt][1] = o[mt][2] = o[mt][3] = 0.f;
    int len_old = 0, flags = 0, cslot = 0;
    float omega = 0.f;

    // one tile of up to 32 slots, the first `valid` of them attended (two: its
    // second half holds rows)
    auto do_tile = [&](uint32_t tile, int valid, bool two) {
      const int mi = lane >> 3, r = lane & 7;
      const int srow = (mi >> 1) * 8 + r;
      float s[8];  // scores of query g at slots 2t, 2t + 1, 8 + 2t, 9 + 2t of each half
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        float sc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
        if (hf == 0 || two) {
#pragma unroll
          for (int kk = 0; kk < KT; ++kk) {
            uint32_t b00, b01, b10, b11;
            ldmatrix_x4(tile + hf * kHalf * ROW + swz(srow, kk * 2 + (mi & 1), ROW), b00, b01, b10, b11);
            mma_bf16_16816(sc[0], qa[kk][0], 0u, qa[kk][1], 0u, b00, b01);
            mma_bf16_16816(sc[1], qa[kk][0], 0u, qa[kk][1], 0u, b10, b11);
          }
        }
        const int left = valid - hf * kHalf - 2 * t;
        s[4 * hf] = left > 0 ? sc[0][0] * qscale : -INFINITY;
        s[4 * hf + 1] = left > 1 ? sc[0][1] * qscale : -INFINITY;
        s[4 * hf + 2] = left > 8 ? sc[1][0] * qscale : -INFINITY;
        s[4 * hf + 3] = left > 9 ? sc[1][1] * qscale : -INFINITY;
      }
      float mx = fmaxf(fmaxf(fmaxf(s[0], s[1]), fmaxf(s[2], s[3])), fmaxf(fmaxf(s[4], s[5]), fmaxf(s[6], s[7])));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
      const float mn = fmaxf(m, mx);
      const float corr = (m == -INFINITY) ? 0.f : exp2f(m - mn);
      float p[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) p[i] = (s[i] == -INFINITY) ? 0.f : exp2f(s[i] - mn);
      float ps = ((p[0] + p[1]) + (p[2] + p[3])) + ((p[4] + p[5]) + (p[6] + p[7]));
      ps += __shfl_xor_sync(0xffffffffu, ps, 1);
      ps += __shfl_xor_sync(0xffffffffu, ps, 2);
      lsum = lsum * corr + ps;
      m = mn;
      // output columns of this lane are queries 2t and 2t + 1
      const float2 c2 = make_float2(__shfl_sync(0xffffffffu, corr, 8 * t), __shfl_sync(0xffffffffu, corr, 8 * t + 4));
      const uint32_t p00 = pack_bf16x2(p[0], p[1]), p01 = pack_bf16x2(p[2], p[3]);
      const uint32_t p10 = pack_bf16x2(p[4], p[5]), p11 = pack_bf16x2(p[6], p[7]);
      const uint32_t r00 = pack_rest(p[0], p[1], p00), r01 = pack_rest(p[2], p[3], p01);
      const uint32_t vtile = tile + kTile * ROW;
#pragma unroll
      for (int mt = 0; mt < KT; ++mt) {
        const float2 lo = mul2(make_float2(o[mt][0], o[mt][1]), c2), hi = mul2(make_float2(o[mt][2], o[mt][3]), c2);
        o[mt][0] = lo.x;
        o[mt][1] = lo.y;
        o[mt][2] = hi.x;
        o[mt][3] = hi.y;
        uint32_t a0, a1, a2, a3;
        ldmatrix_x4_trans(vtile + swz(srow, mt * 2 + (mi & 1), ROW), a0, a1, a2, a3);
        mma_bf16_16816(o[mt], a0, a1, a2, a3, p00, p01);
        mma_bf16_16816(o[mt], a0, a1, a2, a3, r00, r01);
      }
      if (two) {
        const uint32_t r10 = pack_rest(p[4], p[5], p10), r11 = pack_rest(p[6], p[7], p11);
#pragma unroll
        for (int mt = 0; mt < KT; ++mt) {
          uint32_t a0, a1, a2, a3;
          ldmatrix_x4_trans(vtile + kHalf * ROW + swz(srow, mt * 2 + (mi & 1), ROW), a0, a1, a2, a3);
          mma_bf16_16816(o[mt], a0, a1, a2, a3, p10, p11);
          mma_bf16_16816(o[mt], a0, a1, a2, a3, r10, r11);
        }
      }
    };

    for (int k = 0; k < n; ++k) {
      const int u = u0 + k;
      while (U[vh + 1] <= u) ++vh;
      const int hu0 = U[vh], hend = U[vh + 1], nU = hend - hu0, j = u - hu0;
      const bool owner = (j == nU - 1);
      if (k == 0 || j == 0) {
        if (vh - hb >= kGHeadWindow) load_heads(vh);
        const int src = vh - hb;
        len_old = __shfl_sync(0xffffffffu, t_len, src);
        flags = __shfl_sync(0xffffffffu, t_flags, src);
        omega = __shfl_sync(0xffffffffu, t_omega, src);
#pragma unroll
        for (int kk = 0; kk < KT; ++kk) {
          qa[kk][0] = qn[kk][0];
          qa[kk][1] = qn[kk][1];
        }
        if (t == 0) qa[0][0] &= 0xffff0000u;  // q[0] (low half of dims 0, 1) is the gate
        if (hend < u1) load_q(vh + 1, qn);    // the next head's queries, ahead of use
      }
      const int accum = flags & kGFlagAcc;
      if (!owner) {
        const int rows_copied = min(kPage, len_old - j * kPage);
        const int rows = min(kPage, len_old - accum - j * kPage);  // the merged slot is excluded
        const int ntl = ceil_div(rows_copied, kTile);
        for (int tl = 0; tl < ntl; ++tl) {
          issue_next();
          cp_async_wait<RING - 1>();
          __syncwarp();  // every lane's copies of this tile have landed
          do_tile(ring_s + cslot * G_::TILE, max(0, min(kTile, rows - tl * kTile)), rows_copied - tl * kTile > kHalf);
          cslot = (cslot + 1 == RING) ? 0 : cslot + 1;
        }
      } else {
        // Algorithm 1 on the KV head's new token, once for the group: lanes
        // 0..CPR-1 build the key row, lanes CPR..2*CPR-1 the value row, 8
        // dims each, in fp32, rounded to bf16.
        const bool is_v = lane >= CPR;
        const int c = is_v ? lane - CPR : lane;
        const bool act = lane < 2 * CPR;
        // When this warp has just streamed the head's last page (unit u - 1),
        // the old last row is in the tile it consumed last: read it before
        // the issue below reuses that ring slot. The issue window may still
        // hold that page's id.
        const bool ring_row = !kWin && accum && k > 0 && j > 0;
        uint4 oraw = make_uint4(0, 0, 0, 0);
        if (ring_row && act) {
          const int ps = (cslot == 0 ? RING : cslot) - 1;
          oraw = *reinterpret_cast<const uint4*>(smem + (ring_s - smem_u32(smem)) + ps * G_::TILE +
                                                 (is_v ? kTile * ROW : 0) + swz((len_old - 1) % kTile, c, ROW));
        }
        // the new row, the last slot's page and its z are requested before the wait
        // for the reserved tile
        uint4 iraw = make_uint4(0, 0, 0, 0);
        if (act) iraw = __ldg(reinterpret_cast<const uint4*>((is_v ? vL : kL) + (size_t)vh * ROW + c * 16));
        int tgt = -1;
        if (accum || len_old % kPage != 0) {
          const int up = u - 1;
          tgt = (k > 0 && j > 0 && up >= pb && up - pb < kGWindow) ? wpid[up - pb]
                : k == 0 && page0 >= 0 ? page0
                                       : ptab[(size_t)vh * L.MPH + (len_old - 1) / kPage];
        }
        float zold = 0.f;
        if (!kWin && accum) zold = L.z[(size_t)tgt * kPage + (len_old - 1) % kPage];
        issue_next();
        cp_async_wait<RING - 1>();
        __syncwarp();  // the reserved tile's slot is free
        const uint32_t tile = ring_s + cslot * G_::TILE;
        cslot = (cslot + 1 == RING) ? 0 : cslot + 1;
        // window grouping: the slot is the mean of the segment's last W tokens,
        // the W - 1 before this one being in the head's ring
        const int W = kWin ? L.window : 0;
        const int Wm = kWin ? L.window : 1;
        int n_old = 0, nwin = 0;  // tokens before this one, of them in the window
        const char* ring = nullptr;
        const float* ring_w = nullptr;
        float znew = omega;
        if (W > 0) {
          ring = L.ring + ((size_t)layer * NH + vh) * W * 2 * ROW;
          ring_w = L.ring_w + ((size_t)layer * NH + vh) * W;
          if (accum) {
            n_old = L.seglen[((size_t)layer * 2 + parity) * NH + vh];
            nwin = min(n_old, W - 1);
            for (int e = 0; e < nwin; ++e) znew += ring_w[(n_old - 1 - e) % Wm];
          }
        } else if (accum) {
          znew = zold + omega;
        }
        uint4 nrow = make_uint4(0, 0, 0, 0);
        if (act) {
          float in[8], nw[8];
          CK::unpack(iraw, in);
          if (!is_v && c == 0) in[0] = 0.f;  // k[0] <- 0 (Algorithm 1)
          if (W > 0) {
#pragma unroll
            for (int e = 0; e < 8; ++e) nw[e] = in[e] * omega;
            for (int e2 = 0; e2 < nwin; ++e2) {
              const int pos = (n_old - 1 - e2) % Wm;
              float old[8];
              CK::unpack(*reinterpret_cast<const uint4*>(ring + (size_t)pos * 2 * ROW + (is_v ? ROW : 0) + c * 16), old);
              const float w = ring_w[pos];
#pragma unroll
              for (int e = 0; e < 8; ++e) nw[e] = fmaf(w, old[e], nw[e]);
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) nw[e] /= znew;
            // the new token joins the ring at entry n_old % W
            char* re = L.ring + ((size_t)layer * NH + vh) * W * 2 * ROW + (size_t)(n_old % Wm) * 2 * ROW;
            *reinterpret_cast<uint4*>(re + (is_v ? ROW : 0) + c * 16) = CK::pack(in);
          } else if (accum) {
            float old[8];
            if (ring_row) {
              CK::unpack(oraw, old);
            } else {
              const char* orow = L.pages + (size_t)tgt * L.page_bytes +
                                 (size_t)(is_v ? kPage : 0) * ROW + (size_t)((len_old - 1) % kPage) * ROW;
              CK::unpack(*reinterpret_cast<const uint4*>(orow + c * 16), old);
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) nw[e] = (old[e] * zold + in[e] * omega) / znew;
          } else {
#pragma unroll
            for (int e = 0; e < 8; ++e) nw[e] = in[e];
          }
          nrow = CK::pack(nw);
        }
        const int slot = accum ? len_old - 1 : len_old;
        bool ok = slot < L.max_slots;
        int page = tgt;
        if (ok && page < 0) {
          if (lane == 0) {
            const unsigned long long id = atomicAdd(L.pool_top, 1ull);
            if (id >= (unsigned long long)L.num_pages) {
              atomicOr(L.error, DMC_FAULT_PAGES_EXHAUSTED);
              page = -1;
            } else {
              page = (int)id;
              ptab[(size_t)vh * L.MPH + slot / kPage] = page;
            }
          }
          page = __shfl_sync(0xffffffffu, page, 0);
        }
        ok = ok && page >= 0;
        if (lane == 0) {
          if (slot >= L.max_slots) atomicOr(L.error, DMC_FAULT_SLOT_CAPACITY);
          if (ok) L.z[(size_t)page * kPage + slot % kPage] = znew;
          len_nxt[vh] = ok ? slot + 1 : len_old;
          if (W > 0) {
            L.ring_w[((size_t)layer * NH + vh) * W + n_old % Wm] = omega;
            L.seglen[((size_t)layer * 2 + (parity ^ 1)) * NH + vh] = n_old + 1;
          }
          if (flags & kGFlagNaN) atomicOr(L.error, DMC_FAULT_NAN_GATE);
        }
        if (ok && act) {
          char* dst = L.pages + (size_t)page * L.page_bytes + (size_t)(is_v ? kPage : 0) * ROW +
                      (size_t)(slot % kPage) * ROW;
          *reinterpret_cast<uint4*>(dst + c * 16) = nrow;
        }
        // the new row is row 0 of a one-row tile; the other value rows are
        // zero so that their zero weights give exact zeros
        unsigned char* tp = smem + (tile - smem_u32(smem));
        for (int x = lane; x < kHalf * CPR; x += 32) {
          const int r = x / CPR, cc = x % CPR;
          *reinterpret_cast<uint4*>(tp + kTile * ROW + swz(r, cc, ROW)) = make_uint4(0, 0, 0, 0);
        }
        __syncwarp();
        if (act) *reinterpret_cast<uint4*>(tp + (is_v ? kTile * ROW : 0) + swz(0, c, ROW)) = nrow;
        __syncwarp();
        do_tile(tile, 1, false);
      }

      if (owner || k == n - 1) {
        // ---- this warp's part of the head is done
        const int b = vh / L.Hkv, h = vh % L.Hkv;
        __nv_bfloat16* ob = reinterpret_cast<__nv_bfloat16*>(outL) + ((size_t)b * L.Hq + (size_t)h * G) * D;
        const int q_lo = 2 * t, q_hi = 2 * t + 1;
        if (hu0 >= u0 && owner) {
          // the whole head was in this warp
          const float l_lo = __shfl_sync(0xffffffffu, lsum, 8 * t);
          const float l_hi = __shfl_sync(0xffffffffu, lsum, 8 * t + 4);
#pragma unroll
          for (int mt = 0; mt < KT; ++mt) {
            const int d0 = mt * 16 + g;
            if (q_lo < G) {
              ob[(size_t)q_lo * D + d0] = __float2bfloat16_rn(o[mt][0] / l_lo);
              ob[(size_t)q_lo * D + d0 + 8] = __float2bfloat16_rn(o[mt][2] / l_lo);
            }
            if (q_hi < G) {
              ob[(size_t)q_hi * D + d0] = __float2bfloat16_rn(o[mt][1] / l_hi);
              ob[(size_t)q_hi * D + d0 + 8] = __float2bfloat16_rn(o[mt][3] / l_hi);
            }
          }
        } else {
          // publish this warp's partial states (one per query); the last
          // contributor combines
          const int ps = 2 * wid + (hu0 <= u0 ? 0 : 1);
          float* pp = partials + (size_t)ps * G * (D + 2);
          if (t == 0 && g < G) {
            pp[(size_t)g * (D + 2)] = m;
            pp[(size_t)g * (D + 2) + 1] = lsum;
          }
#pragma unroll
          for (int mt = 0; mt < KT; ++mt) {
            const int d0 = mt * 16 + g;
            if (q_lo < G) {
              pp[(size_t)q_lo * (D + 2) + 2 + d0] = o[mt][0];
              pp[(size_t)q_lo * (D + 2) + 2 + d0 + 8] = o[mt][2];
            }
            if (q_hi < G) {
              pp[(size_t)q_hi * (D + 2) + 2 + d0] = o[mt][1];
              pp[(size_t)q_hi * (D + 2) + 2 + d0 + 8] = o[mt][3];
            }
          }
          __threadfence();
          __syncwarp();
          const int wf = worker_of_unit(hu0, Utot, NW);
          const int wl = worker_of_unit(hend - 1, Utot, NW);
          int last = 0;
          if (lane == 0) {
            // every worker in [wf, wl] holds part of the head
            int* cnt = L.counters + (size_t)layer * NH * G + vh;
            const int old = atomicAdd(cnt, 1);
            last = (old == wl - wf);
            if (last) *cnt = 0;
          }
          last = __shfl_sync(0xffffffffu, last, 0);
          if (last) {
            __threadfence();  // every contributor's states are visible to this lane
            // worker wf + i wrote state 2 (wf + i) + 1 if the head starts
            // inside its range (only possible for i = 0), else 2 (wf + i)
            const int first_off = (hu0 > range_start(wf, Utot, NW)) ? 1 : 0;
            combine_gqa<D>(partials, wf, first_off, wl - wf + 1, G, lane, ob);
          }
        }
        m = -INFINITY;
        lsum = 0.f;
#pragma unroll
        for (int mt = 0; mt < KT; ++mt) o[mt][0] = o[mt][1] = o[mt][2] = o[mt][3] = 0.f;
      }
    }
  }
  cp_async_wait<0>();

  // this warp is done with the layer: the grid's last warp out publishes the
  // new slot counts; the block's last warp out builds the prefix of layer
  // li + 2 into the buffer the layer used
  __syncwarp();
  int last_in_block = 0;
  if (lane == 0) {
    __threadfence();
    const int old = atomicAdd(&ctl[1], 1);
    if (old == (int)gridDim.x * kGWarps - 1) {
      ctl[1] = 0;
      ctl[0] = parity ^ 1;
      __threadfence();
    }
    last_in_block = atomicAdd(const_cast<int*>(&s_done[ub]), 1) == kGWarps - 1;
  }
  last_in_block = __shfl_sync(0xffffffffu, last_in_block, 0);
  if (last_in_block) {
    __threadfence_block();  // every warp's reads of the buffer came before its count
    if (li + 2 < a.nlayers)
      scan_units_warp(U, L.ctl + (layer + 2) * 4, L.lengths + (size_t)(layer + 2) * 2 * NH, NH);
    if (lane == 0) {
      s_done[ub] = 0;
      __threadfence_block();
      s_tag[ub] = li + 3;
    }
  }
  }  // layers
}

// Shared memory and blocks per SM with one ring depth (both window variants).
template <int D, int RING>
static cudaError_t setup_ring(int nh, int optin, size_t* smem, int* occ) {
  *smem = GqaGeom<D, RING>::smem_bytes(nh);
  if (*smem > (size_t)optin) return cudaErrorInvalidConfiguration;
  cudaError_t e = cudaFuncSetAttribute(dmc_decode_gqa_kernel<D, false, RING>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)*smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(dmc_decode_gqa_kernel<D, true, RING>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)*smem);
  int o = 0, ow = 0;
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, dmc_decode_gqa_kernel<D, false, RING>, kGThreads, *smem);
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ow, dmc_decode_gqa_kernel<D, true, RING>, kGThreads, *smem);
  if (e != cudaSuccess) return e;
  *occ = min(o, ow);
  return *occ < 1 ? cudaErrorInvalidConfiguration : cudaSuccess;
}

template <int D>
static cudaError_t setup_gqa(const Layout& L, DecodePlan* plan) {
  int dev = 0, sms = 0, optin = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  int occ = 0;
  plan->stages = kGRing;
  plan->warps = kGWarps;
  e = setup_ring<D, kGRing>(L.NH, optin, &plan->smem, &occ);
  if (e == cudaErrorInvalidConfiguration) {
    plan->stages = kGRingMany;
    e = setup_ring<D, kGRingMany>(L.NH, optin, &plan->smem, &occ);
  }
  if (e != cudaSuccess) return e;
  plan->grid = min(sms * occ, kGMaxBlocks);
  const long long max_units = (long long)L.NH * (L.MPH + 1);
  const long long max_blocks = (max_units + kGWarps - 1) / kGWarps;
  if (max_blocks < plan->grid) plan->grid = (int)max_blocks;
  plan->partial_states = 2 * plan->grid * kGWarps * L.G;
  plan->grid_walk = plan->grid;  // one launch shape whatever the layers
  plan->smem_walk = plan->smem;
  if (plan->partial_states > L.partial_cap) return cudaErrorInvalidConfiguration;
  return cudaSuccess;
}

bool gqa_supported(const Layout& L) {
  return L.esize == 2 && L.G >= 2 && L.G <= kGMaxQueries && (L.D == 64 || L.D == 128);
}

cudaError_t gqa_setup(const Layout& L, DecodePlan* plan) {
  if (L.D == 64) return setup_gqa<64>(L, plan);
  if (L.D == 128) return setup_gqa<128>(L, plan);
  return cudaErrorInvalidValue;
}

template <int D>
static cudaError_t launch_gqa(const cudaLaunchConfig_t& cfg, const DecodePlan& plan, const GqaArgs& a) {
  if (plan.stages == kGRing)
    return a.lay.window > 0 ? cudaLaunchKernelEx(&cfg, dmc_decode_gqa_kernel<D, true, kGRing>, a)
                            : cudaLaunchKernelEx(&cfg, dmc_decode_gqa_kernel<D, false, kGRing>, a);
  return a.lay.window > 0 ? cudaLaunchKernelEx(&cfg, dmc_decode_gqa_kernel<D, true, kGRingMany>, a)
                          : cudaLaunchKernelEx(&cfg, dmc_decode_gqa_kernel<D, false, kGRingMany>, a);
}

cudaError_t gqa_launch(const Layout& L, int layer0, int nlayers, const DecodePlan& plan, bool pdl,
                       const void* q, const void* k, const void* v, void* out, cudaStream_t stream) {
  GqaArgs a;
  a.lay = L;
  a.layer0 = layer0;
  a.nlayers = nlayers;
  a.q_ls = (long long)L.B * L.Hq * L.row_bytes;
  a.kv_ls = (long long)L.B * L.Hkv * L.row_bytes;
  a.overlap = pdl;
  a.q = static_cast<const char*>(q);
  a.k = static_cast<const char*>(k);
  a.v = static_cast<const char*>(v);
  a.out = static_cast<char*>(out);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(plan.grid);
  cfg.blockDim = dim3(kGThreads);
  cfg.dynamicSmemBytes = plan.smem;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  cudaError_t e = cudaErrorInvalidValue;
  if (L.D == 64) e = launch_gqa<64>(cfg, plan, a);
  if (L.D == 128) e = launch_gqa<128>(cfg, plan, a);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace dmc

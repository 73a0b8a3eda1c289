// Prompt-phase DMC attention on the fifth-generation tensor cores (tcgen05).
//
// At inference every prompt token attends over the cache as it stands right
// after that token's own update (Eq. attn-softmax; the training mask of
// Sec. 3.2 with binary alpha gives the same pattern): the slots closed before
// the token, plus the slot the token has just merged into or opened, whose
// value at that moment is the running omega-weighted mean of its segment so
// far (Eq. partial-accumulation). With len(i) the slot count after token i,
// query i therefore sees the final values of slots [0, len(i) - 1) and one
// "diagonal" state.
//
// A work item is 256 query rows of one KV head of one sequence, as two query
// tiles of 128 rows; a row is a (token, query head of the group) pair,
// token-major, so a group of G queries shares every K/V tile. One persistent
// CTA per SM, its warps specialised:
//   warps 0-3, 4-7  softmax of query tile 0 / 1, one thread per row
//   warp 8          the tensor-core work of both (one thread issues)
//   warp 9          TMA loads: Q tiles, and a ring of four 32 KB K/V tiles that
//                   both query tiles read
//   warp 10         takes work items from a counter, one ahead of the others, and
//                   prepares them: extents, and per token of the chunk its
//                   decision, omega, slot count and 1 / z (from the scan's weights)
// Per query tile and K/V tile of 128 slots:
//   S = Q K^T          tcgen05.mma kind::f16, M = N = 128, K = head_dim, into TMEM
//   softmax            the row's 128 scores from TMEM, the staircase mask
//                      (slot < len(i) - 1), online softmax in the log2 domain,
//                      P rounded to bf16 and stored over the row's S columns
//   O += P V           tcgen05.mma with P read from TMEM and V as an MN-major B
//                      operand, into TMEM
// The tensor-core warp alternates between the query tiles (P V of tile 0's last
// K/V tile, S of its next, then the same for tile 1), so one's tensor-core work
// runs during the other's softmax. The closed slots come from the cache pages that
// the prefill scan has just written. The diagonal state enters as one more tile
// built from the prompt's k, v rows of the token's 128-token chunk and the
// segment sums the prefill scan recorded at the chunk start ("carry"): its
// score is Q Kraw^T summed with the segment's weights, its value P_d Vraw.
//
// Bound: long prompts by the tensor core (a step of both query tiles is 2 x (S 512
// + P V 512) cycles of MMA; measured ~2,900, the rest being the waits between a P V,
// the S that overwrites its P, and the softmax); short ones by the chain of an
// item's few steps and by HBM. Measured, us of this kernel against the one before it
// (one CTA of 8 warps per 128 rows, two per SM, copies by cp.async, softmax and MMA
// in series; 893 / 3482 / 2726): 7B 4x, 32 x 2048 tokens ~495; 70B 2x, 16 x 4096
// tokens ~1800; one 16384-token prompt in four calls ~1490. What mattered, in order:
// softmax and MMA in warps of their own; one lane issuing under elect.sync (under
// `lane == 0` an MMA took ~100 cycles to issue); no call or wait loop inlined thirty
// times and few unrolled copies (the twelve warps run five different programs, and at
// 100 KB of code they mostly fetched instructions: 7B 0.79 ms, at 65 KB 0.50); P in
// two halves, so that P V starts before the softmax ends. Slower: 64-slot tiles with
// two S buffers per query tile (an MMA of N = 64 costs 49 cycles, of N = 128 65);
// P V of both query tiles before S of both; two MMA warps (they ran in step).
#include <cuda.h>
#include <math.h>
#include <stddef.h>

#include "dmc_internal.cuh"

namespace dmc {

constexpr int kPaRows = 128;     // query rows per tile (M)
constexpr int kPaSlots = 128;    // slots per K/V tile (N of S, K of P V)
constexpr int kPaD = 128;        // head_dim handled by this kernel
constexpr int kPaThreads = 384;  // warp 11 only completes the third warpgroup
constexpr int kPaTileBytes = kPaRows * kPaD * 2;  // 32 KB: [128 rows][256 B]
constexpr int kPaRing = 4;       // K/V tiles in the ring
constexpr int kPaItems = 2;      // work items prepared or worked: with four, CTAs claimed items they reached last
constexpr int kPaMaxSeqs = 768;  // sequences per launch (their item prefix is in shared memory)

struct PaItem {
  int s, h, t0, t1;  // sequence, KV head, the sequence's tokens
  int tok;           // first token of query tile 0 (also where only tile 1 has rows); t0 > t1: no more items
  int base[2];       // slots before the chunk of each query tile
  int nvis[2];       // closed slots that a tile's last row sees; -1: the tile has no rows
  int len_final;
  int pad[6];
};
static_assert(sizeof(PaItem) == 64, "");

// The decisions of a 128-token chunk, and its carried sums
struct PaMeta {
  float om[128];            // omega
  float rz[128];            // 1 / z after the token
  float carry[2 * kPaD];
  unsigned char opened[128];  // slots the chunk has opened up to the token
  signed char seg[128];       // first token of the segment within the chunk, or -1
};

constexpr int kPaStageRow = 80;  // bytes of a row of an epilogue stage: 64 and 16 of padding
struct PaShared {
  unsigned char q[2][kPaTileBytes];
  unsigned char kv[kPaRing][kPaTileBytes];
  unsigned char stage[8][32 * kPaStageRow];
  PaMeta meta[kPaItems][2];  // G = 1: the chunk of each query tile; else [0] for both
  PaItem item[kPaItems];
  int pref[kPaMaxSeqs + 1];
  int wsum[kPaThreads / 32];
  uint32_t tmem;
  int abort;
  uint64_t kv_full[kPaRing], kv_empty[kPaRing];
  uint64_t q_full[2], q_empty[2];
  uint64_t s_full[2], p_full[2][2], o_full[2];  // P in two halves
  uint64_t item_full[kPaItems], item_empty[kPaItems], meta_full[kPaItems];
};
constexpr int kPaSmem = sizeof(PaShared) + 1024;  // + alignment of the tiles to 1024 bytes
static_assert(kPaSmem <= 227 * 1024, "one CTA's shared memory");
static_assert(offsetof(PaShared, stage) % 1024 == 0, "swizzled rows in the stages (pa_value_clipped)");
static_assert(4 * 32 * kPaStageRow >= 16 * kPaD * 2, "16 rows of V in four warps' stages");

struct PrefillAttnArgs {
  Layout lay;
  int layer, first_seq, num_seqs;
  const char* q;   // [total_tokens][Hq][D]
  const int* cu;
  int total_tokens, max_seqlen;
  const float* carry;    // [chunk id][Hkv][2D + 1]
  const float* weights;  // [chunk id][Hkv][128]: omega, its sign bit set where the token opens a slot
  char* out;           // [total_tokens][Hq][D]
  int seq_base;        // this launch's first sequence within the call (chunk ids count sequences)
};

struct PaMaps {
  CUtensorMap q;      // [token][q head][D], box: a query tile's tokens x group x 64 columns
  CUtensorMap k, v;   // [token][KV head][D], box: kPaRawRows tokens x 64 columns
  CUtensorMap pages;  // [page x {K, V}][32 rows][D], box: 32 rows x 64 columns
};

// tokens per box of the raw k, v tiles: the tokens of a work item, at most a chunk
template <int G>
constexpr int kPaRawRows = 2 * kPaRows / G < kPrefillChunk ? 2 * kPaRows / G : kPrefillChunk;

// byte offset of 16-byte chunk j (0..15) of row r in a [128 rows][256 B] tile
// kept as two 128-byte column halves, 128B-swizzled (chunk ^ row % 8)
__device__ __forceinline__ uint32_t pa_swz(int r, int j) {
  return (uint32_t)((j >> 3) * (kPaRows * 128) + r * 128 + (((j & 7) ^ (r & 7)) << 4));
}

// tcgen05 shared-memory matrix descriptor: 128B swizzle, start address, leading
// and stride byte offsets (all in 16-byte units), descriptor version 1
__device__ __forceinline__ uint64_t pa_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

// instruction descriptor, kind::f16: bf16 A and B, fp32 D, M = N = 128;
// b_mn selects an MN-major B operand
__device__ __forceinline__ uint32_t pa_idesc(bool b_mn) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((b_mn ? 1u : 0u) << 16) | ((128u >> 3) << 17) |
         ((128u >> 4) << 24);
}

__device__ __forceinline__ void pa_mma(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc,
                                       bool acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(acc ? 1 : 0)
      : "memory");
}

// the same with A (M x K, bf16 pairs packed in 32-bit columns) read from tensor memory
__device__ __forceinline__ void pa_mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b, uint32_t idesc,
                                          bool acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b), "r"(idesc), "r"(acc ? 1 : 0)
      : "memory");
}

// One lane of a full warp, the same one every time. Unlike a comparison of the
// lane's index it tells the compiler that one lane runs, so that descriptors go
// to the tensor core from uniform registers (see the tensor-core warp).
__device__ __forceinline__ bool pa_elect() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
  return p != 0;
}

// A value that all lanes hold, so that the compiler knows they do: control flow
// and descriptors that depend on it stay on the uniform datapath, which a
// tcgen05.mma takes its operands from (with the values as read from shared
// memory an MMA took 65-100 cycles to issue, whatever its shape).
template <typename T>
__device__ __forceinline__ T pa_uniform(T x) {
  return (T)__shfl_sync(0xffffffffu, x, 0);
}

// 2^x by the SFU (ex2.approx, flushing subnormal results to zero)
__device__ __forceinline__ float pa_ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ void pa_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   bar)
               : "memory");
}

// requests 32 consecutive fp32 columns of this thread's TMEM lane (pa_wait_ld before use)
__device__ __forceinline__ void pa_ld32(uint32_t taddr, float* f) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
      "%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=f"(f[0]), "=f"(f[1]), "=f"(f[2]), "=f"(f[3]), "=f"(f[4]), "=f"(f[5]), "=f"(f[6]),
        "=f"(f[7]), "=f"(f[8]), "=f"(f[9]), "=f"(f[10]), "=f"(f[11]), "=f"(f[12]), "=f"(f[13]),
        "=f"(f[14]), "=f"(f[15]), "=f"(f[16]), "=f"(f[17]), "=f"(f[18]), "=f"(f[19]), "=f"(f[20]),
        "=f"(f[21]), "=f"(f[22]), "=f"(f[23]), "=f"(f[24]), "=f"(f[25]), "=f"(f[26]), "=f"(f[27]),
        "=f"(f[28]), "=f"(f[29]), "=f"(f[30]), "=f"(f[31])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void pa_wait_ld() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void pa_st32(uint32_t taddr, const uint32_t* u) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
      "%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr),
      "r"(u[0]), "r"(u[1]), "r"(u[2]), "r"(u[3]), "r"(u[4]), "r"(u[5]), "r"(u[6]), "r"(u[7]),
      "r"(u[8]), "r"(u[9]), "r"(u[10]), "r"(u[11]), "r"(u[12]), "r"(u[13]), "r"(u[14]), "r"(u[15]),
      "r"(u[16]), "r"(u[17]), "r"(u[18]), "r"(u[19]), "r"(u[20]), "r"(u[21]), "r"(u[22]), "r"(u[23]),
      "r"(u[24]), "r"(u[25]), "r"(u[26]), "r"(u[27]), "r"(u[28]), "r"(u[29]), "r"(u[30]), "r"(u[31])
      : "memory");
}
__device__ __forceinline__ void pa_st16(uint32_t taddr, const uint32_t* u) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(
          taddr),
      "r"(u[0]), "r"(u[1]), "r"(u[2]), "r"(u[3]), "r"(u[4]), "r"(u[5]), "r"(u[6]), "r"(u[7]),
      "r"(u[8]), "r"(u[9]), "r"(u[10]), "r"(u[11]), "r"(u[12]), "r"(u[13]), "r"(u[14]), "r"(u[15])
      : "memory");
}
__device__ __forceinline__ void pa_wait_st() {
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void fence_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// TMA load of one box; elements out of the tensor's range are zero
__device__ __forceinline__ void pa_tma(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cta.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(
          dst),
      "l"(map), "r"(bar), "r"(x), "r"(y), "r"(z)
      : "memory");
}

// asks L2 for a box
__device__ __forceinline__ void pa_prefetch(const CUtensorMap* map, int x, int y, int z) {
  asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];" ::"l"(map), "r"(x), "r"(y), "r"(z)
               : "memory");
}

// multiplies the rows' O (one per lane) by corr
__device__ __forceinline__ void pa_rescale(uint32_t tO, float corr) {
#pragma unroll 1
  for (int c0 = 0; c0 < kPaD; c0 += 32) {
    float f[32];
    uint32_t u[32];
    pa_ld32(tO + c0, f);
    pa_wait_ld();
#pragma unroll
    for (int i = 0; i < 32; ++i) u[i] = __float_as_uint(f[i] * corr);
    pa_st32(tO + c0, u);
  }
}

// O of query tile 0 += P V over the first `sees` rows of V (ring tile rv) alone; its P
// has been announced. One warp. Query tile 1's later tokens may see more of the tile.
// Those rows have weight zero in tile 0, but times a value that is infinite or NaN that
// is not zero, so a call that wrote such a slot comes here. (7B layer call 816 us before
// there was a way to tell, 825 with it and the scan's look at every slot, 879 with the
// rows cut off in every call.) Steps of 16 rows; the last one's, if it is cut, are
// copied, with the rest set to zero, to the
// stages of tile 0's epilogue, which its warps have left.
__device__ __noinline__ void pa_value_clipped(PaShared& sh, uint32_t tmem, int rv, int sees, bool add, bool last) {
  const int lane = threadIdx.x & 31, r0 = sees & ~15;
  unsigned char* cut = sh.stage[0];
#pragma unroll 1
  for (int x = lane; x < 16 * 16 && sees > r0; x += 32) {
    const int r = x >> 4, j = x & 15;
    uint4 v = make_uint4(0, 0, 0, 0);
    if (r0 + r < sees)
      v = *reinterpret_cast<const uint4*>(sh.kv[rv] + (j >> 3) * (kPaRows * 128) + (r0 + r) * 128 + (j & 7) * 16);
    *reinterpret_cast<uint4*>(cut + (j >> 3) * (16 * 128) + r * 128 + (j & 7) * 16) = v;
  }
  fence_async_smem();
  __syncwarp();
  if (pa_elect()) {
    tc_fence_after();
#pragma unroll 1
    for (int r = 0; r < sees; r += 16)
      pa_mma_ts(tmem + 256, tmem + r / 2,
                r + 16 <= sees ? pa_desc(smem_u32(sh.kv[rv]) + r * 128, kPaRows * 128, 1024)
                               : pa_desc(smem_u32(cut), 16 * 128, 1024),
                pa_idesc(true), add || r > 0);
    pa_commit(smem_u32(&sh.o_full[0]));
    if (last) pa_commit(smem_u32(&sh.kv_empty[rv]));
  }
  __syncwarp();
}

template <int G>
__global__ void __launch_bounds__(kPaThreads, 1)
dmc_prefill_attn_kernel(const PrefillAttnArgs a, const __grid_constant__ PaMaps maps) {
  constexpr int D = kPaD;
  constexpr int ROW = D * 2;           // bytes per bf16 row
  constexpr int TT = kPaRows / G;      // tokens per query tile
  constexpr int RAW = kPaRawRows<G>;   // tokens per box of the raw k, v tiles
  extern __shared__ unsigned char smem_raw[];
  PaShared& sh = *reinterpret_cast<PaShared*>(smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u));
  const Layout& L = a.lay;
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // known to be the same in all lanes
  int* ctr = L.ctl + a.layer * 4 + 2;  // [0] the next work item, [1] CTAs done
  volatile int* s_abort = &sh.abort;   // a wait gave up

  // ---- the work items: Hkv x ceil(len / 2 TT) per valid sequence, their
  // exclusive prefix per sequence (2 sequences per thread, one block scan)
  {
    constexpr int PER = (kPaMaxSeqs + kPaThreads - 1) / kPaThreads;
    int cnt[PER], sum = 0;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      const int sq = PER * tid + k;
      cnt[k] = 0;
      if (sq < a.num_seqs) {
        const int t0 = a.cu[sq], t1 = a.cu[sq + 1];
        if (t0 >= 0 && t0 <= t1 && t1 <= a.total_tokens && t1 - t0 <= a.max_seqlen)
          cnt[k] = L.Hkv * ((t1 - t0 + 2 * TT - 1) / (2 * TT));
      }
      sum += cnt[k];
    }
    int incl = sum;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int o = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += o;
    }
    if (lane == 31) sh.wsum[warp] = incl;
    if (tid == 0) {
      for (int i = 0; i < kPaRing; ++i) {
        mbar_init(smem_u32(&sh.kv_full[i]), 1);
        mbar_init(smem_u32(&sh.kv_empty[i]), 1);
      }
      for (int w = 0; w < 2; ++w) {
        mbar_init(smem_u32(&sh.q_full[w]), 1);
        mbar_init(smem_u32(&sh.q_empty[w]), 5);  // the tile's four softmax warps, the MMA warp
        mbar_init(smem_u32(&sh.s_full[w]), 1);
        for (int hf = 0; hf < 2; ++hf) mbar_init(smem_u32(&sh.p_full[w][hf]), 4);  // its softmax warps
        mbar_init(smem_u32(&sh.o_full[w]), 1);
      }
      for (int i = 0; i < kPaItems; ++i) {
        mbar_init(smem_u32(&sh.item_full[i]), 1);
        mbar_init(smem_u32(&sh.item_empty[i]), 10);  // every warp but the one that fills it
        mbar_init(smem_u32(&sh.meta_full[i]), 1);
      }
      fence_mbar_init();
      sh.abort = 0;
    }
    if (warp == 8) {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                       smem_u32(&sh.tmem)),
                   "r"(512));
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    __syncthreads();
    int run = incl - sum;
    for (int w = 0; w < warp; ++w) run += sh.wsum[w];
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      const int sq = PER * tid + k;
      if (sq < a.num_seqs) sh.pref[sq] = run;
      run += cnt[k];
    }
    if (tid == kPaThreads - 1) sh.pref[a.num_seqs] = run;  // the last thread's run is the total
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
  }
  // a programmatic dependent of the scan: what came before reads only cu_seqlens
  griddep_wait();
  const uint32_t tmem = pa_uniform(sh.tmem);
  const int nitems = sh.pref[a.num_seqs];
  const int parity = *reinterpret_cast<volatile int*>(&L.ctl[a.layer * 4]);

  // Every wait but the drains at the end (warp_wait): when one gives up, the warps
  // leave their loops, drain and return. No warp waits for another in any other way
  // until then.
  auto wait = [&](uint64_t* bar, uint32_t ph) -> bool { return warp_wait(smem_u32(bar), ph, s_abort, L.error); };
  auto arrive_warp = [&](uint64_t* bar) {  // one arrival per warp, after all its lanes
    __syncwarp();
    if (lane == 0) mbar_arrive(smem_u32(bar));
  };
  // the K/V tiles of an item: its slot tiles (K, V, K, V, ...), then the raw K
  // tiles and the raw V tiles: one each of the chunk both query tiles lie in, or
  // (G = 1) of each query tile's chunk
  auto slot_tiles = [](int nvis) { return nvis <= 0 ? 0 : (nvis + kPaSlots - 1) / kPaSlots; };
  auto raw_tiles = [](const PaItem& w) { return (G == 1 && w.nvis[0] >= 0 && w.nvis[1] >= 0) ? 2 : 1; };
  auto raw_first = [](const PaItem& w, int t) {  // first token of raw tile t's chunk
    return w.t0 + (w.tok + (t + (w.nvis[0] < 0)) * TT - w.t0) / kPrefillChunk * kPrefillChunk;
  };
  auto raw_end = [](const PaItem& w, int t) {  // one past its last token that counts
    return min(w.tok + (G == 1 ? (t + (w.nvis[0] < 0) + 1) * TT : 2 * TT), w.t1);
  };

  if (warp >= 8) {
  // The softmax warps hold a row of scores each: 208 registers for them, 88 for
  // the others (of 384 x 168 launched: 256 x 208 + 128 x 88 is no more). With 168
  // for all the scores spilled (70B batch 16: 2.61 against 2.50 ms per layer).
  asm volatile("setmaxnreg.dec.sync.aligned.u32 88;");
  if (warp == 10) {
    // ---------------------------------------------------------------- items
    constexpr int NC = G == 1 ? 2 : 1;  // chunks of an item
    int item = blockIdx.x;  // the first without a round trip to the counter
    int turn = 0;
    for (int it = 0;; ++it) {
      const int sl = it % kPaItems;
      if (!wait(&sh.item_empty[sl], ((it / kPaItems) & 1) ^ 1)) break;
      int next = 0;
      if (lane == 0 && item < nitems) next = (int)gridDim.x + atomicAdd(&ctr[0], 1);
      PaItem w;
      w.s = w.h = w.t0 = w.t1 = w.tok = w.len_final = 0;
      w.base[0] = w.base[1] = -1;
      w.nvis[0] = w.nvis[1] = -1;
      if (item >= nitems) {
        w.t0 = 1;
        if (lane == 0) sh.item[sl] = w;
        arrive_warp(&sh.item_full[sl]);
        break;
      }
      int lo = 0, hi = a.num_seqs - 1;  // the sequence: last s with pref[s] <= item
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (sh.pref[mid] <= item) lo = mid; else hi = mid - 1;
      }
      const int per_head = (sh.pref[lo + 1] - sh.pref[lo]) / L.Hkv;
      const int rem = item - sh.pref[lo];
      w.s = lo;
      w.h = rem / per_head;
      const int tile = per_head - 1 - rem % per_head;
      w.t0 = a.cu[lo];
      w.t1 = a.cu[lo + 1];
      w.tok = w.t0 + tile * 2 * TT;
      const int iend = min(w.tok + 2 * TT, w.t1);
      // An item with rows for one query tile only takes the tiles' places in turn, so
      // that its epilogue runs beside the next such item's softmax (32 heads, 48 prompts of
      // 59 tokens in two calls: 191 -> 181 us; 180 with the two CTAs per SM before).
      int only = 0;
      if (w.tok + TT >= w.t1) {
        only = turn;
        turn ^= 1;
        w.tok -= only * TT;
      }
      w.len_final = L.lengths[((size_t)a.layer * 2 + parity) * L.NH + (a.first_seq + lo) * L.Hkv + w.h];
      // lane: tokens 4 lane .. 4 lane + 3 of a chunk
      int op[NC][4], base[NC], a0[NC];
      float om[NC][4];
#pragma unroll
      for (int ci = 0; ci < NC; ++ci) {
        const int c = (w.tok + (G == 1 ? ci : only) * TT - w.t0) / kPrefillChunk;
        a0[ci] = G == 1 && ci < only ? w.t1 : w.t0 + c * kPrefillChunk;
        const int cid = w.t0 / kPrefillChunk + c + a.seq_base + lo;
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
        base[ci] = -1;
        if (a0[ci] < iend) {
          base[ci] = L.plan[(size_t)w.h * L.plan_stride + cid];  // slots before the chunk
          x = reinterpret_cast<const float4*>(a.weights + ((size_t)cid * L.Hkv + w.h) * kPrefillChunk)[lane];
        }
        const float xs[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const bool in = a0[ci] + 4 * lane + k < iend;
          op[ci][k] = in && (__float_as_uint(xs[k]) >> 31);
          om[ci][k] = in ? fabsf(xs[k]) : 0.f;
        }
      }
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        const int ci = G == 1 ? t : 0, tok0 = w.tok + t * TT, tokN = min(tok0 + TT, w.t1);
        int n = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) n += (a0[ci] + 4 * lane + k < tokN) ? op[ci][k] : 0;
        n = __reduce_add_sync(0xffffffffu, n);
        if (t >= only && tok0 < w.t1 && base[ci] >= 0) {
          w.base[t] = base[ci];
          // slots closed before the tile's last token; every slot the scan wrote
          w.nvis[t] = max(0, min(base[ci] + n - 1, w.len_final));
        }
      }
      if (lane == 0) sh.item[sl] = w;
      arrive_warp(&sh.item_full[sl]);
      // ---- per token: omega, slot count, segment and 1 / z. z after token i is
      // the omega sum of i's segment so far: from the segment's opening token, or
      // from the carried sums when no token of the chunk up to i opens a slot (a
      // segmented prefix sum over the chunk).
#pragma unroll
      for (int ci = 0; ci < NC; ++ci) {
        if ((G == 1 ? w.nvis[ci] : only ? w.nvis[1] : w.nvis[0]) < 0) continue;
        PaMeta& M = sh.meta[sl][ci];
        const int cid = w.t0 / kPrefillChunk + (a0[ci] - w.t0) / kPrefillChunk + a.seq_base + lo;
        const float* cg = a.carry + ((size_t)cid * L.Hkv + w.h) * (2 * D + 1);
        float cv[2 * D / 32];
#pragma unroll
        for (int x = 0; x < 2 * D / 32; ++x) cv[x] = cg[x * 32 + lane];
        const float cz = cg[2 * D];
        float z[4], zrun = 0.f;
        int cnt[4], sg[4], run = 0, last = -1;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          zrun = op[ci][k] ? om[ci][k] : zrun + om[ci][k];
          run += op[ci][k];
          if (op[ci][k]) last = 4 * lane + k;
          z[k] = zrun;
          cnt[k] = run;
          sg[k] = last;
        }
        // over the lanes before: openings, the last opening token, and the omega
        // sum back to it
        int ic = run, il = last;
        float iz = zrun;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
          const int oc = __shfl_up_sync(0xffffffffu, ic, off);
          const int ol = __shfl_up_sync(0xffffffffu, il, off);
          const float oz = __shfl_up_sync(0xffffffffu, iz, off);
          if (lane >= off) {
            ic += oc;
            if (il < 0) iz += oz;
            il = max(il, ol);
          }
        }
        int ec = __shfl_up_sync(0xffffffffu, ic, 1), el = __shfl_up_sync(0xffffffffu, il, 1);
        float ez = __shfl_up_sync(0xffffffffu, iz, 1);
        if (lane == 0) {
          ec = 0;
          el = -1;
          ez = 0.f;
        }
        if (el < 0) ez += cz;  // no opening in the chunk so far
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          M.om[4 * lane + k] = om[ci][k];
          M.opened[4 * lane + k] = (unsigned char)(ec + cnt[k]);
          M.seg[4 * lane + k] = (signed char)max(el, sg[k]);
          M.rz[4 * lane + k] = 1.f / (sg[k] < 0 ? z[k] + ez : z[k]);
        }
#pragma unroll
        for (int x = 0; x < 2 * D / 32; ++x) M.carry[x * 32 + lane] = cv[x];
      }
      arrive_warp(&sh.meta_full[sl]);
      item = __shfl_sync(0xffffffffu, next, 0);
    }
  } else if (warp == 9) {
    // ---------------------------------------------------------------- loads
    uint32_t n = 0;            // ring tiles requested
    uint32_t q_par = 0, q_any = 0;  // bit w: parity of query tile w's next Q, whether there was one
    const int oob_page = (int)(2 * L.num_pages);
    for (int it = 0;; ++it) {
      const int sl = it % kPaItems;
      if (!wait(&sh.item_full[sl], (it / kPaItems) & 1)) break;
      const PaItem im = sh.item[sl];
      arrive_warp(&sh.item_empty[sl]);
      if (im.t0 > im.t1) break;
      if (max(im.nvis[0], im.nvis[1]) < 0) continue;  // the plan failed: nothing to do (its fault bit is set)
      const int nvis = max(im.nvis[0], im.nvis[1]);
      const int nslot = slot_tiles(nvis), nraw = raw_tiles(im), ntile = 2 * (nslot + nraw);
      const int* ptab = L.page_table + ((size_t)a.layer * L.NH + (a.first_seq + im.s) * L.Hkv + im.h) * L.MPH;
      const int npages = (nvis + kPage - 1) / kPage;
      int pid = lane < npages ? ptab[lane] : 0;  // page ids of the eight slot tiles from `pid0`
      int pid0 = 0;
      // Q and the raw rows come from HBM: ask L2 for them while the item before
      // still holds the buffers
      if (lane < 4 && im.nvis[lane >> 1] >= 0)
        pa_prefetch(&maps.q, (lane & 1) * 64, im.h * G, im.tok + (lane >> 1) * TT);
#pragma unroll 1
      for (int x = lane; x < 4 * nraw * (kPrefillChunk / RAW); x += 32) {
        const int b = x >> 2, t = b / (kPrefillChunk / RAW);
        const int tau = raw_first(im, t) + b % (kPrefillChunk / RAW) * RAW;
        if (tau < raw_end(im, t)) pa_prefetch(x & 2 ? &maps.v : &maps.k, (x & 1) * 64, im.h, tau);
      }
      bool ok = true;
#pragma unroll 1
      for (int x = 0; x < ntile && ok; ++x) {
        const int i = x >> 1;  // the slot tile, if x < 2 nslot
        const int rs = n % kPaRing;
        ok = wait(&sh.kv_empty[rs], ((n / kPaRing) & 1) ^ 1);
        if (!ok) break;
        const uint32_t bar = smem_u32(&sh.kv_full[rs]), dst = smem_u32(sh.kv[rs]);
        if (lane == 0) mbar_arrive_expect_tx(bar, kPaTileBytes);
        __syncwarp();
        if (i < nslot) {
          if (i - pid0 >= 8) {
            pid0 = i;
            const int p = pid0 * 4 + lane;
            pid = p < npages ? ptab[p] : 0;
          }
          // lane: page lane / 2 of the tile, column half lane % 2
          const int p = i * 4 + (lane >> 1);
          const int id = __shfl_sync(0xffffffffu, pid, ((i - pid0) * 4 + (lane >> 1)) & 31);
          if (lane < 8)
            pa_tma(dst + (lane & 1) * (kPaRows * 128) + (lane >> 1) * (kPage * 128), &maps.pages, bar,
                   (lane & 1) * 64, 0, p < npages ? 2 * id + (x & 1) : oob_page);
        } else {
          // the chunk's rows up to the item's last token, the rest zero
          const int y = x - 2 * nslot, t = y % nraw, which = y / nraw;
          if (lane < 2 * (kPrefillChunk / RAW)) {
            const int b = lane >> 1, tau = raw_first(im, t) + b * RAW;
            pa_tma(dst + (lane & 1) * (kPaRows * 128) + b * (RAW * 128), which ? &maps.v : &maps.k, bar,
                   (lane & 1) * 64, im.h, tau < raw_end(im, t) ? tau : a.total_tokens);
          }
        }
        ++n;
        if (x == 0) {
          // Q, once the item before no longer needs the buffers
#pragma unroll 1
          for (int w = 0; w < 2 && ok; ++w) {
            if ((w ? im.nvis[1] : im.nvis[0]) < 0) continue;
            ok = wait(&sh.q_empty[w], ~q_par >> w & 1);
            if (!ok) break;
            q_par ^= 1u << w;
            q_any |= 1u << w;
            const uint32_t qb = smem_u32(&sh.q_full[w]);
            if (lane == 0) mbar_arrive_expect_tx(qb, kPaTileBytes);
            __syncwarp();
            if (lane < 2)
              pa_tma(smem_u32(sh.q[w]) + lane * (kPaRows * 128), &maps.q, qb, lane * 64, im.h * G, im.tok + w * TT);
          }
        }
      }
      if (!ok) break;
    }
    // every copy has landed before the CTA may end (at once unless a wait gave up)
    for (uint32_t i = n > kPaRing ? n - kPaRing : 0; i < n; ++i)
      mbar_wait(smem_u32(&sh.kv_full[i % kPaRing]), (i / kPaRing) & 1, L.error);
    for (int w = 0; w < 2; ++w)
      if (q_any >> w & 1) mbar_wait(smem_u32(&sh.q_full[w]), ~q_par >> w & 1, L.error);
  } else if (warp == 8) {
    // ---------------------------------------------------------------- tensor cores
    uint32_t n = 0;  // ring tiles passed
    const bool unbounded = pa_uniform(*reinterpret_cast<volatile unsigned int*>(L.unbounded)) != 0;
    // bit w, for query tile w: the parity of the next S / P V / item, and whether
    // there has been one
    uint32_t s_par = 0, v_par = 0, q_par = 0, s_any = 0, v_any = 0;
    bool ok = true;
    // descriptors of K and V tiles but for the address (16-byte units, low bits)
    const uint64_t k_desc = pa_desc(0, 16, 1024), v_desc = pa_desc(0, kPaRows * 128, 1024);
    const uint32_t kv0 = smem_u32(sh.kv[0]) >> 4, q0 = smem_u32(sh.q[0]) >> 4;
    // O of query tile w += P V (ring tile rv); `last`: nobody else needs V
    auto value = [&](int w, int rv, bool add, bool last) -> bool {
      const uint32_t tS = tmem + w * 128, tO = tmem + 256 + w * 128;
      const uint64_t vd = v_desc + (kv0 + rv * (kPaTileBytes / 16));
#pragma unroll 1
      for (int hf = 0; hf < 2; ++hf) {
        if (!wait(&sh.p_full[w][hf], v_par >> w & 1)) return false;
        if (pa_elect()) {
          tc_fence_after();
#pragma unroll
          for (int kk = 0; kk < kPaSlots / 32; ++kk)
            pa_mma_ts(tO, tS + (hf * 4 + kk) * 8, vd + (hf * 4 + kk) * (2048 / 16), pa_idesc(true), add || hf || kk > 0);
          if (hf) {
            pa_commit(smem_u32(&sh.o_full[w]));
            if (last) pa_commit(smem_u32(&sh.kv_empty[rv]));
          }
        }
        __syncwarp();
      }
      v_par ^= 1u << w;
      v_any |= 1u << w;
      return true;
    };
    // S of query tile w = Q K^T (ring tile rk). S overwrites P of the K/V tile
    // before: its P V has to be over
    auto score = [&](int w, int rk, bool last, bool raw) -> bool {
      const uint32_t tS = tmem + w * 128;
      const uint64_t qd = k_desc + (q0 + w * (kPaTileBytes / 16)), kd = k_desc + (kv0 + rk * (kPaTileBytes / 16));
      if ((v_any >> w & 1) && !wait(&sh.o_full[w], ~v_par >> w & 1)) return false;
      if (pa_elect()) {
        tc_fence_after();
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk) {
          const uint32_t off = ((kk >> 2) * (kPaRows * 128) + (kk & 3) * 32) / 16;
          pa_mma(tS, qd + off, kd + off, pa_idesc(false), kk > 0);
        }
        pa_commit(smem_u32(&sh.s_full[w]));
        if (last) pa_commit(smem_u32(&sh.kv_empty[rk]));
        if (raw) pa_commit(smem_u32(&sh.q_empty[w]));
      }
      __syncwarp();
      s_par ^= 1u << w;
      s_any |= 1u << w;
      return true;
    };
    // rows [r0, r1) of a V tile set to zero: their weights are zero, but what
    // the page or the prompt holds there need not be a number
    auto zero_rows = [&](int rs, int r0, int r1) {
#pragma unroll 1
      for (int x = lane; x < (r1 - r0) * 16; x += 32) {
        const int r = r0 + (x >> 4), j = x & 15;
        *reinterpret_cast<uint4*>(sh.kv[rs] + (j >> 3) * (kPaRows * 128) + r * 128 + (j & 7) * 16) =
            make_uint4(0, 0, 0, 0);
      }
      fence_async_smem();
      __syncwarp();
    };
    for (int it = 0; ok; ++it) {
      const int sl = it % kPaItems;
      if (!wait(&sh.item_full[sl], (it / kPaItems) & 1)) break;
      PaItem im;
      im.t0 = pa_uniform(sh.item[sl].t0);
      im.t1 = pa_uniform(sh.item[sl].t1);
      im.tok = pa_uniform(sh.item[sl].tok);
      im.nvis[0] = pa_uniform(sh.item[sl].nvis[0]);
      im.nvis[1] = pa_uniform(sh.item[sl].nvis[1]);
      arrive_warp(&sh.item_empty[sl]);
      if (im.t0 > im.t1) break;
      if (max(im.nvis[0], im.nvis[1]) < 0) continue;
      const int nvis = max(im.nvis[0], im.nvis[1]);
      const int nslot = slot_tiles(nvis), nraw = raw_tiles(im);
      int due = 0;       // query tiles whose P V of the K/V tile before is due
      uint32_t acc = 0;  // query tiles whose O holds a value
      uint32_t np = n;   // the ring index of the step before
      // (the first P V of an item does not add)
      const int nboth = min(slot_tiles(im.nvis[0]), slot_tiles(im.nvis[1]));
      // step i: P V of the K/V tile before, then S of slot tile i (i = nslot: of
      // the raw tile), query tile by query tile
#pragma unroll 1
      for (int i = 0; i <= nslot + 1 && ok; ++i) {
        // the slot tiles that both query tiles see, but for the first: nothing to
        // decide or prepare, so little stands between the tensor core's pieces of work
        for (; ok && i > 0 && i < nboth; ++i) {
          const int rk = n % kPaRing, rv = (n - 1) % kPaRing;
          ok = wait(&sh.kv_full[rv], ((n - 1) / kPaRing) & 1) && value(0, rv, i > 1, false) &&
               wait(&sh.kv_full[rk], (n / kPaRing) & 1) && score(0, rk, false, false) &&
               value(1, rv, i > 1, true) && score(1, rk, true, false);
          np = n;
          n += 2;
          acc = 3;
        }
        if (!ok) break;
        int mask = 0;
        if (i <= nslot)
          mask = (im.nvis[0] >= 0 && (i == nslot || i < slot_tiles(im.nvis[0])) ? 1 : 0) |
                 (im.nvis[1] >= 0 && (i == nslot || i < slot_tiles(im.nvis[1])) ? 2 : 0);
#pragma unroll 1
        for (int w = 0; w < 2; ++w) {
          if (ok && (due >> w & 1)) {
            const bool raw = i - 1 == nslot, own = raw && nraw == 2;
            const uint32_t vt = np + (raw ? nraw : 1) + (own ? w : 0);
            const int rv = vt % kPaRing;
            if (!(ok = wait(&sh.kv_full[rv], (vt / kPaRing) & 1))) break;
            // V rows beyond what the tile's rows see hold other slots or tokens, or
            // nothing yet, which need not be numbers: the first to use them clears them
            if (own || !(due & (w ? 1 : 0))) {
              const int rows = raw ? raw_end(im, own ? w : 0) - raw_first(im, own ? w : 0) : nvis - (i - 1) * kPaSlots;
              const int unit = raw ? RAW : kPage;
              if (rows < kPaSlots && rows % unit) zero_rows(rv, rows, (rows + unit - 1) / unit * unit);
            }
            const int sees = raw ? im.tok + TT - raw_first(im, 0) : im.nvis[0] - (i - 1) * kPaSlots;
            if (unbounded && w == 0 && due == 3 && !own && sees < kPaSlots) {
              if (!(ok = wait(&sh.p_full[0][0], v_par & 1) && wait(&sh.p_full[0][1], v_par & 1))) break;
              pa_value_clipped(sh, tmem, rv, sees, acc & 1, false);
              v_par ^= 1u;
              v_any |= 1u;
            } else if (!(ok = value(w, rv, acc >> w & 1, own || !(due >> (w + 1))))) {
              break;
            }
            acc |= 1u << w;
          }
          if (ok && (mask >> w & 1)) {
            const bool raw = i == nslot, own = raw && nraw == 2;
            const uint32_t kt = n + (own ? w : 0);
            const int rk = kt % kPaRing;
            if (!(acc >> w & 1)) {  // its first of the item
              if (!(ok = wait(&sh.q_full[w], q_par >> w & 1))) break;
              q_par ^= 1u << w;
              // q[0] is the importance gate, not a feature
              for (int r = lane; r < kPaRows; r += 32)
                *reinterpret_cast<__nv_bfloat16*>(sh.q[w] + pa_swz(r, 0)) = __float2bfloat16_rn(0.f);
              fence_async_smem();
              __syncwarp();
            }
            if (!(ok = wait(&sh.kv_full[rk], (kt / kPaRing) & 1))) break;
            if (!(ok = score(w, rk, own || !(mask >> (w + 1)), raw))) break;
          }
        }
        due = mask;
        np = n;
        if (i <= nslot) n += i < nslot ? 2 : 2 * nraw;
      }
    }
    // every MMA is over before the CTA may end
    for (int w = 0; w < 2; ++w) {
      if (s_any >> w & 1) mbar_wait(smem_u32(&sh.s_full[w]), ~s_par >> w & 1, L.error);
      if (v_any >> w & 1) mbar_wait(smem_u32(&sh.o_full[w]), ~v_par >> w & 1, L.error);
    }
  }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 208;");
    // ---------------------------------------------------------------- softmax
    const int w = warp >> 2;              // query tile
    const int r = tid & (kPaRows - 1);    // row of the tile
    const int wq = warp & 3;
    const uint32_t lane_base = (uint32_t)(wq * 32) << 16;  // this warp's TMEM lanes
    const uint32_t tS = tmem + w * 128 + lane_base, tO = tmem + 256 + w * 128 + lane_base;
    const float qscale = 1.4426950408889634f / sqrtf((float)D);  // log2(e) / sqrt(d_h)
    uint32_t steps = 0, nq = 0;
    bool ok = true;
    for (int it = 0; ok; ++it) {
      const int sl = it % kPaItems;
      if (!wait(&sh.item_full[sl], (it / kPaItems) & 1)) break;
      const PaItem im = sh.item[sl];
      if (im.t0 > im.t1) break;
      if (!wait(&sh.meta_full[sl], (it / kPaItems) & 1)) break;
      if (im.nvis[w] < 0) {
        arrive_warp(&sh.item_empty[sl]);
        continue;
      }
      const PaMeta& M = sh.meta[sl][G == 1 ? w : 0];
      const int h = im.h, tok0 = im.tok + w * TT;
      const int tokN = min(tok0 + TT, im.t1);
      const int a0 = im.t0 + (tok0 - im.t0) / kPrefillChunk * kPrefillChunk;  // the chunk holding the tile
      // ---- the row: token tok0 + r / G, query head h G + r % G
      const int tau_r = tok0 + r / G;
      const bool row_ok = tau_r < tokN;
      const int ti = (row_ok ? r / G : 0) + (tok0 - a0);     // the row's token in the chunk
      const int nvis = row_ok ? min(im.base[w] + M.opened[ti] - 1, im.len_final) : 0;  // closed slots this row sees
      const int sg = row_ok ? M.seg[ti] : 0;  // its segment's first token in the chunk, or -1
      const float rz = M.rz[ti];
      const int ntile = slot_tiles(im.nvis[w]);

      float m = -INFINITY, l = 0.f;
      // The running maximum m moves only when a tile's row maximum mt exceeds it
      // by more than 8 (P then stays below 2^8); O and l are rescaled on a move
      // (rows that saw nothing yet hold zeros).
      auto new_max = [&](float mt) {
        const bool grow = mt > m + 8.f, resc = grow && m != -INFINITY;
        const float corr = resc ? pa_ex2(m - mt) : 1.f;
        if (grow) m = mt;
        l *= corr;
        if (__any_sync(0xffffffffu, resc)) pa_rescale(tO, corr);
      };
      for (int jt = 0; jt < ntile; ++jt, ++steps) {
        const int vis = min(max(nvis - jt * kPaSlots, 0), kPaSlots);  // visible columns of the row
        const bool full = __all_sync(0xffffffffu, vis == kPaSlots);   // no mask in this warp
        if (!(ok = wait(&sh.s_full[w], steps & 1))) break;
        tc_fence_after();
        // ---- online softmax, in the log2 domain (qscale > 0)
        float s[kPaSlots];
#pragma unroll
        for (int c0 = 0; c0 < kPaSlots; c0 += 32) pa_ld32(tS + c0, s + c0);
        pa_wait_ld();
        if (!full) {
          // (only the columns that some row of the warp does not see)
          const int seen = __reduce_min_sync(0xffffffffu, vis);
#pragma unroll
          for (int c0 = 0; c0 < kPaSlots; c0 += 32) {
            if (c0 + 32 <= seen) continue;
            const int left = min(max(vis - c0, 0), 32);
            const uint32_t hide = left == 32 ? 0u : 0xffffffffu << left;
#pragma unroll
            for (int i = 0; i < 32; ++i) s[c0 + i] = (hide >> i & 1u) ? -INFINITY : s[c0 + i];
          }
        }
        float mx[4] = {s[0], s[1], s[2], s[3]};
#pragma unroll
        for (int i = 4; i < kPaSlots; i += 8) {
#pragma unroll
          for (int e = 0; e < 4; ++e)
            mx[e] = i + e + 4 < kPaSlots ? fmaxf(fmaxf(mx[e], s[i + e]), s[i + e + 4]) : fmaxf(mx[e], s[i + e]);
        }
        new_max(fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * qscale);
        const float nm = m == -INFINITY ? 0.f : -m;  // nothing seen: every s is -inf
        const float2 scale2 = make_float2(qscale, qscale), shift2 = make_float2(nm, nm);
        float2 sum[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
        for (int c0 = 0; c0 < kPaSlots; c0 += 64) {
          uint32_t pk[32];
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            const float2 x = fma2(make_float2(s[c0 + 2 * i], s[c0 + 2 * i + 1]), scale2, shift2);
            const float2 p = make_float2(pa_ex2(x.x), pa_ex2(x.y));
            sum[i & 1] = add2(sum[i & 1], p);
            pk[i] = Chunk<__nv_bfloat16>::pack2(p.x, p.y);
          }
          // P over the row's own S columns: slots c0 + 2 i, + 1 in column c0 / 2 + i
          pa_st32(tS + c0 / 2, pk);
          if (c0 == 0) {
            pa_wait_st();
            tc_fence_before();
            arrive_warp(&sh.p_full[w][0]);
          }
        }
        l += (sum[0].x + sum[0].y) + (sum[1].x + sum[1].y);
        pa_wait_st();
        tc_fence_before();
        arrive_warp(&sh.p_full[w][1]);
      }
      if (!ok) break;

      // ---- the diagonal state as one more tile. When token i of the chunk
      // attends, its own slot holds k~ = (c_k [no opening in the chunk up to i] +
      // sum over j = lo..i of omega_j k_j) / z_i, lo being its segment's first
      // token in the chunk (c_k: the carried sums), and v~ alike. Its score
      // q . k~ and its share of O come from the chunk's raw rows: S_d = Q Kraw^T
      // summed with the weights omega_j / z_i, then O += P_d Vraw with
      // P_d[j] = exp2(score - m) omega_j / z_i over the segment's columns.
      // q . c_k, when the segment runs in from before the chunk
      float cdot = 0.f;
      if (__any_sync(0xffffffffu, sg < 0)) {
        if (!(ok = wait(&sh.q_full[w], nq & 1))) break;
        if (sg < 0) {
#pragma unroll 1
          for (int j = 0; j < 16; ++j) {
            float qf[8];
            Chunk<__nv_bfloat16>::unpack(*reinterpret_cast<const uint4*>(sh.q[w] + pa_swz(r, j)), qf);
            if (j == 0) qf[0] = 0.f;  // q[0] is the gate
            const float4 c0 = *reinterpret_cast<const float4*>(M.carry + j * 8);
            const float4 c1 = *reinterpret_cast<const float4*>(M.carry + j * 8 + 4);
            cdot = fmaf(qf[0], c0.x, cdot);
            cdot = fmaf(qf[1], c0.y, cdot);
            cdot = fmaf(qf[2], c0.z, cdot);
            cdot = fmaf(qf[3], c0.w, cdot);
            cdot = fmaf(qf[4], c1.x, cdot);
            cdot = fmaf(qf[5], c1.y, cdot);
            cdot = fmaf(qf[6], c1.z, cdot);
            cdot = fmaf(qf[7], c1.w, cdot);
          }
        }
      }
      ++nq;
      arrive_warp(&sh.q_empty[w]);

      const int lo = max(sg, 0);
      // columns c0 .. c0 + 31 within the row's segment [lo, ti], as bits
      auto seg_bits = [&](int c0) -> uint32_t {
        const int b = max(lo - c0, 0), e = min(ti + 1 - c0, 32);
        if (b >= e) return 0u;
        return (0xffffffffu >> (32 - (e - b))) << b;
      };
      const int w_lo = __reduce_min_sync(0xffffffffu, lo), w_hi = __reduce_max_sync(0xffffffffu, ti);
      if (!(ok = wait(&sh.s_full[w], steps & 1))) break;
      tc_fence_after();
      float wsum = cdot;
      // the columns where a row of the warp has its segment, 32 at a time
#pragma unroll 1
      for (int c0 = w_lo & ~31; c0 <= w_hi; c0 += 32) {
        float f[32];
        pa_ld32(tS + c0, f);
        const uint32_t in = seg_bits(c0);
        pa_wait_ld();
#pragma unroll
        for (int i = 0; i < 32; i += 4) {
          const float4 om = *reinterpret_cast<const float4*>(M.om + c0 + i);
          wsum = fmaf(in & (1u << i) ? om.x : 0.f, in & (1u << i) ? f[i] : 0.f, wsum);
          wsum = fmaf(in & (2u << i) ? om.y : 0.f, in & (2u << i) ? f[i + 1] : 0.f, wsum);
          wsum = fmaf(in & (4u << i) ? om.z : 0.f, in & (4u << i) ? f[i + 2] : 0.f, wsum);
          wsum = fmaf(in & (8u << i) ? om.w : 0.f, in & (8u << i) ? f[i + 3] : 0.f, wsum);
        }
      }
      const float dsc = wsum * rz * qscale;  // the diagonal score (log2 units)
      new_max(dsc);
      const float pd = pa_ex2(dsc - m);  // the diagonal's weight, below 2^8
      const float pw = pd * rz;
#pragma unroll 1
      for (int c0 = 0; c0 < kPaSlots; c0 += 32) {
        uint32_t pk[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) pk[i] = 0u;
        if (!(c0 > w_hi || c0 + 32 <= w_lo)) {
          const uint32_t in = seg_bits(c0);
#pragma unroll
          for (int i = 0; i < 16; i += 2) {
            const float4 om = *reinterpret_cast<const float4*>(M.om + c0 + 2 * i);
            pk[i] = Chunk<__nv_bfloat16>::pack2(in & (1u << (2 * i)) ? pw * om.x : 0.f,
                                                in & (2u << (2 * i)) ? pw * om.y : 0.f);
            pk[i + 1] = Chunk<__nv_bfloat16>::pack2(in & (4u << (2 * i)) ? pw * om.z : 0.f,
                                                    in & (8u << (2 * i)) ? pw * om.w : 0.f);
          }
        }
        pa_st16(tS + c0 / 2, pk);
      }
      pa_wait_st();
      tc_fence_before();
      arrive_warp(&sh.p_full[w][0]);
      arrive_warp(&sh.p_full[w][1]);

      // ---- epilogue: the row of O, with the carried value sums' share, over the row sum
      const float inv = 1.f / (l + pd);
      if (!(ok = wait(&sh.o_full[w], steps & 1))) break;
      ++steps;
      tc_fence_after();
      const bool carried = __any_sync(0xffffffffu, sg < 0);
      const float cw = sg < 0 ? pw : 0.f;  // weight of the carried value sums
      const float2 cw2 = make_float2(cw, cw), inv2 = make_float2(inv, inv);
      unsigned char* st = sh.stage[warp];
      // four lanes write 64 bytes of a row, eight rows at a time
      const int row0 = wq * 32 + (lane >> 2);
      char* op = a.out + ((size_t)(tok0 + row0 / G) * L.Hq + (size_t)h * G + row0 % G) * ROW + (lane & 3) * 16;
      const size_t step = (size_t)(8 / G) * L.Hq * ROW;  // eight rows on (G divides 8)
#pragma unroll 1
      for (int c0 = 0; c0 < D; c0 += 32) {
        float o[32];
        pa_ld32(tO + c0, o);
        pa_wait_ld();
        if (carried) {
#pragma unroll
          for (int i = 0; i < 32; i += 4) {
            const float4 cv = *reinterpret_cast<const float4*>(M.carry + D + c0 + i);
            if (sg < 0) {  // otherwise nothing was carried, and the buffer need not hold numbers
              const float2 x = fma2(cw2, make_float2(cv.x, cv.y), make_float2(o[i], o[i + 1]));
              const float2 y = fma2(cw2, make_float2(cv.z, cv.w), make_float2(o[i + 2], o[i + 3]));
              o[i] = x.x; o[i + 1] = x.y; o[i + 2] = y.x; o[i + 3] = y.y;
            }
          }
        }
#pragma unroll
        for (int i = 0; i < 32; i += 2) {
          const float2 x = mul2(make_float2(o[i], o[i + 1]), inv2);
          o[i] = x.x; o[i + 1] = x.y;
        }
        __syncwarp();  // the stage has been read
#pragma unroll
        for (int q4 = 0; q4 < 4; ++q4)
          *reinterpret_cast<uint4*>(st + lane * kPaStageRow + q4 * 16) = Chunk<__nv_bfloat16>::pack(o + q4 * 8);
        __syncwarp();
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const uint4 v = *reinterpret_cast<const uint4*>(st + (k * 8 + (lane >> 2)) * kPaStageRow + (lane & 3) * 16);
          if (tok0 + (row0 + 8 * k) / G < tokN) *reinterpret_cast<uint4*>(op + k * step + c0 * 2) = v;
        }
      }
      tc_fence_before();  // this item's TMEM loads are done before the next item's P is announced
      arrive_warp(&sh.item_empty[sl]);
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 8) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
  }
  if (tid == 0) {  // the last CTA out resets the work counter for the next call
    __threadfence();
    if (atomicAdd(&ctr[1], 1) == (int)gridDim.x - 1) {
      ctr[0] = 0;
      ctr[1] = 0;
      __threadfence();
    }
  }
}

// A 3-D bf16 tensor map: rows of 128 columns (box 64, 128-byte swizzle), `ny`
// rows of stride `sy` bytes (box by), `nz` planes of stride `sz` bytes (box bz).
static cudaError_t pa_map(CUtensorMap* map, const void* base, uint64_t ny, uint64_t sy, uint32_t by, uint64_t nz,
                          uint64_t sz, uint32_t bz) {
  using Encode = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                              const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  static const Encode encode = [] {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult found;
    const cudaError_t e =
        cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &found);
    return e == cudaSuccess && found == cudaDriverEntryPointSuccess ? reinterpret_cast<Encode>(fn) : nullptr;
  }();
  if (!encode) return cudaErrorNotSupported;
  const cuuint64_t dims[3] = {(cuuint64_t)kPaD, ny, nz};
  const cuuint64_t strides[2] = {sy, sz};
  const cuuint32_t box[3] = {64, by, bz}, unit[3] = {1, 1, 1};
  const CUresult r = encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box,
                            unit, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

template <int G>
static cudaError_t launch_pa(PrefillAttnArgs a, const void* k, const void* v, cudaStream_t stream) {
  const Layout& L = a.lay;
  constexpr uint64_t ROW = kPaD * 2;
  cudaError_t e = cudaFuncSetAttribute(dmc_prefill_attn_kernel<G>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       kPaSmem);
  int dev = 0, sms = 0;
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  PaMaps maps;
  constexpr uint32_t raw = kPaRawRows<G>;
  if (e == cudaSuccess) e = pa_map(&maps.q, a.q, L.Hq, ROW, G, a.total_tokens, L.Hq * ROW, kPaRows / G);
  if (e == cudaSuccess) e = pa_map(&maps.k, k, L.Hkv, ROW, 1, a.total_tokens, L.Hkv * ROW, raw);
  if (e == cudaSuccess) e = pa_map(&maps.v, v, L.Hkv, ROW, 1, a.total_tokens, L.Hkv * ROW, raw);
  if (e == cudaSuccess)
    e = pa_map(&maps.pages, L.pages, kPage, ROW, kPage, 2 * (uint64_t)L.num_pages, kPage * ROW, 1);
  if (e != cudaSuccess) return e;
  constexpr int TT2 = 2 * kPaRows / G;
  const long long tiles = (a.max_seqlen + TT2 - 1) / TT2;
  const int num_seqs = a.num_seqs, first_seq = a.first_seq;
  const int* cu = a.cu;
  // at most kPaMaxSeqs sequences per launch (the work-item table)
  for (int s0 = 0; s0 < num_seqs; s0 += kPaMaxSeqs) {
    a.seq_base = s0;
    a.num_seqs = min(kPaMaxSeqs, num_seqs - s0);
    a.first_seq = first_seq + s0;
    a.cu = cu + s0;
    const long long items = tiles * L.Hkv * a.num_seqs;  // an upper bound
    if (items == 0) continue;
    const int grid = (int)(items < sms ? items : sms);  // one CTA per SM: its shared memory and TMEM
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kPaThreads);
    cfg.dynamicSmemBytes = kPaSmem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, dmc_prefill_attn_kernel<G>, a, maps);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t prefill_attn_launch(const Layout& L, int layer, int first_seq, int num_seqs,
                                const void* q, const void* k, const void* v, const int* cu,
                                int total_tokens, int max_seqlen, const float* carry, const float* weights,
                                void* out, cudaStream_t stream) {
  PrefillAttnArgs a;
  a.lay = L;
  a.layer = layer;
  a.first_seq = first_seq;
  a.num_seqs = num_seqs;
  a.q = static_cast<const char*>(q);
  a.cu = cu;
  a.total_tokens = total_tokens;
  a.max_seqlen = max_seqlen;
  a.carry = carry;
  a.weights = weights;
  a.out = static_cast<char*>(out);
  switch (L.G) {
    case 1: return launch_pa<1>(a, k, v, stream);
    case 2: return launch_pa<2>(a, k, v, stream);
    case 4: return launch_pa<4>(a, k, v, stream);
    case 8: return launch_pa<8>(a, k, v, stream);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace dmc

// A layer call of 9 to 32 tokens in a dependent chain (x is what the call before left) as one kernel on
// clusters of four CTAs: router (Eq. 3), or scores and maybe the union list given, Union(x) (Sec. 3.3), up and
// down projection (Eq. 1, Eq. 2). Which calls come here: cluster_plan, below. The steps and the two exchanges
// over the whole device are those of
// expert_chain.cu (which see); this file is about what 32 tokens cost there: every CTA took in all
// of x and of h, 128 + 344 KB, next to 290 KB of weights, and 16 warps fed mma.sync from registers,
// so that a layer was bound by issue slots (22.6 K of its 46 K cycles per scheduler), by L2 -> SM
// bytes and by the latencies between them: 24.4 us at d = 2048, E = 128, d_e = 128, 32 tokens with a
// union of 43. Here 18.4 (45 MB of weights: 6.9 at the copy rate).
//
//   clusters of 4        the CTAs of a cluster work on the same rows of U (columns of D) and split K:
//                        each takes a quarter of x and of h, so the broadcast is a quarter. Partial
//                        sums go to the CTA that finishes a token by st.async through distributed
//                        shared memory (320 cycles, and the receiver's mbarrier counts the bytes).
//   tcgen05              the weights are the M operand (K-major, 128-byte swizzle, rows as they are in
//                        memory, 64 k at a time), the tokens N; one thread issues, sums stay in
//                        tensor memory. 64 rows x 16 k take 24 cycles, 128 rows 40, whatever N is.
//   logits               stay on mma.sync with sums of 32 products added in fp32 and the rest in 64
//                        bits (a chain inside the tensor core would lose bits).
//   copies of U          by cp.async: 70 to 80 GB/s per SM from L2 where tiles of 64 rows by TMA came to
//                        60 to 68, and 5.7 against 5.1 TB/s from DRAM (132 SMs). D comes by TMA all the
//                        same: one thread asks, so the warps that store h and partial sums do not queue
//                        behind ten thousand 16-byte copies (20.3 -> 19.5 us per layer).
//   shared memory        a ring of k blocks of U, x behind it; then the ring holds D, four k blocks to a
//                        slot, and x and the receive buffers behind it four slots of h (with two, h waited
//                        for the tensor core every 0.5 us: 19.5 -> 18.8).
//
// What is left, from time stamps (us after the layer before): 0.7 launch, 1.8 x, 3.8 logits published,
// 5.3 all in, 6.1 union, 8.1 first block of U, 10.3 last, 10.9 its products, 12.3 h written, 14.2 first h in,
// 17.3 products with D, 18.4 out. U takes what an SM takes in (172 KB, 2.4 us) and a latency of DRAM.
//
// The grid is as many clusters as fit the device at one CTA per SM (33 of B200's 148 / 4 = 37: SMs come
// in groups that four does not divide).
#include <cuda.h>

#include "exchange.cuh"

namespace {

constexpr int kCluster = 4;
constexpr int kDRows = 64;             // columns of out a cluster takes (rows of a D tile)
constexpr int kDBlock = kDRows * 128;  // a 64-wide k block of D
constexpr int kDSlot = 4 * kDBlock;    // D is copied four blocks at a time

// NTG: groups of 8 tokens, 4 (2: 9 .. 16 tokens)
template <int NTG>
struct Dims {
  static constexpr int T = 8 * NTG, NTH = 128 * NTG, W = 4 * NTG;
  static constexpr int TR = T / kCluster;       // tokens a CTA finishes
  static constexpr int QR = TR / 4;             // ... in groups of four
  static constexpr int RP = 192;                // rows of U a cluster takes at a time
  static constexpr int kSweep = NTH / 8;        // rows copied by one instruction of all threads
  static constexpr int kTmem = NTG == 4 ? 128 : 64;     // columns: three accumulators of T
  static constexpr int kHBlock = T * 128;       // a 64-wide k block of h
  static constexpr int kHSlot = 4 * kHBlock;    // h goes through the down projection four blocks at a time
  // receive buffers: partial sums of the logits, [source][token][16 experts] doubles, and of U x, [source][4
  // tokens][row][token]
  static constexpr int kLrecv = kCluster * TR * 16 * 8, kUrecv = kCluster * TR * RP * 4;
  static constexpr int kRecv = (kLrecv + kUrecv + kHSlot - 1) / kHSlot * kHSlot;
};

constexpr int kSlots = 8;              // of either ring, at most
constexpr int kLagBytes = 64 * 1024;   // of U on the way (20 KB: 698 us a pass of 36 layers, 48 KB 659, 80 KB 655)
constexpr int kBarBytes = 512;         // mbarriers: 10 + 6 kSlots; at the end the address of the tensor memory

struct ClusterLayout {
  int off_x, off_lrecv, off_urecv, off_bar, off_ctl, off_ids, off_tok, off_mask, off_score, off_hit, off_drecv, total;
};
// ring: k blocks of U, later the slots of D; x: [k block][token][64], with the receive buffers behind it
// later the slots of h
template <int NTG>
__host__ __device__ inline ClusterLayout cluster_layout(int d, int E, int ring) {
  using C = Dims<NTG>;
  ClusterLayout s;
  s.off_x = ring;
  s.off_lrecv = s.off_x + (((d >> 6) + kCluster - 1) / kCluster) * C::T * 128;
  s.off_urecv = s.off_lrecv + C::kLrecv;
  s.off_bar = s.off_lrecv + C::kRecv;
  s.off_ctl = s.off_bar + kBarBytes;
  s.off_ids = s.off_ctl + kCtlBytes;
  s.off_tok = s.off_ids + align128(E * 4);
  s.off_mask = s.off_tok + align128(E * 4);
  s.off_score = s.off_mask + (((E + 31) >> 5) + 1) * 128;
  s.off_hit = s.off_score + align128(C::TR * (E | 1) * 4);
  s.off_drecv = s.off_hit + 128;
  s.total = s.off_drecv + kCluster * C::TR * kDRows * 4 + 1024;   // (the base is aligned up)
  return s;
}

struct ClusterParams {
  const uint16_t* x;       // bf16 [L][d]
  const uint16_t* U;       // bf16 [E][d_e][d]
  const uint16_t* D;       // bf16 [E][d][d_e]
  const uint16_t* W_r;     // MODE 3: bf16 [E][d]
  const float* gain;       // f32 [E]
  const float* bias;       // f32 [E] or NULL
  float eps;
  const float* scores;     // MODE 0, 1: f32 [L][E]
  const int32_t* ids_in;   // MODE 1: the caller's union list
  const int32_t* n_in;
  unsigned long long* logits;   // kCopies times [L][E] words {logit, call number}
  size_t logit_copy;       // words from one copy to the next
  uint16_t* h;             // two buffers of h_slot elements, bf16 [q][d_e / 64][L][64]
  size_t h_slot;
  uint32_t* used;          // [2] 16-byte pieces of each buffer that its last call wrote
  unsigned long long* seq; // tickets, `sms` per call (the kernels that share the counter agree on that)
  int sms;
  float* out;
  uint16_t* x_next;
  int L, d, E, d_e, de_shift;
  int cols_q, cols_rem;    // pairs of columns of out per cluster
  uint32_t magic_g;        // ceil(2^32 / clusters)
  int ring;                // bytes
  int accumulate;
  int early;               // the weights are stable: read before the wait
  int reps;                // clusters that compute the logits of the same 16 experts
  int hold;                // test aid: wait for what never comes, 1 the logits, 2 h, 3 and 4 one CTA alone for
                           // the masks, for h
  int time_shift;          // ... of waits inside one: two to three times 2^time_shift ns from the call's start
  unsigned long long wait_ns;   // limit of a wait for other clusters
  uint32_t* status;
  RoutingOut pub;
};

// ---- PTX wrappers ----------------------------------------------------------------------------
__device__ __forceinline__ void mbar_init(uint32_t bar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint32_t bar, int bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, int parity) {
  uint32_t ok;
  asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
               "selp.b32 %0, 1, 0, p;\n}"
               : "=r"(ok)
               : "r"(bar), "r"(parity)
               : "memory");
  return ok != 0;
}
// (for what other CTAs' arrivals release)
__device__ __forceinline__ bool mbar_try_cluster(uint32_t bar, int parity) {
  uint32_t ok;
  asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
               "selp.b32 %0, 1, 0, p;\n}"
               : "=r"(ok)
               : "r"(bar), "r"(parity)
               : "memory");
  return ok != 0;
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, int rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(addr), "r"(rank));
  return a;
}
__device__ __forceinline__ void st_async_f64(uint32_t addr, double v, uint32_t bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(addr),
               "l"(__double_as_longlong(v)), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void st_async_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d,
                                            uint32_t bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(
                   addr),
               "r"(a), "r"(b), "r"(c), "r"(d), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// what this thread has written to shared memory is visible to the tensor core's reads after it
__device__ __forceinline__ void fence_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ bool elect_one() {
  uint32_t e;
  asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.b32 %0, 1, 0, p;\n}" : "=r"(e));
  return e != 0;
}
// The three below are called by whole warps and issued by one thread of them. (A branch around them would
// take the operands out of the uniform registers the instructions want them in.)
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("{\n.reg .pred q;\nelect.sync _|q, 0xffffffff;\n"
               "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}" ::"r"(bar)
               : "memory");
}
// Lower word of the descriptor of an operand in shared memory: rows of 64 bf16 (128 bytes, 16-byte
// pieces xor-ed with the row modulo 8), groups of 8 rows 1024 bytes apart, K-major.
__device__ __forceinline__ uint32_t tc_desc(uint32_t addr) { return ((addr & 0x3ffffu) >> 4) | (1u << 16); }
// bf16 x bf16 -> f32, M rows, N columns
__host__ __device__ constexpr uint32_t tc_idesc(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
// one 64-wide k block; first: the accumulator starts here
template <uint32_t IDESC>
__device__ __forceinline__ void tc_mma64(uint32_t acc, uint32_t a, uint32_t b, bool first) {
  constexpr uint32_t hi = 64u | (1u << 14) | (2u << 29);       // 1024 bytes, version, 128-byte swizzle
  asm volatile(
      "{\n.reg .pred p, q, t;\n.reg .b32 r;\n.reg .b64 a, b;\n"
      "elect.sync _|q, 0xffffffff;\nsetp.ne.b32 p, %5, 0;\nsetp.eq.b32 t, 0, 0;\n"
      "mov.b64 a, {%1, %4};\nmov.b64 b, {%2, %4};\n"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, p;\n"
      "add.s64 a, a, 2;\nadd.s64 b, b, 2;\n"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, t;\n"
      "add.s64 a, a, 2;\nadd.s64 b, b, 2;\n"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, t;\n"
      "add.s64 a, a, 2;\nadd.s64 b, b, 2;\n"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, t;\n}" ::"r"(acc),
      "r"(a), "r"(b), "n"(IDESC), "n"(hi), "r"(first ? 0 : 1)
      : "memory");
}
// 8 columns of this warp's 32 lanes
__device__ __forceinline__ void tc_ld8(uint32_t (&v)[8], uint32_t addr) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
               "tcgen05.wait::ld.sync.aligned;"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
               : "r"(addr)
               : "memory");
}
// at most n (0 .. 7) of this thread's newest commit groups are still in flight afterwards
__device__ __forceinline__ void cp_async_wait_newest(int n) {
  switch (n) {
    case 0: cp_async_wait_group<0>(); break;
    case 1: cp_async_wait_group<1>(); break;
    case 2: cp_async_wait_group<2>(); break;
    case 3: cp_async_wait_group<3>(); break;
    case 4: cp_async_wait_group<4>(); break;
    case 5: cp_async_wait_group<5>(); break;
    case 6: cp_async_wait_group<6>(); break;
    default: cp_async_wait_group<7>(); break;
  }
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void st_async_b32(uint32_t addr, uint32_t v, uint32_t bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(addr), "r"(v),
               "r"(bar)
               : "memory");
}
__device__ __forceinline__ void sts128(uint32_t a, const uint4& v) {
  asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
// global address = base + 16 * idx16 (idx16 < 2^32)
__device__ __forceinline__ const void* at16(const void* base, uint32_t idx16) {
  unsigned long long a;
  asm("mad.wide.u32 %0, %1, 16, %2;" : "=l"(a) : "r"(idx16), "l"(base));
  return reinterpret_cast<const void*>(a);
}

// The threads that copy, add and store are warps 0 .. W - 1; warp W only feeds the tensor core. (A fence
// between the proxies waits for the issuing thread's own copies in flight, 0.5 us a stage when the
// copying threads did it; warp W has none.)
// MODE: 0 scores given, 1 scores and the caller's union list given, 3 the router runs in the kernel.
template <int NTG, int MODE>
__global__ void __launch_bounds__(Dims<NTG>::NTH + 64, NTG == 4 ? 1 : 2)
    expert_cluster_kernel(const ClusterParams p, const __grid_constant__ CUtensorMap d_map) {
  using C = Dims<NTG>;
  constexpr int T = C::T, NTH = C::NTH, W = C::W, TR = C::TR, QR = C::QR, RP = C::RP;
  extern __shared__ unsigned char smem_raw[];
  const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(~0u, tid >> 5, 0);
  const int g = lane >> 2, tg = lane & 3;
  const int d = p.d, d_e = p.d_e, L = p.L, E = p.E, sh = p.de_shift;
  const int bx = blockIdx.x, G = gridDim.x, rank = bx % kCluster, cl = bx / kCluster, GC = G / kCluster;
  const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
  unsigned char* smem = smem_raw + (sbase - smem_u32(smem_raw));
  const ClusterLayout lay = cluster_layout<NTG>(d, E, p.ring);
  const int Es = E | 1, words = (E + 31) >> 5;
  int* ctl = reinterpret_cast<int*>(smem + lay.off_ctl);
  int* ids_sm = reinterpret_cast<int*>(smem + lay.off_ids);
  uint32_t* tok_sm = reinterpret_cast<uint32_t*>(smem + lay.off_tok);
  uint32_t* tm = reinterpret_cast<uint32_t*>(smem + lay.off_mask);     // token masks [word][32], then flags [32]
  float* a_sm = reinterpret_cast<float*>(smem + lay.off_score);        // scores of this CTA's tokens
  float* red = reinterpret_cast<float*>(smem);                           // (router: before U is asked for)
  const uint32_t xs = sbase + lay.off_x, ring = sbase;
  const uint32_t bar = sbase + lay.off_bar;
  const uint32_t bar_logit = bar, bar_mask = bar + 8, bar_up = bar + 16, bar_out = bar + 24;
  const uint32_t u_done = bar + 32;                                // all products with U
  const uint32_t full = bar + 40, freed = full + 8 * kSlots;       // slots of U: landed, read by the tensor core
  const uint32_t full_d = freed + 8 * kSlots, freed_d = full_d + 8 * kSlots;   // of D
  const uint32_t full_h = freed_d + 8 * kSlots, freed_h = full_h + 8 * kSlots;       // of h
  const uint32_t u_begun = freed_h + 8 * kSlots, bar_hit = u_begun + 8;

  const uint32_t acc_read = bar_hit + 8, recv_read = acc_read + 8;  // sums of a pass read, by this CTA, by the cluster
  const uint32_t bar_end = recv_read + 8;

  // How a call gives up. Waits for other clusters (logits, h) have a limit; one that runs out is told to the
  // CTA's mates, with the masks or with the last partial sums, and sets ctl[5]: this CTA writes no out. All go on
  // as if what was waited for had come, so the mates' waits (mbar_wait, for one another and inside a CTA) end.
  // Those have one limit for the call, well above the others, in case a mate makes no progress at all. A wait that
  // passes it sets ctl[4], and all later ones of the CTA are over at once: it sends no sums of U x any more, stores no
  // h and copies no D. However a call ends, all threads pass the same barriers of the CTA and of the cluster: their
  // number depends on nothing that was waited for.
  // (There are some thirty such waits, and code that every warp runs once is short of instruction fetch: with a start
  // time and the bookkeeping of a wait that ran out in each of them 32 tokens took 690 us a pass of 36 layers, so 668.)
  auto broken = [&]() { return *reinterpret_cast<const volatile int*>(ctl + 4) != 0; };
  auto coarse_time = [&]() { return (uint32_t)(clock_ns() >> p.time_shift); };
  uint32_t deadline = coarse_time() + 3;
  auto wait_for = [&](auto&& done) {
    while (!done()) {
      if ((int)(coarse_time() - deadline) >= 0) {
        ctl[4] = 1;
        break;
      }
    }
    __syncwarp();
  };
  auto mbar_wait = [&](uint32_t b, int parity) { wait_for([&]() { return mbar_try(b, parity); }); };
  auto copy_sync = [&]() { asm volatile("bar.sync 1, %0;" ::"n"(NTH) : "memory"); };   // the copying warps

  // Everything that is asked for from memory first (ticket, router weights, then x) is on its way at once.
  unsigned long long ticket = 0;
  // (a call draws p.sms tickets whatever its grid)
  if (tid == 0) {
    const int more = p.sms - G;
    ticket = atomicAdd(p.seq, (unsigned long long)(1 + more / G + (bx < more % G ? 1 : 0)));
  }
  if (!p.early) pdl_wait();
  // this CTA's quarter of K = d: 64-wide blocks kb0 .. kb0 + nkb
  const int nbk = d >> 6, kb0 = (nbk * rank) >> 2, nkb = ((nbk * (rank + 1)) >> 2) - kb0;
  // W_r: the cluster has the 16 experts from 16 grp on (p.reps clusters have the same ones). A warp
  // takes the half blocks v = warp UN + i of the quarter: of block v / 2 lane tg has, in both
  // operands, the 16-byte piece 2 tg + v % 2.
  constexpr int UN = 16 / W, kHitWords = TR / 2;
  const int ngroups = (E + 15) >> 4;
  const int rep = cl / ngroups;
  const bool routes = MODE == 3 && rep < p.reps;
  uint4 wf[UN][2];
  float bias = 0.0f;
  auto load_wr = [&](int grp) {
    const int e0 = 16 * grp, rrows = min(16, E - e0);
#pragma unroll
    for (int i = 0; i < UN; ++i) {
      const int v = warp * UN + i;
      wf[i][0] = wf[i][1] = make_uint4(0, 0, 0, 0);
      const uint16_t* w = p.W_r + (size_t)(e0 + g) * d + (kb0 + (v >> 1)) * 64 + (2 * tg + (v & 1)) * 8;
      if ((v >> 1) < nkb && g < rrows) wf[i][0] = __ldg(reinterpret_cast<const uint4*>(w));
      if ((v >> 1) < nkb && g + 8 < rrows) wf[i][1] = __ldg(reinterpret_cast<const uint4*>(w + 8 * (size_t)d));
    }
    bias = p.bias && (tid & 15) < rrows ? __ldg(p.bias + e0 + (tid & 15)) : 0.0f;
  };
  if (MODE == 3 && routes && warp < W) load_wr(cl - rep * ngroups);
  float gains[4];                  // of experts lane, lane + 32, ...
#pragma unroll
  for (int u = 0; u < 4; ++u) gains[u] = MODE == 3 && warp < TR && 32 * u + lane < E ? __ldg(p.gain + 32 * u + lane) : 0.0f;
  if (tid < 6) ctl[tid] = 0;       // ([6], [7]: by thread 0 below, with no barrier in between)
  if (tid == 32) {
    for (int i = 0; i < 5; ++i) mbar_init(bar + 8 * i, 1);
    mbar_init(u_begun, 1);
    mbar_init(bar_hit, 1);
    mbar_init(acc_read, W);
    mbar_init(recv_read, kCluster * W);
    mbar_init(bar_end, 1);
    for (int i = 0; i < kSlots; ++i) {
      mbar_init(full + 8 * i, W);
      mbar_init(freed + 8 * i, 1);
      mbar_init(full_d + 8 * i, 1);
      mbar_init(freed_d + 8 * i, 1);
    }
    for (int i = 0; i < kSlots; ++i) {
      mbar_init(full_h + 8 * i, W);
      mbar_init(freed_h + 8 * i, 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == W) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     sbase + (uint32_t)lay.off_bar + kBarBytes - 8),
                 "n"(C::kTmem)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }

  // x: this CTA's quarter of every token
  auto copy_x = [&]() {
    uint4 v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int k = tid + NTH * i, t = (k >> 3) & (T - 1), kb = k / (8 * T);
      if (t < L && kb < nkb) v[i] = ld_cg128(p.x + (size_t)t * d + (kb0 + kb) * 64 + (k & 7) * 8);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int k = tid + NTH * i, t = (k >> 3) & (T - 1), kb = k / (8 * T);
      if (t < L && kb < nkb) sts128(xs + kb * (T * 128) + t * 128 + (((k & 7) ^ (t & 7)) << 4), v[i]);
    }
  };
  if constexpr (MODE == 3) {
    pdl_wait();
    deadline = coarse_time() + 3;
    if (warp < W) copy_x();
  }
  if (tid == 0) {
    const unsigned long long n = ticket / (unsigned)p.sms;
    ctl[6] = (int)(n & 1);
    ctl[7] = (int)(uint32_t)(n + 1);
    pdl_trigger();
  }
  // this thread's output: token rank TR + tid / 64, column tid % 64 of the cluster's
  const int c0 = 2 * (cl * p.cols_q + min(cl, p.cols_rem));
  const int ncols = 2 * (p.cols_q + (cl < p.cols_rem ? 1 : 0));
  const int ot = rank * TR + (tid >> 6), om = tid & 63;
  const bool has_out = tid < NTH && ot < L && om < ncols;
  tc_before();
  __syncthreads();
  tc_after();
  // (the barriers are set up; relaxed: a release would wait for the router weights)
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  if (MODE == 3 && tid == 0) mbar_expect(bar_mask, T * (words + 1) * 4);
  __syncwarp();
  const uint32_t tmem = *reinterpret_cast<const uint32_t*>(smem + lay.off_bar + kBarBytes - 8);

  float resid = 0.0f;
  uint32_t clear_n = 0;            // pieces of the other h buffer to reset
  auto after_wait = [&]() {
    if (p.accumulate && has_out) resid = __ldcg(p.out + (size_t)ot * d + c0 + om);
    clear_n = __ldcg(p.used + (ctl[6] ^ 1));
  };
  auto clear_other = [&](uint32_t i, uint32_t n) {     // by n threads of a CTA, i: this one
    uint4* other = reinterpret_cast<uint4*>(p.h + (size_t)(ctl[6] ^ 1) * p.h_slot);
    for (i += bx * n; i < clear_n; i += G * n) other[i] = make_uint4(~0u, ~0u, ~0u, ~0u);
  };
  uint32_t odd_tokens = 0;         // tokens with a logit that is not finite
  bool lost = false;
  int nu;
  if constexpr (MODE == 3) {
    // ---- router: logits of the cluster's experts
    uint32_t phase_logit = 0;
    bool joined = false;             // whether the cluster's CTAs are known to have set up their barriers
    for (int grp = cl - rep * ngroups; routes && grp < ngroups; grp += GC) {
      const int e0 = 16 * grp, rrows = min(16, E - e0);
      if (phase_logit) {             // (more experts than 16 per cluster)
        if (warp < W) load_wr(grp);
        __syncwarp();
        cluster_arrive();            // the receive buffers of the group before have been read
        cluster_wait();
      }
      if (warp < W) {
        float f[NTG][4];
        zero_acc<NTG>(f);
#pragma unroll
        for (int i = 0; i < UN; ++i) {
          const int v = warp * UN + i;
          if ((v >> 1) < nkb) {
#pragma unroll
            for (int n = 0; n < NTG; ++n) {
              const uint4 xv = lds128(xs + (v >> 1) * (T * 128) + (8 * n + g) * 128 + (((2 * tg + (v & 1)) ^ g) << 4));
              float c[4] = {0.f, 0.f, 0.f, 0.f};
              mma_bf16(c, wf[i][0].x, wf[i][1].x, wf[i][0].y, wf[i][1].y, xv.x, xv.y);
              mma_bf16(c, wf[i][0].z, wf[i][1].z, wf[i][0].w, wf[i][1].w, xv.z, xv.w);
#pragma unroll
              for (int q = 0; q < 4; ++q) f[n][q] += c[q];
            }
          }
        }
        float* o = red + (warp * T + 2 * tg) * 20 + g;
#pragma unroll
        for (int n = 0; n < NTG; ++n, o += 8 * 20) {
          o[0] = f[n][0];
          o[20] = f[n][1];
          o[8] = f[n][2];
          o[28] = f[n][3];
        }
      }
      // (nothing is expected while what was expected before is still open)
      const bool expects = phase_logit == 0 || !broken();
      if (tid == 0 && expects) mbar_expect(bar_logit, T * 16 * 8);
      if (tid == NTH + 32 && expects) mbar_expect(bar_hit, kCluster * kHitWords * 4);
      __syncthreads();
      if (!joined) cluster_wait();
      joined = true;
      if (warp < W) {                // a CTA finishes the logits of its TR tokens
        const int t = tid >> 4, m = tid & 15, to = t / TR;
        // (four of the warps' sums of 32 products in 32 bits, the rest in 64)
        double sum = 0.0;
#pragma unroll
        for (int w = 0; w < W; w += 4) {
          const float* r = red + (w * T + t) * 20 + m;
          sum += (double)((r[0] + r[T * 20]) + (r[2 * T * 20] + r[3 * T * 20]));
        }
        st_async_f64(map_rank(sbase + lay.off_lrecv + (rank * TR * 16 + (tid & (TR * 16 - 1))) * 8, to), sum,
                     map_rank(bar_logit, to));
      }
      if (warp < kHitWords) {
        mbar_wait(bar_logit, phase_logit & 1);
        const int t = rank * TR + (tid >> 4), m = tid & 15;
        const bool whole = !broken();
        float v = 0.0f;
        if (t < L && m < rrows && whole) {
          // (in 64 bits: the bias cancels most of the sum of an expert that is just active)
          const double* in = reinterpret_cast<const double*>(smem + lay.off_lrecv) + tid;
          constexpr int s = TR * 16;
          v = (float)(((in[0] + in[s]) + (in[2 * s] + in[3 * s])) + (double)bias);
          const unsigned long long word = ((unsigned long long)(uint32_t)ctl[7] << 32) | __float_as_uint(v);
          unsigned long long* o = p.logits + (size_t)t * E + e0 + m;
          for (int k = rep; k < kCopies; k += p.reps)
            asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(o + k * p.logit_copy), "l"(word) : "memory");
        }
        // which of the experts some token activates, to the cluster
        const uint32_t up = __ballot_sync(0xffffffffu, v > 0.0f);
        if (lane < kCluster)
          st_async_b32(map_rank(sbase + lay.off_hit + (rank * kHitWords + warp) * 4, lane), (up | (up >> 16)) & 0xffffu,
                       map_rank(bar_hit, lane));
      }
      if (warp == W + 1) {
        // U of those experts is asked for in L2 here, where that is known first; the CTAs that have the same
        // experts share them out, a piece per thread
        mbar_wait(bar_hit, phase_logit & 1);
        uint32_t hit = 0;
#pragma unroll
        for (int k = 0; k < kCluster * kHitWords; ++k) hit |= reinterpret_cast<const uint32_t*>(smem + lay.off_hit)[k];
        if (lane < rrows && ((hit >> lane) & 1u)) {
          const uint32_t eb = (uint32_t)d * (uint32_t)d_e * 2u;      // bytes of U_e
          const uint32_t n = p.reps * kCluster, i = rep * kCluster + rank;
          const uint32_t share = ((eb + n - 1) / n + 127u) & ~127u, from = i * share;
          const char* src = reinterpret_cast<const char*>(p.U) + (size_t)(e0 + lane) * eb;
          if (from < eb)
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src + from), "r"(min(share, eb - from))
                         : "memory");
        }
      }
      ++phase_logit;
      __syncwarp();
    }
    if (!joined) cluster_wait();
    after_wait();                    // (not before: what the router waits for would come behind these)
    // ---- everybody's logits of this CTA's tokens, as they arrive, and Eq. 3 on them: a warp has a token
    if (warp < TR) {
      const int t = rank * TR + warp;
      const uint32_t tag = (uint32_t)ctl[7] + (p.hold == 1 ? 0x80000000u : 0u);
      const unsigned long long* words_in = p.logits + (cl & (kCopies - 1)) * p.logit_copy + (size_t)t * E;
      SpinBound bound;
      bool dead = false, finite = true;
      float ss = 0.0f;
      for (int w0 = 0; w0 < words && t < L && !dead; w0 += 4) {
        unsigned long long v[4];
        uint32_t pend = 0;
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (32 * (w0 + u) + lane < E) pend |= 1u << u;
        const uint32_t mine = pend;
        do {
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if ((pend >> u) & 1u) v[u] = ld_relaxed_u64(words_in + 32 * (w0 + u) + lane);
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (((pend >> u) & 1u) && (uint32_t)(v[u] >> 32) == tag) pend &= ~(1u << u);
          if (!__any_sync(0xffffffffu, pend != 0)) break;
          dead = __any_sync(0xffffffffu, bound.expired(p));
        } while (!dead);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if ((mine >> u) & 1u) {
            const float a = __uint_as_float((uint32_t)v[u]);
            finite &= ((uint32_t)v[u] & 0x7f800000u) != 0x7f800000u;
            const float r = a > 0.0f ? a : 0.0f;
            ss = fmaf(r, r, ss);
            a_sm[warp * Es + 32 * (w0 + u) + lane] = r;
          }
        }
      }
      finite = __all_sync(0xffffffffu, finite);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
      // (a negative eps marks the router without RMSNorm, Sec. 4.2.3; the gain is then all ones)
      const float r = p.eps < 0.0f ? 1.0f : 1.0f / sqrtf(ss / (float)E + p.eps);
      // the token's mask, to the four CTAs of the cluster
      const uint32_t to = map_rank(sbase + lay.off_mask + t * 4, lane & 3), to_bar = map_rank(bar_mask, lane & 3);
      for (int w = 0; w < words; ++w) {
        const int e = 32 * w + lane;
        float s = 0.0f;
        if (t < L && e < E) {
          const float gn = w == 0 ? gains[0] : w == 1 ? gains[1] : w == 2 ? gains[2] : w == 3 ? gains[3] : __ldg(p.gain + e);
          s = gn * a_sm[warp * Es + e] * r;
          a_sm[warp * Es + e] = s;
        }
        const uint32_t m = __ballot_sync(0xffffffffu, s != 0.0f);
        if (lane < kCluster) st_async_b32(to + w * 128, m, to_bar);
      }
      if (dead && lane == 0) atomicOr(p.status, BLOCKFFN_DEV_WAIT_EXPIRED);
      if (lane < kCluster) st_async_b32(to + words * 128, (finite ? 0u : 1u) | (dead ? 2u : 0u), to_bar);
      __syncwarp();
    } else if (warp < W) {           // the others put the other h buffer back meanwhile
      clear_other(tid - 32 * TR, NTH - 32 * TR);
    }
    mbar_wait(bar_mask, 0);
    if (p.hold == 3 && cl == 0 && rank == 1 && lane == 0) ctl[4] = 1;
    const uint32_t flag = lane < T ? tm[words * 32 + lane] : 0u;
    odd_tokens = __ballot_sync(0xffffffffu, flag & 1u);      // with a logit that is not finite
    // A wait for logits that ran out: the four CTAs, all of which have the flags, go through the rest with an
    // empty union.
    if (__any_sync(0xffffffffu, flag & 2u) && lane == 0) ctl[5] = 1;
    __syncthreads();
    lost = (ctl[4] | ctl[5]) != 0;                  // (the same for all threads)
    nu = union_of_masks(tm, L, words, ids_sm, ctl);
    if (lost) nu = 0;
  } else {
    nu = derive_union<MODE>(p.scores, RouterLogits{}, p.ids_in, p.n_in, L, E, ids_sm, ctl, tm);
    cluster_wait();
  }

  // ---- the cluster's rows of U: [r0, r0 + nrows) of the union's u * d_e, in fours, RP at a time ------
  const int R = nu * d_e;
  const int rq = (int)__umulhi((unsigned)R >> 2, p.magic_g), rrem = (R >> 2) - rq * GC;
  const int r0 = 4 * (cl * rq + min(cl, rrem)), nrows = 4 * (rq + (cl < rrem ? 1 : 0));
  // rows of a pass: evenly, the same in every cluster
  const int npass_max = (4 * (rq + 1) + RP - 1) / RP, rmax = 4 * ((rq + npass_max) / npass_max);
  const int slot_bytes = ((rmax + 7) & ~7) * 128;
  const int S = min(kSlots, p.ring / slot_bytes);
  const int npass = (nrows + rmax - 1) / rmax;
  const int pshift = sh - 6;
  // D: 64-wide blocks, this CTA's quarter b0 .. b0 + nb of the union's nu * d_e / 64, four at a time
  const int nblk = nu << pshift, b0 = (nblk * rank) >> 2, nb = ((nblk * (rank + 1)) >> 2) - b0;
  const int nsw = (nb + 3) >> 2, npairs = d_e >> 6;
  const int SD = min(kSlots, lay.off_x / kDSlot), SH = min(kSlots, (lay.off_bar - lay.off_x) / C::kHSlot);
  const uint32_t acc = tmem + 2 * T;
  // (what the two warps below wait for comes behind x: their limits must not run while the call before does)
  if (MODE != 3 && warp >= W) {
    pdl_wait();
    deadline = coarse_time() + 3;
  }

  if (warp == W) {
    // ======== the warp that feeds the tensor core ========
    int slot = 0, round = 0;
    for (int ps = 0; ps < npass; ++ps) {
      const int nr = min(rmax, nrows - ps * rmax);
      if (ps > 0) mbar_wait(acc_read, (ps - 1) & 1);
      for (int kb = 0; kb < nkb; ++kb) {
        mbar_wait(full + 8 * slot, round & 1);
        fence_async();
        tc_after();
        const uint32_t a = tc_desc(ring + slot * slot_bytes), b = tc_desc(xs + kb * (T * 128));
        if (nr <= 64) {
          tc_mma64<tc_idesc(64, T)>(tmem, a, b, kb == 0);
        } else {
          tc_mma64<tc_idesc(128, T)>(tmem, a, b, kb == 0);
          if (nr > 128) tc_mma64<tc_idesc(64, T)>(tmem + T, a + 1024, b, kb == 0);
        }
        tc_commit(freed + 8 * slot);
        if (ps == 0 && kb == min(4, nkb - 1) && lane == 0) mbar_arrive(u_begun);
        if (++slot == S) {
          slot = 0;
          ++round;
        }
      }
      if (ps + 1 == npass) tc_commit(u_done);
    }
    slot = round = 0;
    int hs = 0, hround = 0;
    for (int s = 0; s < nsw; ++s) {
      mbar_wait(full_d + 8 * slot, round & 1);
      mbar_wait(full_h + 8 * hs, hround & 1);
      fence_async();
      tc_after();
      const uint32_t a = tc_desc(sbase + slot * kDSlot);
      const uint32_t b = tc_desc(xs + hs * C::kHSlot);
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (4 * s + j < nb)
          tc_mma64<tc_idesc(64, T)>(acc, a + j * (kDBlock >> 4), b + j * (C::kHBlock >> 4), 4 * s + j == 0);
      tc_commit(freed_h + 8 * hs);
      if (++hs == SH) {
        hs = 0;
        ++hround;
      }
      tc_commit(freed_d + 8 * slot);
      if (++slot == SD) {
        slot = 0;
        ++round;
      }
    }
    if (__any_sync(0xffffffffu, broken())) {       // (nobody may have seen the newest products complete)
      tc_commit(bar_end);
      SpinBound limit;
      while (!mbar_try(bar_end, 0) && !limit.expired(p)) {
      }
    }
    __syncwarp();
    cluster_arrive();
  } else if (warp == W + 1) {
    // ======== the warp that copies D: first into L2, then where U and x were ========
    // (behind U, which is needed first)
    if (npass > 0) mbar_wait(u_begun, 0);
    const int qa = b0 >> pshift, qb = (b0 + nb + npairs - 1) >> pshift;
    for (int q = qa + lane; q < qb; q += 32)       // (an expert's columns are contiguous)
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p.D + ((size_t)ids_sm[q] * d + c0) * d_e),
                   "r"(ncols * d_e * 2)
                   : "memory");
    __syncwarp();
    // (a cluster without rows still copies D: the router's partial sums were there, and no fence for the
    // tensor core has come between them and these copies)
    if (npass > 0)
      mbar_wait(u_done, 0);
    else
      fence_async();
    int slot = 0, round = 0, s = 0;
    for (; s < nsw; ++s) {
      if (s >= SD) mbar_wait(freed_d + 8 * slot, (round - 1) & 1);
      if (__any_sync(0xffffffffu, broken())) break;
      if (elect_one()) {
        const int n = min(4, nb - 4 * s);
        mbar_expect(full_d + 8 * slot, n * kDBlock);
        for (int j = 0; j < n; ++j) {
          const int b = b0 + 4 * s + j;
          asm volatile("cp.async.bulk.tensor.2d.shared::cta.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
                       "[%4];" ::"r"(sbase + slot * kDSlot + j * kDBlock),
                       "l"(&d_map), "r"(64 * (b & (npairs - 1))), "r"(ids_sm[b >> pshift] * d + c0),
                       "r"(full_d + 8 * slot)
                       : "memory");
        }
      }
      __syncwarp();
      if (++slot == SD) {
        slot = 0;
        ++round;
      }
    }
    if (__any_sync(0xffffffffu, broken())) {       // (nobody may have seen the newest copies land)
      for (int k = max(0, s - SD); k < s; ++k) {
        SpinBound limit;
        while (!mbar_try(full_d + 8 * (k % SD), (k / SD) & 1) && !limit.expired(p)) {
        }
      }
      __syncwarp();
    }
    cluster_arrive();
  } else {
    // ======== the warps that copy, add and store ========
    uint16_t* hbuf = p.h + (size_t)ctl[6] * p.h_slot;
    const int cr = tid >> 3, cc = tid & 7;                     // row (modulo a sweep) and piece this thread copies
    constexpr int kCopy = RP / C::kSweep;
    auto mark_tokens = [&]() {     // tokens whose h of an expert is nonzero (and wanted below): a bit each
      for (int q = warp; q < nu; q += W) {
        const int id = ids_sm[q];
        const bool act = lane < L && (((tm[(id >> 5) * 32 + lane] >> (id & 31)) & 1u) || ((odd_tokens >> lane) & 1));
        const uint32_t m = __ballot_sync(0xffffffffu, act);
        if (lane == 0) tok_sm[q] = m;
      }
    };
    auto rest_of_inputs = [&]() {  // MODE 0, 1: what the work before may have written, and the scores of this CTA's tokens
      pdl_wait();
      deadline = coarse_time() + 3;
      copy_x();
      after_wait();
      if (warp < TR && rank * TR + warp < L)
        for (int e = lane; e < E; e += 32) a_sm[warp * Es + e] = __ldcg(p.scores + (size_t)(rank * TR + warp) * E + e);
      copy_sync();
    };
    int slot = 0, round = 0;       // of the next stage to wait for
    int islot = 0, iround = 0;     // of the next stage to ask for
    for (int ps = 0; ps < npass; ++ps) {
      const int ra = r0 + ps * rmax, nr = min(rmax, nrows - ps * rmax);
      uint32_t roff[kCopy];        // this thread's rows, in 16-byte units from U
#pragma unroll
      for (int i = 0; i < kCopy; ++i) {
        const int m = cr + C::kSweep * i, r = ra + m, q = r >> sh;
        roff[i] = m < nr ? (uint32_t)(ids_sm[q] * d_e + (r - (q << sh))) * (uint32_t)(d >> 3) + (uint32_t)kb0 * 8u + cc : 0u;
      }
      auto issue_u = [&](int kb) {
        const uint32_t dst = ring + islot * slot_bytes + cr * 128 + ((cc ^ (cr & 7)) << 4);
#pragma unroll
        for (int i = 0; i < kCopy; ++i)
          if (cr + C::kSweep * i < nr) cp_async16(dst + C::kSweep * 128 * i, at16(p.U, roff[i] + 8 * kb));
        if (++islot == S) {
          islot = 0;
          ++iround;
        }
      };
      if (tid == 0 && (ps == 0 || !broken())) mbar_expect(bar_up, nr * T * 4);
      if (MODE == 3 && ps == 0) mark_tokens();
      // A stage is handed on when it has landed, `lag` stages (64 to 80 KB) behind the one asked for.
      const int lag = max(1, min(S - 1, kLagBytes / slot_bytes));
      int asked = 0;
      auto ask = [&]() {
        if (asked < nkb) {
          if (asked >= S) mbar_wait(freed + 8 * islot, (iround - 1) & 1);
          issue_u(asked);
        }
        cp_async_commit();
        ++asked;
      };
      if (MODE != 3 && ps == 0) {  // U is on its way before the call before has left x
        while (asked <= lag) ask();
        rest_of_inputs();
      }
      for (int kb = 0; kb < nkb; ++kb) {
        while (asked <= kb + lag) ask();
        cp_async_wait_newest(lag);
        __syncwarp();
        if (lane == 0) mbar_arrive(full + 8 * slot);
        if (kb + 1 == nkb) mbar_wait(freed + 8 * slot, round & 1);
        if (++slot == S) {
          slot = 0;
          ++round;
        }
      }
      // (the cluster has read the pass before)
      if (ps > 0) wait_for([&]() { return mbar_try_cluster(recv_read, (ps - 1) & 1); });
      tc_after();
      // partial sums: a lane has a row, a warp 8 tokens; to the CTA that finishes the token
      {
        const bool sends = !broken();
        const int quad = warp & 3, cg = warp >> 2;
        auto send = [&](uint32_t from, int m, bool ok) {
          uint32_t v[8];
          tc_ld8(v, from + 8 * cg + ((uint32_t)(32 * quad) << 16));
          if (ok && sends) {
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              const int tq = 2 * cg + k, to = tq / QR, q = tq % QR;
              const uint32_t a = sbase + lay.off_urecv + ((rank * QR + q) * RP + m) * 16;
              st_async_v4(map_rank(a, to), v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3], map_rank(bar_up, to));
            }
          }
          __syncwarp();
        };
        if (nr <= 64) {
          const int m = 16 * quad + lane;
          send(tmem, m, lane < 16 && m < nr);
        } else {
          const int m = 32 * quad + lane;
          send(tmem, m, m < nr);
          if (nr > 128) send(tmem + T, 128 + 16 * quad + lane, lane < 16 && 128 + 16 * quad + lane < nr);
        }
        tc_before();
      }
      if (ps + 1 < npass) {        // (every lane is past its reads: send ends with a __syncwarp)
        if (lane == 0) mbar_arrive(acc_read);
      }
      mbar_wait(bar_up, ps & 1);
      const bool whole = !broken();
      for (int i0 = 0; i0 < nr * QR; i0 += NTH) {
        const int i = i0 + tid;
        const bool ok = i < nr * QR;
        const int q = QR == 2 && i >= nr ? 1 : 0, m = ok ? i - q * nr : 0, r = ra + m, qe = r >> sh;
        const int t0 = rank * TR + 4 * q, id = ids_sm[qe];
        float4 v;
        {
          const float4* in = reinterpret_cast<const float4*>(smem + lay.off_urecv) + q * RP + m;
          const float4 a = in[0], b = in[QR * RP], c = in[2 * QR * RP], e = in[3 * QR * RP];
          v.x = (a.x + b.x) + (c.x + e.x);
          v.y = (a.y + b.y) + (c.y + e.y);
          v.z = (a.z + b.z) + (c.z + e.z);
          v.w = (a.w + b.w) + (c.w + e.w);
        }
        auto hv = [&](float z, int k) {
          const float sc = t0 + k < L ? a_sm[(4 * q + k) * Es + id] : 0.0f;
          const uint32_t b = f32_to_bf16_bits(sc * swish_fast(z));
          return b == 0xffffu ? 0xfffeu : b;        // (0xffff: not written yet)
        };
        const uint32_t w01 = hv(v.x, 0) | (hv(v.y, 1) << 16), w23 = hv(v.z, 2) | (hv(v.w, 3) << 16);
        // four lanes have four rows of four tokens: to one token and four rows each
        const bool o1 = lane & 1, o2 = lane & 2;
        const uint32_t got1 = __shfl_xor_sync(0xffffffffu, o1 ? w01 : w23, 1), own1 = o1 ? w23 : w01;
        const uint32_t ev = o1 ? got1 : own1, od = o1 ? own1 : got1;    // even, odd row: tokens 2 o1, 2 o1 + 1
        const uint32_t ta = __byte_perm(ev, od, 0x5410), tb = __byte_perm(ev, od, 0x7632);
        const uint32_t got2 = __shfl_xor_sync(0xffffffffu, o2 ? ta : tb, 2), own2 = o2 ? tb : ta;
        const int t = t0 + 2 * (o1 ? 1 : 0) + (o2 ? 1 : 0);
        const int rb = r & ~3, j = rb - (qe << sh);
        if (ok && t < L && whole)
          asm volatile("st.relaxed.gpu.global.v2.u32 [%0], {%1, %2};" ::"l"(
                           hbuf + ((((size_t)(qe << pshift) + (j >> 6)) * L + t) << 6) + (j & 63)),
                       "r"(o2 ? got2 : own2), "r"(o2 ? own2 : got2)
                       : "memory");
      }
      if (ps + 1 < npass) {        // this warp has read the receive buffer
        __syncwarp();
        if (lane < kCluster) mbar_arrive_cluster(map_rank(recv_read, lane));
      }
    }
    if (MODE == 3 && npass == 0) mark_tokens();
    if (MODE != 3 && npass == 0) rest_of_inputs();
    if (MODE != 3) clear_other(tid, NTH);
    if (tid == 0) mbar_expect(bar_out, ncols * T * 4 + kCluster * 4);
    copy_sync();

    // ---- down projection ----
    // Four blocks at a time; a thread fetches 32 bytes of h of one block and token, until nothing there is
    // unwritten. (A token that does not activate an expert has zeros there, which need not be fetched,
    // unless a logit of the token is no finite number: then its x may not be either, and zero times that
    // is a NaN. Where the scores are given nothing is known about x, and all of h is fetched.)
    constexpr int kHS = NTG == 4 ? 6 : 4;
    const int hj = tid / (4 * T), ht = (tid >> 2) & (T - 1), hp = tid & 3;
    const bool held = p.hold == 2 || (p.hold == 4 && cl == 0 && rank == 1);
    bool dead = false;
    SpinBound bound;
    int hs = 0, hround = 0;
    for (int base = 0; base < nsw; base += kHS) {
      Frag64 f[kHS];
      uint32_t pend = 0;
      const uint16_t* h_at = hbuf + ((size_t)(b0 + 4 * base + hj) * L + ht) * 64 + 16 * hp;
      const uint32_t h_step = (uint32_t)L * 256u;
#pragma unroll
      for (int k = 0; k < kHS; ++k) {
        const int i = 4 * (base + k) + hj;
        f[k].lo = f[k].hi = make_uint4(0, 0, 0, 0);
        if (i < nb && ht < L && (MODE != 3 || ((tok_sm[(b0 + i) >> pshift] >> ht) & 1u))) pend |= 1u << k;
      }
      // (all of them at once: waiting for the first four blocks alone first cost 24 tokens with scores given 4 %)
      auto look = [&]() {
#pragma unroll
        for (int k = 0; k < kHS; ++k)
          if ((pend >> k) & 1u) ld_relaxed_v8(f[k], h_at + k * h_step);
#pragma unroll
        for (int k = 0; k < kHS; ++k)
          if (((pend >> k) & 1u) && !unwritten(f[k]) && !held) pend &= ~(1u << k);
      };
      look();
#pragma unroll
      for (int k = 0; k < kHS; ++k) {
        const int s = base + k;
        if (s < nsw) {
          while (!dead && __any_sync(0xffffffffu, (pend >> k) & 1u)) {
            dead = __any_sync(0xffffffffu, bound.expired(p));
            if (dead) ctl[5] = 1;    // (seen by whoever waits for the products with what is stored below)
            look();
          }
          if (hround > 0) mbar_wait(freed_h + 8 * hs, (hround - 1) & 1);
          if (4 * s + hj < nb) {
            const uint32_t to = xs + hs * C::kHSlot + hj * C::kHBlock + ht * 128;
            sts128(to + (((2 * hp) ^ (ht & 7)) << 4), f[k].lo);
            sts128(to + (((2 * hp + 1) ^ (ht & 7)) << 4), f[k].hi);
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(full_h + 8 * hs);
          if (++hs == SH) {
            hs = 0;
            ++hround;
          }
        }
      }
    }
    if (dead && lane == 0) atomicOr(p.status, BLOCKFFN_DEV_WAIT_EXPIRED);
    // routing results, spread over clusters: a CTA has its tokens' scores
    if (MODE == 3 && !lost) {
      for (int i = GC - 1 - cl; i < TR; i += GC) {
        const int t = rank * TR + i;
        for (int w = warp; w < words && t < L; w += W) {
          const int e = 32 * w + lane;
          if (e < E && p.pub.scores) p.pub.scores[(size_t)t * E + e] = a_sm[i * Es + e];
          if (p.pub.tok_mask && lane == 0) p.pub.tok_mask[(size_t)t * words + w] = tm[w * 32 + t];
        }
      }
    }
    if (nsw > 0) mbar_wait(freed_h + 8 * (hs == 0 ? SH - 1 : hs - 1), (hs == 0 ? hround - 1 : hround) & 1);
    tc_after();
    {
      const int quad = warp & 3, cg = warp >> 2, m = 16 * quad + lane;
      uint32_t v[8];
      tc_ld8(v, acc + 8 * cg + ((uint32_t)(32 * quad) << 16));
      if (lane < 16 && m < ncols) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const int tq = 2 * cg + k, to = tq / QR, q = tq % QR;
          const uint32_t a = sbase + lay.off_drecv + ((rank * QR + q) * kDRows + m) * 16;
          const bool any = nb > 0;             // (no block: no sum either)
          st_async_v4(map_rank(a, to), any ? v[4 * k] : 0u, any ? v[4 * k + 1] : 0u, any ? v[4 * k + 2] : 0u,
                      any ? v[4 * k + 3] : 0u, map_rank(bar_out, to));
        }
      }
      tc_before();
    }
    // whether they are worth anything
    const uint32_t out_flags = lay.off_hit + kCluster * C::TR / 2 * 4;
    if (tid < kCluster)
      st_async_b32(map_rank(sbase + out_flags + rank * 4, tid),
                   *reinterpret_cast<const volatile uint32_t*>(ctl + 5) | (broken() ? 1u : 0u), map_rank(bar_out, tid));
    __syncwarp();
    cluster_arrive();
    mbar_wait(bar_out, 0);
    copy_sync();
    const uint4 bad = lds128(sbase + out_flags);
    if (!broken() && (bad.x | bad.y | bad.z | bad.w) == 0 && has_out) {
      const int t = tid >> 6;
      const float* r = reinterpret_cast<const float*>(smem + lay.off_drecv) + ((t >> 2) * kDRows + om) * 4 + (t & 3);
      constexpr int s = QR * kDRows * 4;
      float v = (r[0] + r[s]) + (r[2 * s] + r[3 * s]);
      if (p.accumulate) v += resid;
      const size_t o = (size_t)ot * d + c0 + om;
      p.out[o] = v;
      if (p.x_next) p.x_next[o] = (uint16_t)f32_to_bf16_bits(v);
    }
    if (bx == 0 && tid == 0) p.used[ctl[6]] = lost ? (uint32_t)(p.h_slot >> 3) : (uint32_t)((R * L) >> 3);
    if (!lost && rank == 0 && cl == max(GC - 1 - TR, 0)) {
      if (MODE == 1 && tid == 0 && ctl[3]) atomicOr(p.status, (uint32_t)ctl[3]);
      for (int e = tid; e < E; e += NTH) {
        if (p.pub.union_ids) p.pub.union_ids[e] = e < nu ? ids_sm[e] : -1;
        if (p.pub.union_mask && e < words) p.pub.union_mask[e] = (uint32_t)ctl[8 + e];
      }
      if (tid == 0) {
        if (p.pub.n_union) *p.pub.n_union = nu;
        if (p.pub.stats) {
          atomicAdd(reinterpret_cast<unsigned long long*>(&p.pub.stats->n_tokens), (unsigned long long)L);
          atomicAdd(reinterpret_cast<unsigned long long*>(&p.pub.stats->n_active), (unsigned long long)ctl[2]);
          atomicAdd(reinterpret_cast<unsigned long long*>(&p.pub.stats->n_chunks), 1ull);
          atomicAdd(reinterpret_cast<unsigned long long*>(&p.pub.stats->n_union), (unsigned long long)nu);
        }
      }
    }
    cp_async_wait_all();
  }
  __syncthreads();
  if (warp == W) {
    tc_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(C::kTmem));
  }
  cluster_wait();                  // nobody sends to this CTA any more
  if (broken()) {
    if (tid == 0) atomicOr(p.status, BLOCKFFN_DEV_WAIT_EXPIRED);
    // (what it sent last may be on its way yet, for 0.2 us, and no wait has covered it)
    const unsigned long long t0 = clock_ns();
    while (clock_ns() - t0 < 100000ull) {
    }
  }
}

// ---- host side -------------------------------------------------------------------------------
struct ClusterPlan {
  int clusters, ntg, ring, cols_q, cols_rem, smem;
  bool ok;
};

// Shapes: d a multiple of 64 from 256 (every CTA has a part of K) to 2048, at most 64 columns of out
// per cluster, d_e a power of two >= 64.
template <int NTG>
ClusterPlan cluster_plan_of(const blockffn_config& cfg, int L, int clusters) {
  using C = Dims<NTG>;
  ClusterPlan pl{};
  const int d = cfg.d, d_e = cfg.d_e;
  if (clusters < 1 || d % 64 || d < 256 || d > 2048 || d_e % 64 || (d_e & (d_e - 1)) || d_e > 4096 || cfg.E > 1024)
    return pl;
  pl.clusters = clusters;
  pl.ntg = NTG;
  pl.cols_q = d / 2 / clusters;
  pl.cols_rem = d / 2 % clusters;
  if (2 * (pl.cols_q + (pl.cols_rem ? 1 : 0)) > kDRows) return pl;
  const int budget = NTG == 4 ? kSmemMax : (kSmemMax + 1024) / 2 - 1024;
  pl.ring = (budget - cluster_layout<NTG>(d, cfg.E, 0).total) & ~1023;
  // two stages of the most rows, two slots of D, the router's partial sums
  if (pl.ring < 2 * C::RP * 128 || pl.ring < 2 * kDSlot || pl.ring < C::W * C::T * 80) return pl;
  pl.smem = cluster_layout<NTG>(d, cfg.E, pl.ring).total;
  pl.ok = true;
  return pl;
}
// Where a call comes here. The hops through distributed shared memory cost a few microseconds that the smaller
// broadcast and the one pass over the weights have to save, so the lines lie at the number of elements of the
// expected union's U (the hint of the configuration, or 30 % of the experts: the union itself is known on the device
// only, and a call whose union is another one takes the kernel of the expected one). us per layer of a captured
// stack, kernel of expert_chain.cu, or with scores given expert_wide.cuh / this one (M elements):
//   router on, 17 to 32 tokens: below d = 1024 always, above from 24 M elements times tokens; 9 to 16: from 6 M, up to d = 1024
//     from 9 M. These two lines are older than the present form of the other kernel, which would put them at the rows of U
//     that it has room for (16 a CTA with 17 to 32 tokens, 21 with 9 to 16 at d above 1024). They have not been moved: the
//     kernels round differently, and in a stack whose tokens activate one or two experts each (E = 20, 12 % active) a
//     logit on the other side of zero changes a token's output as a whole. 17 to 32: d = 256, E = 16, d_e = 64 (307 rows), 17
//     tokens 8.8 / 11.0; d = 768, E = 48, d_e = 64 (896), 24 tokens 10.3 / 12.2; d = 2048, E = 48, d_e = 128 (1792), 32 tokens
//     13.4 / 14.7; d = 512, E = 64 (2432), 18 tokens 12.9 / 12.6; d = 1024, E = 64, 32 tokens 14.6 / 13.6; d = 2048, E = 64, 17
//     and 32 tokens 15.3 / 15.1 and 16.2 / 15.4; d = 1536, E = 128 (4864), 32 tokens 21.3 / 17.0. 9 to 16: d = 2048, E = 64, d_e = 128
//     (16 rows a CTA), 16 tokens 11.4 / 13.9; d = 1792, E = 80 (21), 16 tokens 14.9 / 14.9; d = 1280, E = 100 (26), 16 tokens
//     16.0 / 14.3; d = 2048, E = 128, 9 tokens 20.0 / 17.8; d = 1024, E = 100, 16 tokens 12.3 / 13.8; E = 80, d_e = 256 (6.3 M),
//     9 tokens 15.4 / 16.7; E = 120 (9.4 M), 16 tokens 22.2 / 21.5
//   scores given, 17 to 32: from 4 M. d = 1536, E = 48 (2.9 M), 18 tokens 11.3 / 11.7; d = 2048, E = 100,
//     d_e = 64 (3.9 M), 24 tokens 11.2 / 11.5; E = 54, d_e = 128 (4.2 M), 17 tokens 13.1 / 12.4; E = 64 (5 M), 24 tokens
//     15.7 / 13.2; E = 128 (10 M), 32 tokens 24.2 / 16.9. A list given: from 4.5 M (it is known sooner than a union that
//     has to be derived, which the other kernel is the better for). d = 2048, 17 tokens, E = 104, d_e = 64 (4.1 M)
//     10.6 / 11.6; E = 64, d_e = 128 (5 M), 24 tokens, nothing promised 14.1 / 12.6
//   scores given, 9 to 16: from 6 M, and from 9.3 G elements times d: the 64 columns of D that are copied at a time are a
//     cluster's own at d = 2048 and twice those at d = 1024. d = 2048, E = 64 (5 M) 8.8 / 8.7; E = 80 (6.3 M), 9 tokens
//     12.5 / 11.6; E = 128 (10 M), 16 tokens 20.1 / 16.1; d = 1536, E = 52, d_e = 256 (6.3 M), 9 tokens 12.2 / 12.1;
//     d = 1024, d_e = 256, 9 tokens, E = 80 (6.3 M) 12.9 / 15.4, E = 128 (10 M) 21.5 / 21.0; d = 512, E = 128, d_e = 512
//     (10 M), 9 tokens 27.2 / 32.5. A list given: from 12 G. d = 1536, E = 110, d_e = 128 (6.5 M), 9 tokens 9.3 / 10.8,
//     16 tokens 10.4 / 10.9; d = 2048, E = 80 (6.3 M) 9.3 / 9.7 and 10.3 / 10.0, E = 128 (10 M) 15.5 / 14.3 and 16.5 / 14.6
ClusterPlan cluster_plan(const blockffn_ctx* c, int L, int mode) {
  const long long u = expected_union_elements(c);
  const int d = c->cfg.d;
  if (L > 16 && L <= 32) {
    if (mode == 3 ? d >= 1024 && u * L < 24000000 && expert_chain_supported(c, L, 3) : u < (mode == 1 ? 4500000 : 4000000))
      return ClusterPlan{};
    return cluster_plan_of<4>(c->cfg, L, c->clusters);
  }
  if (L > 8 && L <= 16) {
    if (mode == 3 ? u < (d <= 1024 ? 9000000 : 6000000) : u < 6000000 || u * d < (mode == 1 ? 12000000000 : 9300000000))
      return ClusterPlan{};
    return cluster_plan_of<2>(c->cfg, L, c->clusters);
  }
  return ClusterPlan{};
}

void cluster_config(cudaLaunchConfig_t& lc, cudaLaunchAttribute* attr, int clusters, int threads, int smem) {
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kCluster;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  lc.gridDim = dim3(kCluster * clusters);
  lc.blockDim = dim3(threads);
  lc.dynamicSmemBytes = smem;
  lc.attrs = attr;
  lc.numAttrs = 1;
}
// The driver's encoder of tensor maps (0.04 to 0.07 us of host time a call), NULL where there is none.
typedef CUresult (*TensorMapEncoder)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                     const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                                     CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                     CUtensorMapFloatOOBfill);
TensorMapEncoder tensor_map_encoder() {
  static const TensorMapEncoder f = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult found;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &found) != cudaSuccess ||
        found != cudaDriverEntryPointSuccess)
      p = nullptr;
    return reinterpret_cast<TensorMapEncoder>(p);
  }();
  return f;
}
template <int NTG, int MODE>
cudaError_t cluster_attr() {
  const void* f = reinterpret_cast<const void*>(&expert_cluster_kernel<NTG, MODE>);
  cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout,
                              cudaSharedmemCarveoutMaxShared);
}

}  // namespace

bool expert_cluster_supported(const blockffn_ctx* c, int L, int mode) {
  if (c->chain_ws == nullptr || (c->cfg.flags & BLOCKFFN_CFG_TWO_KERNELS)) return false;
  return cluster_plan(c, L, mode).ok;
}

// How many clusters fit the device at one CTA per SM (0: none do, or no chunk length takes them).
cudaError_t expert_cluster_setup(blockffn_ctx* c) {
  c->clusters = 0;
  if (!c->chain_ws || c->cfg.L_max <= 8 || !tensor_map_encoder()) return cudaSuccess;
  cudaError_t e = cluster_attr<4, 3>();
  if (e == cudaSuccess) e = cluster_attr<4, 0>();
  if (e == cudaSuccess) e = cluster_attr<4, 1>();
  if (e == cudaSuccess) e = cluster_attr<2, 3>();
  if (e == cudaSuccess) e = cluster_attr<2, 0>();
  if (e == cudaSuccess) e = cluster_attr<2, 1>();
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t lc{};
  cudaLaunchAttribute attr[2];
  cluster_config(lc, attr, c->num_sms / kCluster, Dims<4>::NTH + 64, kSmemMax);
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, reinterpret_cast<const void*>(&expert_cluster_kernel<4, 3>), &lc) !=
      cudaSuccess) {
    cudaGetLastError();
    return cudaSuccess;
  }
  c->clusters = n < c->num_sms / kCluster ? n : c->num_sms / kCluster;
  return cudaSuccess;
}

cudaError_t launch_expert_cluster(blockffn_ctx* c, const blockffn_weights* w, const void* x, const float* scores,
                                  int L, const int32_t* union_ids, const int32_t* n_union, float* out,
                                  void* x_next, int call_flags, const RoutingOut* pub, cudaStream_t st) {
  const int mode = !scores ? 3 : union_ids ? 1 : 0;
  const ClusterPlan pl = cluster_plan(c, L, mode);
  if (!pl.ok || !c->chain_ws) return cudaErrorNotSupported;
  const ChainWorkspace ws = chain_workspace(c);
  ClusterParams p{};
  p.x = static_cast<const uint16_t*>(x);
  p.U = static_cast<const uint16_t*>(w->U);
  p.D = static_cast<const uint16_t*>(w->D);
  if (!scores) {
    p.W_r = static_cast<const uint16_t*>(w->W_r);
    p.gain = router_gain(c, w);
    p.bias = w->bias;
  }
  p.scores = scores;
  p.ids_in = union_ids;
  p.n_in = n_union;
  p.eps = c->cfg.rms_eps;
  p.seq = ws.seq;
  p.sms = c->num_sms;
  p.used = ws.used;
  p.logits = ws.logits;
  p.logit_copy = ws.logit_copy;
  p.h = ws.h;
  p.h_slot = ws.h_slot;
  p.out = out;
  p.x_next = static_cast<uint16_t*>(x_next);
  p.L = L;
  p.d = c->cfg.d;
  p.E = c->cfg.E;
  p.d_e = c->cfg.d_e;
  p.de_shift = __builtin_ctz(c->cfg.d_e);
  p.cols_q = pl.cols_q;
  p.cols_rem = pl.cols_rem;
  p.magic_g = (uint32_t)((0x100000000ull + (unsigned)pl.clusters - 1) / (unsigned)pl.clusters);
  p.ring = pl.ring;
  p.accumulate = (call_flags & BLOCKFFN_CALL_ACCUMULATE) ? 1 : 0;
  p.early = (call_flags & (BLOCKFFN_CALL_INDEPENDENT | BLOCKFFN_CALL_INDEPENDENT_X)) ? 1 : 0;
  const int groups = (c->cfg.E + 15) / 16;
  p.reps = pl.clusters >= groups ? pl.clusters / groups : 1;
  p.hold = !(c->cfg.flags & BLOCKFFN_CFG_TEST_EXPIRE_WAIT) ? 0 : scores || (c->cfg.flags & BLOCKFFN_CFG_NO_SPLIT) ? 2 : 1;
  if (p.hold && (c->cfg.flags & BLOCKFFN_CFG_NO_CHAINING)) p.hold += 2;
  p.wait_ns = 1000000000ull;      // one second
  p.time_shift = p.hold ? 22 : 31;
  p.status = c->status;
  if (pub) p.pub = *pub;
  cudaLaunchConfig_t lc{};
  cudaLaunchAttribute attr[2];
  cluster_config(lc, attr, pl.clusters, 128 * pl.ntg + 64, pl.smem);
  lc.stream = st;
  lc.numAttrs = (c->cfg.flags & BLOCKFFN_CFG_NO_CHAINING) ? 1 : 2;
  if (scores && !p.early) {
    // A call that promises nothing is not to depend on what other streams run: a cooperative launch starts
    // when all its CTAs fit, so that none of them waits for one that has no place.
    attr[1].id = cudaLaunchAttributeCooperative;
    attr[1].val.cooperative = 1;
    lc.numAttrs = 2;
  }
  // D as rows of d_e, copied 64 rows x 64 at a time (rows beyond the last expert's come as zeros)
  CUtensorMap map;
  const cuuint64_t dims[2] = {(cuuint64_t)c->cfg.d_e, (cuuint64_t)c->cfg.E * c->cfg.d};
  const cuuint64_t strides[1] = {(cuuint64_t)c->cfg.d_e * 2};
  const cuuint32_t box[2] = {64, kDRows}, steps[2] = {1, 1};
  if (tensor_map_encoder()(&map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(w->D), dims, strides, box,
                           steps, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                           CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return cudaErrorInvalidValue;
  const cudaError_t e = pl.ntg == 4 ? mode == 3   ? cudaLaunchKernelEx(&lc, expert_cluster_kernel<4, 3>, p, map)
                                      : mode == 1 ? cudaLaunchKernelEx(&lc, expert_cluster_kernel<4, 1>, p, map)
                                                  : cudaLaunchKernelEx(&lc, expert_cluster_kernel<4, 0>, p, map)
                        : mode == 3   ? cudaLaunchKernelEx(&lc, expert_cluster_kernel<2, 3>, p, map)
                        : mode == 1   ? cudaLaunchKernelEx(&lc, expert_cluster_kernel<2, 1>, p, map)
                                      : cudaLaunchKernelEx(&lc, expert_cluster_kernel<2, 0>, p, map);
  if (e == cudaSuccess) c->launches += 1;
  return e;
}

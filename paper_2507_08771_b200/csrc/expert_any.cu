// Expert stage (Eq. 1, Eq. 2 restricted to Union(x), Sec. 3.3) for any shape, with a 32-bit
// intermediate: the kernels behind BLOCKFFN_VARIANT_SIMT, behind every shape the staged
// tensor-core kernels do not take (d and d_e only have to be multiples of 8) and behind
// blockffn_expert_ffn_noalloc.
//
//   any_up_kernel    a CTA takes 16 of the union's u * d_e neuron rows at a time, its eight warps
//                    split K = d, multiply the rows with all L tokens (mma.sync m16n8k16, weights
//                    are the M operand), sum across warps, apply Swish and the token's score and
//                    store h[q][t][j].
//   any_down_kernel  a CTA takes 16 output columns at a time, its warps split K = u * d_e, and
//                    writes every out[t][c] once (no atomics: results are run-to-run identical).
//
// h is kept to 32 bits: it is stored as three bf16 planes that give the fp32 value exactly (24
// significand bits, cut off 8 at a time), and the down projection multiplies all three with D. The
// second and third plane are scaled by 2^7 and 2^15, or they would be denormal, which the tensor
// cores lose, for h below 1e-31. No plane is then larger than the first, so a sum of products with
// it overflows only where the sum of |h D| does. Their part is left out where it is no number: an
// infinite weight times a plane that is zero (a NaN of h or D is in the first plane's part as well).
// Products of bf16 are exact; the sum of 32 of them leaves the tensor core after two mma and is
// added in fp32 there (a longer chain inside the tensor core would lose bits to its truncation).
//
// What bounds these kernels is memory latency: a call is a few MB over a device that holds 10 MB
// in flight. Every thread therefore keeps S steps of its own operands on the way: it copies its
// fragments (16 bytes = 8 consecutive k of a row; the k permutation is the same for both mma
// operands) with cp.async into shared memory nobody else reads, so nothing has to be laid out,
// padded or waited for at a barrier, and K and row tails are zero-filled copies. The weights of
// the first S steps are requested before griddepcontrol.wait, under the kernel before. The dot
// products on CUDA cores that these kernels replace were one load deep per warp: 96 us per call
// at d = 2048, E = 64, d_e = 128, union 19, 8 tokens, where these take 10.3, and 62 us per layer at
// d = 1000, E = 40, d_e = 96, router included, now 12.0 (both in a dependent chain of layers; 3.0
// and 0.7 us are the weights at the copy rate). Error against 64 bits of the expert stage alone:
// 1.87e-7 before, 1.41e-7 now at the first shape, 1.45e-7 and 1.27e-7 at the second.
#include <mutex>

#include "mma_tiles.cuh"

namespace {

constexpr int kRedTok = 20;   // floats per token of a 16-row partial tile: stores hit 32 banks

// steps a thread keeps in flight, and 16-byte pieces of a step: rows g and g + 8 of the weights
// and, per group of 8 tokens, x (up) or the three planes of h (down). An up and a down CTA
// share an SM (104 + 108 KB of its 233 at E = 64 with one token group, 109 + 109 with two, 95 + 136
// with four, there only up to 96 experts).
__host__ __device__ constexpr int up_pieces(int ntg) { return 2 + ntg; }
__host__ __device__ constexpr int up_steps(int ntg) { return ntg == 1 ? 8 : ntg == 2 ? 6 : 3; }
__host__ __device__ constexpr int down_pieces(int ntg) { return 2 + 3 * ntg; }
__host__ __device__ constexpr int down_steps(int ntg) { return ntg == 1 ? 5 : ntg == 2 ? 3 : 2; }

struct AnyLayout {
  int off_red, off_ring, total;
};
__host__ __device__ inline AnyLayout any_layout(int E, int ntg, int steps, int pieces) {
  AnyLayout s;
  s.off_red = kOffIds + align128(E * 4);
  s.off_ring = s.off_red + kWarps * 8 * ntg * kRedTok * 4;
  s.total = s.off_ring + steps * pieces * kThreads * 16;
  return s;
}

// v / n for v n < 2^44 (rows and 8-wide pieces of a union: at most 1024 experts of 2^16 rows)
__device__ __forceinline__ uint32_t div44(uint32_t v, unsigned long long magic) {
  return (uint32_t)((v * magic) >> 44);
}
inline unsigned long long magic44(unsigned n) { return ((1ull << 44) + n - 1) / n; }

// 16-byte asynchronous copy, zeros instead when !ok (nothing is read then; src stays a valid address)
__device__ __forceinline__ void cp_async16_or_zero(uint32_t dst, const void* src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ uint4 lds_v4(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "r"(a)
               : "memory");
  return v;
}
// one step (32 k): c += a (rows g, g + 8) * b (8 tokens)
__device__ __forceinline__ void mma32(float (&c)[4], const uint4& a, const uint4& a8, const uint4& b) {
  mma_bf16(c, a.x, a8.x, a.y, a8.y, b.x, b.y);
  mma_bf16(c, a.z, a8.z, a.w, a8.w, b.z, b.w);
}
// accumulator tile of one warp -> red[token][row] of its 16 x 8 NTG block
template <int NTG>
__device__ __forceinline__ void store_tile(float* mine, const float (&c)[NTG][4], int g, int tg) {
#pragma unroll
  for (int n = 0; n < NTG; ++n) {
    float* o = mine + (8 * n + 2 * tg) * kRedTok + g;
    o[0] = c[n][0];
    o[kRedTok] = c[n][1];
    o[8] = c[n][2];
    o[kRedTok + 8] = c[n][3];
  }
}
// sum over the warps of element (token, row), e = token * kRedTok + row
template <int NTG>
__device__ __forceinline__ float sum_warps(const float* red, int e) {
  constexpr int s = 8 * NTG * kRedTok;
  const float* r = red + e;
  return ((r[0] + r[s]) + (r[2 * s] + r[3 * s])) + ((r[4 * s] + r[5 * s]) + (r[6 * s] + r[7 * s]));
}

struct AnyUpParams {
  const uint16_t* x;       // bf16 [L][d]
  const uint16_t* U;       // bf16 [E][d_e][d]
  const float* scores;     // f32 [L][E] (unused when lg.a0 is set)
  RouterLogits lg;         // raw router logits to finish here, or a0 == NULL
  const int32_t* ids_in;   // caller's union list, or NULL: derive from scores / logits
  const int32_t* n_in;
  uint16_t* h;             // three planes of bf16 [q][L][d_e]
  size_t plane;            // elements of one plane
  unsigned long long de_magic;
  int L, d, E, d_e;
  int early;               // 0 wait first; 1 routing inputs and weights before the wait; 2 x as well
  uint32_t* status;
  RoutingOut pub;
};

// MODE as derive_union: 0 from scores, 1 the caller's list, 2 raw router logits
template <int NTG, int MODE>
__global__ void __launch_bounds__(kThreads, 2) any_up_kernel(const AnyUpParams p) {
  extern __shared__ __align__(128) unsigned char smem[];
  constexpr int S = up_steps(NTG), P = up_pieces(NTG);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, tg = lane & 3;
  const int d = p.d, d_e = p.d_e, L = p.L;
  const AnyLayout lay = any_layout(p.E, NTG, S, P);
  int* ctl = reinterpret_cast<int*>(smem + kOffCtl);
  int* ids_sm = reinterpret_cast<int*>(smem + kOffIds);
  float* red = reinterpret_cast<float*>(smem + lay.off_red);
  const uint32_t ring = smem_u32(smem) + lay.off_ring + tid * 16;

  if (tid < 8) ctl[tid] = 0;
  if (p.early == 0) pdl_wait();   // scores / ids / logits may come from the kernel just before
  pdl_trigger();
  __syncthreads();
  const int nu = derive_union<MODE>(p.scores, p.lg, p.ids_in, p.n_in, L, p.E, ids_sm, ctl,
                                    reinterpret_cast<uint32_t*>(red));

  const int R = nu * d_e, tiles = (R + 15) >> 4;
  const int pieces = d >> 3, blocks = (d + 31) >> 5;
  const int nb = blocks > warp ? (blocks - warp + kWarps - 1) / kWarps : 0;   // steps per tile
  // copies of the weights run S steps ahead of the math: their position
  int w_tile = blockIdx.x, w_b = 0;
  const uint16_t *row_a = p.U, *row_b = p.U;
  bool ok_a = false, ok_b = false;
  auto w_rows = [&]() {
    const int ra = 16 * w_tile + g, rb = ra + 8;
    ok_a = ra < R;
    ok_b = rb < R;
    const uint32_t qa = ok_a ? div44(ra, p.de_magic) : 0, qb = ok_b ? div44(rb, p.de_magic) : 0;
    if (ok_a) row_a = p.U + ((size_t)ids_sm[qa] * d_e + (ra - qa * d_e)) * d;
    if (ok_b) row_b = p.U + ((size_t)ids_sm[qb] * d_e + (rb - qb * d_e)) * d;
  };
  auto issue_w = [&](int slot) {
    if (w_tile < tiles && nb > 0) {
      if (w_b == 0) w_rows();
      const int pc = 4 * (warp + kWarps * w_b) + tg;
      const bool in = pc < pieces;
      const uint32_t dst = ring + slot * (P * kThreads * 16);
      cp_async16_or_zero(dst, in && ok_a ? row_a + 8 * pc : p.U, in && ok_a);
      cp_async16_or_zero(dst + kThreads * 16, in && ok_b ? row_b + 8 * pc : p.U, in && ok_b);
      if (++w_b == nb) {
        w_b = 0;
        w_tile += gridDim.x;
      }
    }
  };
  int x_tile = blockIdx.x, x_b = 0;
  auto issue_x = [&](int slot) {
    if (x_tile < tiles && nb > 0) {
      const int pc = 4 * (warp + kWarps * x_b) + tg;
      const uint32_t dst = ring + slot * (P * kThreads * 16) + 2 * kThreads * 16;
#pragma unroll
      for (int n = 0; n < NTG; ++n) {
        const bool in = pc < pieces && 8 * n + g < L;
        cp_async16_or_zero(dst + n * kThreads * 16, in ? p.x + (size_t)(8 * n + g) * d + 8 * pc : p.x, in);
      }
      if (++x_b == nb) {
        x_b = 0;
        x_tile += gridDim.x;
      }
    }
  };
  // One commit group per step (empty ones included), or, while x may still change, one for the
  // weights of each of the first S steps and then one for its x: either way the S - 1 newest
  // groups belong to later steps.
#pragma unroll 1
  for (int s = 0; s < S; ++s) {
    issue_w(s);
    if (p.early != 1) issue_x(s);
    cp_async_commit();
  }
  if (p.early == 1) {
    pdl_wait();
#pragma unroll 1
    for (int s = 0; s < S; ++s) {
      issue_x(s);
      cp_async_commit();
    }
  }

  // h elements this thread finishes per tile: e = token * 16 + row, e = tid, tid + 256, ...
  constexpr int kFin = (NTG + 1) / 2;
  bool waited = p.early != 2;
  int slot = 0;
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    float sc[kFin];
    size_t at[kFin];
#pragma unroll
    for (int k = 0; k < kFin; ++k) {
      const int e = tid + k * kThreads, t = e >> 4, r = 16 * tile + (e & 15);
      sc[k] = 0.0f;
      at[k] = ~(size_t)0;
      if (t < L && r < R) {
        const int q = div44(r, p.de_magic), id = ids_sm[q];
        at[k] = ((size_t)q * L + t) * d_e + (r - q * d_e);
        if constexpr (MODE == 2) {     // gain * ReLU(logit) / rms, as in derive_union
          float v = __ldcg(p.lg.a0 + (size_t)t * p.E + id);
          v = v > 0.0f ? v : 0.0f;
          sc[k] = __ldg(p.lg.gain + id) * v * reinterpret_cast<const float*>(ctl + 104)[t];
        } else {
          sc[k] = __ldcg(p.scores + (size_t)t * p.E + id);
        }
      }
    }
    float acc[NTG][4];
    zero_acc<NTG>(acc);
#pragma unroll 1
    for (int b = 0; b < nb; ++b) {
      cp_async_wait_group<S - 1>();
      const uint32_t src = ring + slot * (P * kThreads * 16);
      const uint4 wa = lds_v4(src), wb = lds_v4(src + kThreads * 16);
#pragma unroll
      for (int n = 0; n < NTG; ++n) {
        const uint4 xv = lds_v4(src + (2 + n) * kThreads * 16);
        float c[4] = {0.f, 0.f, 0.f, 0.f};
        mma32(c, wa, wb, xv);
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[n][v] += c[v];
      }
      issue_w(slot);               // (this thread has read the slot)
      issue_x(slot);
      cp_async_commit();
      slot = slot + 1 == S ? 0 : slot + 1;
    }
    store_tile<NTG>(red + warp * (8 * NTG * kRedTok), acc, g, tg);
    if (!waited) pdl_wait();       // h may still be read by the call before
    waited = true;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kFin; ++k) {
      const int e = tid + k * kThreads;
      if (at[k] != ~(size_t)0) {
        const float h = sc[k] * swish(sum_warps<NTG>(red, (e >> 4) * kRedTok + (e & 15)));
        // three bf16, h = h1 + h2 / 2^7 + h3 / 2^15: its significand cut off 8 bits at a time. An
        // infinity or NaN has no remainder (and a NaN keeps a bit where the cut would lose it).
        uint32_t h1 = __float_as_uint(h) >> 16, h2 = 0, h3 = 0;
        if ((__float_as_uint(h) & 0x7f800000u) != 0x7f800000u) {
          const float r = (h - __uint_as_float(h1 << 16)) * 128.0f;
          h2 = __float_as_uint(r) >> 16;
          h3 = __float_as_uint((r - __uint_as_float(h2 << 16)) * 256.0f) >> 16;
        } else if (h != h) {
          h1 |= 0x40u;
        }
        p.h[at[k]] = (uint16_t)h1;
        p.h[p.plane + at[k]] = (uint16_t)h2;
        p.h[2 * p.plane + at[k]] = (uint16_t)h3;
      }
    }
    __syncthreads();               // red is free for the next tile
  }
  if (!waited) pdl_wait();         // every kernel waits before it ends
  cp_async_wait_all();
  if (blockIdx.x == 0) publish_routing<MODE>(p.pub, p.lg, L, p.E, nu, ids_sm, ctl, p.status);
}

struct AnyDownParams {
  const uint16_t* D;       // bf16 [E][d][d_e]
  const uint16_t* h;       // three planes of bf16 [q][L][d_e]
  size_t plane;
  const float* scores;
  RouterLogits lg;
  const int32_t* ids_in;
  const int32_t* n_in;
  float* out;              // f32 [L][d]
  uint16_t* x_next;        // bf16 [L][d] or NULL
  unsigned long long pe_magic;
  int L, d, E, d_e, accumulate;
};

template <int NTG, int MODE>
__global__ void __launch_bounds__(kThreads, 2) any_down_kernel(const AnyDownParams p) {
  extern __shared__ __align__(128) unsigned char smem[];
  constexpr int S = down_steps(NTG), P = down_pieces(NTG);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, tg = lane & 3;
  const int d = p.d, d_e = p.d_e, L = p.L;
  const AnyLayout lay = any_layout(p.E, NTG, S, P);
  int* ctl = reinterpret_cast<int*>(smem + kOffCtl);
  int* ids_sm = reinterpret_cast<int*>(smem + kOffIds);
  float* red = reinterpret_cast<float*>(smem + lay.off_red);
  const uint32_t ring = smem_u32(smem) + lay.off_ring + tid * 16;

  if (tid < 8) ctl[tid] = 0;
  pdl_trigger();
  __syncthreads();
  // The routing inputs were final before the up kernel of this call let this one start.
  const int nu = derive_union<MODE>(p.scores, p.lg, p.ids_in, p.n_in, L, p.E, ids_sm, ctl,
                                    reinterpret_cast<uint32_t*>(red));

  const int dpe = d_e >> 3;                      // 8-wide pieces of an expert's rows
  const int pieces = nu * dpe, blocks = (pieces + 3) >> 2, tiles = (d + 15) >> 4;
  const int nb = blocks > warp ? (blocks - warp + kWarps - 1) / kWarps : 0;
  int w_tile = blockIdx.x, w_b = 0;
  auto issue_w = [&](int slot) {
    if (w_tile < tiles && nb > 0) {
      const int pc = 4 * (warp + kWarps * w_b) + tg, col = 16 * w_tile + g;
      const bool in = pc < pieces, in_a = in && col < d, in_b = in && col + 8 < d;
      const uint32_t q = in ? div44(pc, p.pe_magic) : 0;
      const uint16_t* src = p.D;
      if (in) src += ((size_t)ids_sm[q] * d + col) * d_e + 8 * (pc - q * dpe);
      const uint32_t dst = ring + slot * (P * kThreads * 16);
      cp_async16_or_zero(dst, in_a ? src : p.D, in_a);
      cp_async16_or_zero(dst + kThreads * 16, in_b ? src + 8 * (size_t)d_e : p.D, in_b);
      if (++w_b == nb) {
        w_b = 0;
        w_tile += gridDim.x;
      }
    }
  };
  int h_tile = blockIdx.x, h_b = 0;
  auto issue_h = [&](int slot) {
    if (h_tile < tiles && nb > 0) {
      const int pc = 4 * (warp + kWarps * h_b) + tg;
      const uint32_t q = pc < pieces ? div44(pc, p.pe_magic) : 0;
      const uint32_t dst = ring + slot * (P * kThreads * 16) + 2 * kThreads * 16;
#pragma unroll
      for (int n = 0; n < NTG; ++n) {
        const bool in = pc < pieces && 8 * n + g < L;
        const uint16_t* src = p.h + (in ? ((size_t)q * L + 8 * n + g) * d_e + 8 * (pc - q * dpe) : 0);
#pragma unroll
        for (int k = 0; k < 3; ++k)
          cp_async16_or_zero(dst + (3 * n + k) * kThreads * 16, src + (in ? k * p.plane : 0), in);
      }
      if (++h_b == nb) {
        h_b = 0;
        h_tile += gridDim.x;
      }
    }
  };
#pragma unroll 1
  for (int s = 0; s < S; ++s) {
    issue_w(s);
    cp_async_commit();
  }
  pdl_wait();                      // h, out and x_next are safe to touch from here on
#pragma unroll 1
  for (int s = 0; s < S; ++s) {
    issue_h(s);
    cp_async_commit();
  }

  constexpr int kFin = (NTG + 1) / 2;
  int slot = 0;
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    float resid[kFin];             // requested now, used in the epilogue
#pragma unroll
    for (int k = 0; k < kFin; ++k) {
      const int e = tid + k * kThreads, t = e >> 4, c = 16 * tile + (e & 15);
      resid[k] = p.accumulate && t < L && c < d ? __ldcg(p.out + (size_t)t * d + c) : 0.0f;
    }
    float hi[NTG][4], mid[NTG][4], lo[NTG][4];   // products with the three planes
    zero_acc<NTG>(hi);
    zero_acc<NTG>(mid);
    zero_acc<NTG>(lo);
#pragma unroll 1
    for (int b = 0; b < nb; ++b) {
      cp_async_wait_group<S - 1>();
      const uint32_t src = ring + slot * (P * kThreads * 16);
      const uint4 wa = lds_v4(src), wb = lds_v4(src + kThreads * 16);
#pragma unroll
      for (int n = 0; n < NTG; ++n) {
        const uint32_t hs = src + (2 + 3 * n) * kThreads * 16;
        float c[4] = {0.f, 0.f, 0.f, 0.f};
        mma32(c, wa, wb, lds_v4(hs));
        mma32(mid[n], wa, wb, lds_v4(hs + kThreads * 16));
        mma32(lo[n], wa, wb, lds_v4(hs + 2 * kThreads * 16));
#pragma unroll
        for (int v = 0; v < 4; ++v) hi[n][v] += c[v];
      }
      issue_w(slot);               // (this thread has read the slot)
      issue_h(slot);
      cp_async_commit();
      slot = slot + 1 == S ? 0 : slot + 1;
    }
#pragma unroll
    for (int n = 0; n < NTG; ++n)
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const float rest = mid[n][v] * 0x1p-7f + lo[n][v] * 0x1p-15f;
        hi[n][v] += rest == rest ? rest : 0.0f;
      }
    store_tile<NTG>(red + warp * (8 * NTG * kRedTok), hi, g, tg);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kFin; ++k) {
      const int e = tid + k * kThreads, t = e >> 4, c = 16 * tile + (e & 15);
      if (t < L && c < d) {
        float v = sum_warps<NTG>(red, t * kRedTok + (e & 15));
        if (p.accumulate) v += resid[k];
        const size_t o = (size_t)t * d + c;
        p.out[o] = v;
        if (p.x_next) p.x_next[o] = (uint16_t)f32_to_bf16_bits(v);
      }
    }
    __syncthreads();               // red is free for the next tile
  }
  cp_async_wait_all();
}

template <int NTG, int MODE>
cudaError_t any_attr() {
  const void* f[2] = {reinterpret_cast<const void*>(&any_up_kernel<NTG, MODE>),
                      reinterpret_cast<const void*>(&any_down_kernel<NTG, MODE>)};
  for (const void* k : f) {
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout,
                               cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <int NTG, int MODE>
cudaError_t any_launch(const AnyUpParams& up, const AnyDownParams& dn, int grid_up, int grid_down,
                       bool chained, cudaStream_t st) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t lc{};
  lc.blockDim = dim3(kThreads);
  lc.stream = st;
  lc.attrs = attr;
  lc.numAttrs = chained ? 1 : 0;
  lc.gridDim = dim3(grid_up);
  lc.dynamicSmemBytes = any_layout(up.E, NTG, up_steps(NTG), up_pieces(NTG)).total;
  const cudaError_t e = cudaLaunchKernelEx(&lc, any_up_kernel<NTG, MODE>, up);
  if (e != cudaSuccess) return e;
  lc.gridDim = dim3(grid_down);
  lc.dynamicSmemBytes = any_layout(up.E, NTG, down_steps(NTG), down_pieces(NTG)).total;
  return cudaLaunchKernelEx(&lc, any_down_kernel<NTG, MODE>, dn);
}

template <int MODE>
cudaError_t any_launch_mode(const AnyUpParams& up, const AnyDownParams& dn, int grid_up,
                            int grid_down, bool chained, cudaStream_t st) {
  if (up.L <= 8) return any_launch<1, MODE>(up, dn, grid_up, grid_down, chained, st);
  if (up.L <= 16) return any_launch<2, MODE>(up, dn, grid_up, grid_down, chained, st);
  return any_launch<4, MODE>(up, dn, grid_up, grid_down, chained, st);
}

}  // namespace

size_t expert_any_h_bytes(const blockffn_config* cfg) {
  return 3 * sizeof(uint16_t) * (size_t)cfg->E * cfg->L_max * cfg->d_e;
}

cudaError_t expert_any_setup(int L_max) {
  cudaError_t e = any_attr<1, 0>();
  if (e == cudaSuccess) e = any_attr<1, 1>();
  if (e == cudaSuccess) e = any_attr<1, 2>();
  if (e == cudaSuccess && L_max > 8) e = any_attr<2, 0>();
  if (e == cudaSuccess && L_max > 8) e = any_attr<2, 1>();
  if (e == cudaSuccess && L_max > 8) e = any_attr<2, 2>();
  if (e == cudaSuccess && L_max > 16) e = any_attr<4, 0>();
  if (e == cudaSuccess && L_max > 16) e = any_attr<4, 1>();
  if (e == cudaSuccess && L_max > 16) e = any_attr<4, 2>();
  return e;
}

cudaError_t launch_expert_any(blockffn_ctx* c, const blockffn_weights* w, const void* x,
                              const float* scores, int L, const int32_t* union_ids,
                              const int32_t* n_union, float* out, void* x_next, int call_flags,
                              const RoutingOut* pub, const RouterLogits* logits, cudaStream_t st) {
  const blockffn_config& cfg = c->cfg;
  AnyUpParams up{};
  up.x = static_cast<const uint16_t*>(x);
  up.U = static_cast<const uint16_t*>(w->U);
  up.scores = scores;
  if (logits) up.lg = *logits;
  up.ids_in = union_ids;
  up.n_in = n_union;
  up.h = static_cast<uint16_t*>(c->h32);
  up.plane = (size_t)cfg.E * cfg.L_max * cfg.d_e;
  up.de_magic = magic44(cfg.d_e);
  up.L = L;
  up.d = cfg.d;
  up.E = cfg.E;
  up.d_e = cfg.d_e;
  up.early = logits ? 0
             : (call_flags & BLOCKFFN_CALL_INDEPENDENT_X) ? 2
             : (call_flags & BLOCKFFN_CALL_INDEPENDENT)   ? 1
                                                          : 0;
  up.status = c->status;
  if (pub) up.pub = *pub;
  AnyDownParams dn{};
  dn.D = static_cast<const uint16_t*>(w->D);
  dn.h = up.h;
  dn.plane = up.plane;
  dn.scores = scores;
  dn.lg = up.lg;
  dn.ids_in = union_ids;
  dn.n_in = n_union;
  dn.out = out;
  dn.x_next = static_cast<uint16_t*>(x_next);
  dn.pe_magic = magic44(cfg.d_e / 8);
  dn.L = L;
  dn.d = cfg.d;
  dn.E = cfg.E;
  dn.d_e = cfg.d_e;
  dn.accumulate = (call_flags & BLOCKFFN_CALL_ACCUMULATE) ? 1 : 0;
  // Grids: a CTA per 16 rows / columns, two per SM at most (larger calls go through their tiles
  // in turn; an SM has no room for two down CTAs of 17 to 32 tokens, so from d = 2376 on some of
  // them come after the others). The union is not known here: a quarter more row tiles than the
  // caller's hint, or the paper's sparsity, gives (CTAs that find no rows only keep the down
  // kernel's from an SM).
  int u_exp = (cfg.flags >> 17) & 0x7ff;
  if (u_exp == 0) u_exp = (L == 1 ? cfg.E + 4 : 3 * cfg.E + 5) / (L == 1 ? 8 : 10);
  u_exp += u_exp / 4 + 1;
  if (u_exp > cfg.E) u_exp = cfg.E;
  long long grid_up = ((long long)u_exp * cfg.d_e + 15) / 16, grid_down = ((long long)cfg.d + 15) / 16;
  if (grid_up > 2 * c->num_sms) grid_up = 2 * c->num_sms;
  if (grid_down > 2 * c->num_sms) grid_down = 2 * c->num_sms;
  const bool chained = !(cfg.flags & BLOCKFFN_CFG_NO_CHAINING);
  const cudaError_t e =
      logits      ? any_launch_mode<2>(up, dn, (int)grid_up, (int)grid_down, chained, st)
      : union_ids ? any_launch_mode<1>(up, dn, (int)grid_up, (int)grid_down, chained, st)
                  : any_launch_mode<0>(up, dn, (int)grid_up, (int)grid_down, chained, st);
  if (e == cudaSuccess) c->launches += 2;
  return e;
}

// ---- expert stage without a handle and without any allocation ---------------------------
//
// Scratch for blockffn_expert_ffn_noalloc: the intermediate h[q][t][j] of the two kernels above
// (6 bytes an element), preceded by a 256-byte header whose first word is the status word those
// kernels want (never read: the callers have no handle to ask). The array is part of the library
// image: every GPU that loads the library holds these bytes until the process exits.
#define BLOCKFFN_NOALLOC_HEADER 256
static __device__ __align__(256) unsigned char
    g_noalloc_scratch[BLOCKFFN_NOALLOC_HEADER + BLOCKFFN_NOALLOC_SCRATCH_BYTES / 4 * 6];

namespace {
constexpr int kMaxDevices = 64;
// Device address of g_noalloc_scratch per device, looked up once per device. In host code
// the array's name is only a handle for the runtime, never an address a kernel may be given.
// The pair (address, SM count) of a device is written and read under the mutex, so that a
// second host thread never sees one without the other.
struct NoallocDevice {
  unsigned char* ptr;
  int sms;
};
NoallocDevice g_noalloc_dev[kMaxDevices] = {};
std::mutex g_noalloc_mutex;
}  // namespace

extern "C" blockffn_status blockffn_expert_ffn_noalloc(
    const blockffn_config* cfg, const blockffn_weights* w, const void* x, const float* scores,
    int32_t L, const int32_t* union_ids, const int32_t* n_union, float* out, void* x_next,
    int32_t call_flags, void* stream) {
  auto bad16 = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) != 0; };
  auto bad4 = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 3u) != 0; };
  if (!cfg || !w || !w->U || !w->D || !x || !scores || !union_ids || !n_union || !out)
    return BLOCKFFN_ERR_INVALID_ARG;
  if (cfg->d < 8 || cfg->d_e < 8 || cfg->E < 1 || L < 1) return BLOCKFFN_ERR_INVALID_ARG;
  if (cfg->d % 8 || cfg->d_e % 8 || cfg->E > 1024 || L > 32 || cfg->d > (1 << 20) ||
      cfg->d_e > (1 << 16))
    return BLOCKFFN_ERR_UNSUPPORTED;
  // the intermediate of this call must fit the fixed scratch
  if ((size_t)cfg->E * (size_t)L * (size_t)cfg->d_e * sizeof(float) >
      (size_t)BLOCKFFN_NOALLOC_SCRATCH_BYTES)
    return BLOCKFFN_ERR_WORKSPACE;
  if (bad16(w->U) || bad16(w->D) || bad16(x) || bad16(out) || bad16(x_next) || bad4(scores) ||
      bad4(union_ids) || bad4(n_union) || x_next == x)
    return BLOCKFFN_ERR_INVALID_ARG;
  if (call_flags & ~(BLOCKFFN_CALL_ACCUMULATE | BLOCKFFN_CALL_INDEPENDENT | BLOCKFFN_CALL_INDEPENDENT_X))
    return BLOCKFFN_ERR_INVALID_ARG;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return BLOCKFFN_ERR_CUDA;
  NoallocDevice nd;
  {
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_dev[dev].ptr) {   // first call on this device, with this device current
      unsigned char* ptr = nullptr;
      int sms = 0;
      if (cudaGetSymbolAddress(reinterpret_cast<void**>(&ptr), g_noalloc_scratch) != cudaSuccess ||
          !ptr ||
          cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
          expert_any_setup(32) != cudaSuccess) {
        cudaGetLastError();
        return BLOCKFFN_ERR_CUDA;
      }
      g_noalloc_dev[dev].sms = sms;
      g_noalloc_dev[dev].ptr = ptr;
    }
    nd = g_noalloc_dev[dev];
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  blockffn_ctx tmp{};          // a view for the launcher: nothing in it owns memory
  tmp.cfg = *cfg;
  tmp.cfg.L_max = L;           // a plane of h is E L d_e elements
  tmp.cfg.flags = 0;
  tmp.device = dev;
  tmp.num_sms = nd.sms;
  tmp.words = (cfg->E + 31) / 32;
  tmp.status = reinterpret_cast<uint32_t*>(nd.ptr);
  tmp.h32 = nd.ptr + BLOCKFFN_NOALLOC_HEADER;
  const cudaError_t e =
      launch_expert_any(&tmp, w, x, scores, L, union_ids, n_union, out, x_next, call_flags, nullptr,
                        nullptr, st);
  return e == cudaSuccess ? BLOCKFFN_OK : BLOCKFFN_ERR_CUDA;
}

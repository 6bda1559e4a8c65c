// Router (Eq. 3), chunk union (Sec. 3.3), reuse ratio (Sec. 4.1.2) and the copy of routing results.
//
// All of them are a few KB of data and a chain of memory latencies: what counts is how many of
// those follow one another, and that the launch runs under the kernel before (programmatic
// dependent launch). Each kernel asks for all it reads at once; before, a block went through the
// tokens one after the other (24 tokens, E = 64, d = 2048, one call
// after the other from a graph: router 12.05 us, union 3.81, reuse ratio 5.57, copy of the routing results 4.36;
// now 6.3, 2.0, 2.6 and 1.5).
//
// router_kernel: a block computes one expert's logits for 8 tokens (x . W_r[i] + bias[i]) with
// 128-bit loads and fp32 FMAs; of the blocks with the same tokens the one that finishes last (a
// ticket counter per 8 tokens, no waiting) applies ReLU and RMSNorm with the per-expert gain,
// writes the scores and the per-token nonzero masks (warp ballot).
//
// union_kernel: one block ORs the per-token nonzero patterns of a score matrix,
// compacts the union's expert ids in ascending order with a warp prefix count, and
// advances the TLS / CLS counters (Sec. 2.1).
#include "mma_tiles.cuh"

namespace {

constexpr int kMaxWords = 32;  // E <= 1024

// A launch that may start while the work before it on the stream still runs. These kernels do not
// let their own dependents go early, and fence what they write (union lists, copied scores) before
// they exit: a call after them may read it as a stable input before it waits, and nothing but the
// exit of their blocks orders it behind them then.
template <class... P, class... A>
cudaError_t launch_chained(const blockffn_ctx* c, void (*kernel)(P...), int grid, cudaStream_t st, A... args) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t lc{};
  lc.gridDim = dim3(grid);
  lc.blockDim = dim3(kThreads);
  lc.stream = st;
  lc.attrs = attr;
  lc.numAttrs = (c->cfg.flags & BLOCKFFN_CFG_NO_CHAINING) ? 0 : 1;
  return cudaLaunchKernelEx(&lc, kernel, args...);
}

__global__ void __launch_bounds__(kThreads)
union_kernel(const float* scores, int L, int E, RoutingOut pub) {
  __shared__ __align__(16) int ctl[kCtlBytes / 4];
  __shared__ int ids[32 * kMaxWords];
  __shared__ uint32_t tm[32 * kMaxWords];
  pdl_wait();
  const int nu = derive_union<0>(scores, RouterLogits{}, nullptr, nullptr, L, E, ids, ctl, tm);
  publish_routing<0>(pub, RouterLogits{}, L, E, nu, ids, ctl, nullptr);
  __threadfence();
}

__global__ void __launch_bounds__(kThreads)
router_kernel(const uint16_t* __restrict__ x, const uint16_t* __restrict__ W_r,
              const float* __restrict__ gain, const float* __restrict__ bias, float* a0,
              float* scores, uint32_t* tok_mask, int L, int d, int E, float eps,
              unsigned int* ticket, int raw, int mode) {
  __shared__ float red[kWarps][8];
  __shared__ int is_last;
  const int npass = (L + 7) >> 3;                      // passes of 8 tokens
  const int i = blockIdx.x / npass, pass = blockIdx.x - i * npass, t0 = 8 * pass;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int chunks = d >> 3;
  const uint4* wrow = reinterpret_cast<const uint4*>(W_r + (size_t)i * d);
  const float b = bias ? bias[i] : 0.0f;
  // The kernel may have been started while the work before it on the stream still runs
  // (programmatic dependent launch): the router weights are stable and are requested now,
  // x and everything this kernel writes are touched only after the wait.
  // mode 2 (raw, launched on a stream of its own): dependents are let go only by the exit of
  // the blocks, behind a fence, because they read the logits without waiting (see the end).
  // raw: the expert kernels that follow wait themselves before they let anything go. A router call
  // of its own lets its dependents go by the exit of its blocks, behind a fence: a promised call behind
  // it lets its own go before it has waited, and the call behind that one may read these scores as stable
  // before it waits. (Letting them go behind the wait had the next launch under this kernel, 0.6 to 0.8 us
  // less a call, but then nothing ordered those reads behind the scores.)
  if (raw && mode != 2) pdl_trigger();
  uint4 w_first = make_uint4(0u, 0u, 0u, 0u);
  if ((int)threadIdx.x < chunks) w_first = __ldg(wrow + threadIdx.x);
  {  // x may still change until the wait is over, but asking L2 for its lines now is harmless
    // (L2 is where writes land too); the blocks share the lines out between them
    const int lines = (L * d * 2 + 127) >> 7;
    for (int ln = blockIdx.x + (int)gridDim.x * (int)threadIdx.x; ln < lines; ln += gridDim.x * kThreads)
      asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const char*>(x) + (size_t)ln * 128));
  }
  // mode 1 (raw only): x does not come from the work before and a0 is a buffer that work
  // does not read, so the logits are computed under it; the wait moves to the end.
  if (mode == 0) pdl_wait();

  float acc[8];
#pragma unroll
  for (int t = 0; t < 8; ++t) acc[t] = 0.0f;
  for (int c = threadIdx.x; c < chunks; c += kThreads) {
    const uint4 wv = c == (int)threadIdx.x ? w_first : __ldg(wrow + c);
    const uint32_t wp[4] = {wv.x, wv.y, wv.z, wv.w};
    // all eight token vectors are requested before the first is used: one memory latency
    uint4 xv[8];
#pragma unroll
    for (int t = 0; t < 8; ++t)
      xv[t] = t0 + t < L ? __ldcg(reinterpret_cast<const uint4*>(x + (size_t)(t0 + t) * d) + c)
                         : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const uint32_t xp[4] = {xv[t].x, xv[t].y, xv[t].z, xv[t].w};
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        acc[t] = fmaf(bf16_lo(wp[p]), bf16_lo(xp[p]), acc[t]);
        acc[t] = fmaf(bf16_hi(wp[p]), bf16_hi(xp[p]), acc[t]);
      }
    }
  }
#pragma unroll
  for (int t = 0; t < 8; ++t) {
    float v = acc[t];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) red[warp][t] = v;
  }
  __syncthreads();
  if (threadIdx.x < 8 && t0 + threadIdx.x < L) {
    float v = b;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) v += red[w][threadIdx.x];
    a0[(size_t)(t0 + threadIdx.x) * E + i] = v;
  }

  // raw: the logits are all the caller wants (the tensor-core expert kernels normalise them
  // themselves, which saves this kernel's serial tail)
  if (raw) {
    // every kernel of a chain waits before it ends: completion of one implies all before it
    if (mode == 1) asm volatile("griddepcontrol.wait;" ::: "memory");
    // mode 2: a kernel launched with the programmatic attribute treats every kernel it depends
    // on as a programmatic prerequisite, event edges from other streams included, so the expert
    // kernels may start as soon as this grid's blocks have exited. The fence makes each block's
    // logits visible device-wide before that exit.
    if (mode == 2) __threadfence();
    return;
  }
  // the last block of these tokens normalises them, a token per warp. The ticket is reset for the
  // next call.
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned int tk = atomicAdd(ticket + pass, 1u);
    is_last = (tk == (unsigned)E - 1u);
    if (is_last) ticket[pass] = 0u;
  }
  __syncthreads();
  if (!is_last) return;
  __threadfence();

  const int words = (E + 31) >> 5, t = t0 + warp;
  if (t >= L) return;
  const bool few = words <= 4;   // logits and gains of a token in registers: one round trip
  float v4[4], g4[4], ss = 0.0f;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int e = 32 * u + lane;
    v4[u] = few && e < E ? __ldcg(a0 + (size_t)t * E + e) : 0.0f;
    g4[u] = few && e < E ? gain[e] : 0.0f;
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    v4[u] = v4[u] > 0.0f ? v4[u] : 0.0f;
    ss = fmaf(v4[u], v4[u], ss);
  }
  for (int e = lane; !few && e < E; e += 32) {
    float v = __ldcg(a0 + (size_t)t * E + e);
    v = v > 0.0f ? v : 0.0f;
    ss = fmaf(v, v, ss);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  // eps < 0 marks the router without RMSNorm (Sec. 4.2.3): the ReLU values are the scores
  // (the host passes a gain of ones)
  const float r = eps < 0.0f ? 1.0f : 1.0f / sqrtf(ss / (float)E + eps);
  auto put = [&](int w, float s) {
    const int e = 32 * w + lane;
    if (e < E) scores[(size_t)t * E + e] = s;
    const uint32_t m = __ballot_sync(0xffffffffu, s != 0.0f);
    if (tok_mask && lane == 0) tok_mask[(size_t)t * words + w] = m;
  };
  if (few) {
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (u < words) put(u, g4[u] * v4[u] * r);
  } else {
    for (int w = 0; w < words; ++w) {
      const int e = 32 * w + lane;
      float v = e < E ? __ldcg(a0 + (size_t)t * E + e) : 0.0f;
      v = v > 0.0f ? v : 0.0f;
      put(w, e < E ? gain[e] * v * r : 0.0f);
    }
  }
  __threadfence();
}

}  // namespace

cudaError_t launch_router(blockffn_ctx* c, const blockffn_weights* w, const void* x, int L,
                          float* scores, uint32_t* tok_mask, bool raw, float* logits, int mode,
                          cudaStream_t st) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t lc{};
  lc.gridDim = dim3(c->cfg.E * ((L + 7) / 8));
  lc.blockDim = dim3(kThreads);
  lc.stream = st;
  lc.attrs = attr;
  lc.numAttrs = (mode == 2 || (c->cfg.flags & BLOCKFFN_CFG_NO_CHAINING)) ? 0 : 1;
  const cudaError_t e = cudaLaunchKernelEx(
      &lc, router_kernel, static_cast<const uint16_t*>(x), static_cast<const uint16_t*>(w->W_r),
      router_gain(c, w), w->bias, logits, scores, tok_mask, L, c->cfg.d, c->cfg.E, c->cfg.rms_eps,
      c->ticket, raw ? 1 : 0, raw ? mode : 0);
  if (e == cudaSuccess) c->launches += 1;
  return e;
}

namespace {

constexpr int kPairs = 64;     // token pairs of a round

// Reuse ratio (Sec. 4.1.2). One block. A round takes 65 successive tokens: their nonzero masks (a
// warp per token, four tokens' loads in flight), the 64 ratios (a thread each), and thread 0 adds
// them in token order, so the sum has one summation order.
__global__ void __launch_bounds__(kThreads)
reuse_ratio_kernel(const float* scores, int L, int E, double* reuse) {
  __shared__ uint32_t mask[kPairs + 1][kMaxWords];
  __shared__ double ratio[kPairs];               // negative: the pair does not count
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, words = (E + 31) >> 5;
  pdl_wait();
  double sum = 0.0, pairs = 0.0;
  if (threadIdx.x == 0) {
    sum = reuse[0];
    pairs = reuse[1];
  }
  for (int i0 = 0; i0 + 1 < L; i0 += kPairs) {
    const int nt = min(kPairs + 1, L - i0);
    for (int w0 = 0; w0 < words; w0 += 4) {
      for (int tb = warp; tb < nt; tb += 4 * kWarps) {
        float v[4][4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int t = tb + j * kWarps, e = 32 * (w0 + u) + lane;
            v[j][u] = t < nt && e < E ? scores[(size_t)(i0 + t) * E + e] : 0.0f;
          }
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const uint32_t m = __ballot_sync(0xffffffffu, v[j][u] != 0.0f);
            if (lane == 0 && tb + j * kWarps < nt && w0 + u < words) mask[tb + j * kWarps][w0 + u] = m;
          }
      }
    }
    __syncthreads();
    if (threadIdx.x + 1 < nt) {
      int a = 0, b = 0;
      for (int w = 0; w < words; ++w) {
        const uint32_t now = mask[threadIdx.x][w];
        a += __popc(now);
        b += __popc(now & mask[threadIdx.x + 1][w]);
      }
      ratio[threadIdx.x] = a ? (double)b / (double)a : -1.0;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int k = 0; k + 1 < nt; ++k) {
        if (ratio[k] < 0.0) continue;
        sum += ratio[k];
        pairs += 1.0;
      }
    }
  }
  if (threadIdx.x == 0) {
    reuse[0] = sum;
    reuse[1] = pairs;
  }
}

// 32-bit words of up to five arrays to the caller's buffers
struct CopyParams {
  const uint32_t* src[5];
  uint32_t* dst[5];
  uint32_t words[5];
};
__global__ void __launch_bounds__(kThreads) copy_routing_kernel(const CopyParams p) {
  pdl_wait();
#pragma unroll
  for (int k = 0; k < 5; ++k)
    for (uint32_t i = blockIdx.x * kThreads + threadIdx.x; i < p.words[k]; i += gridDim.x * kThreads)
      p.dst[k][i] = p.src[k][i];
  __threadfence();
}

}  // namespace

cudaError_t launch_reuse_ratio(blockffn_ctx* c, const float* scores, int L, double* reuse,
                               cudaStream_t st) {
  const cudaError_t e = launch_chained(c, reuse_ratio_kernel, 1, st, scores, L, (int)c->cfg.E, reuse);
  if (e == cudaSuccess) c->launches += 1;
  return e;
}

cudaError_t launch_chunk_union(blockffn_ctx* c, const float* scores, int L, uint32_t* union_mask,
                               int32_t* union_ids, int32_t* n_union, blockffn_stats* stats,
                               cudaStream_t st) {
  const RoutingOut pub{union_mask, union_ids, n_union, stats, nullptr, nullptr};
  const cudaError_t e = launch_chained(c, union_kernel, 1, st, scores, L, (int)c->cfg.E, pub);
  if (e == cudaSuccess) c->launches += 1;
  return e;
}

// One kernel instead of a copy per array: a copy of 1 KB takes as long as a launch.
cudaError_t launch_copy_routing(blockffn_ctx* c, int L, float* scores, uint32_t* tok_mask,
                                uint32_t* union_mask, int32_t* union_ids, int32_t* n_union,
                                cudaStream_t st) {
  const uint32_t E = c->cfg.E, W = c->words;
  CopyParams p{};
  const void* src[5] = {c->scores, c->tok_mask, c->union_mask, c->union_ids, c->n_union};
  void* dst[5] = {scores, tok_mask, union_mask, union_ids, n_union};
  const uint32_t words[5] = {L * E, L * W, W, E, 1};
  uint32_t most = 0;
  for (int k = 0; k < 5; ++k) {
    p.src[k] = static_cast<const uint32_t*>(src[k]);
    p.dst[k] = static_cast<uint32_t*>(dst[k]);
    p.words[k] = dst[k] ? words[k] : 0;
    if (p.words[k] > most) most = p.words[k];
  }
  if (most == 0) return cudaSuccess;
  const uint32_t blocks = (most + kThreads - 1) / kThreads;
  const cudaError_t e = launch_chained(c, copy_routing_kernel, (int)(blocks < 32 ? blocks : 32), st, p);
  if (e == cudaSuccess) c->launches += 1;
  return e;
}

// Endpoint contraction for few rows (Eq. 11 over the kept vocabulary ids,
// fused with Eq. 13) over a short hidden dimension: 4..32 hidden-state rows,
// tcgen05 + TMEM on sm_103a.
//
// The endpoint's share of the hidden dimension is short (d_l of 48..512), so
// a tile of 128 ids is a few microseconds of work and the call is decided by
// what surrounds it.  Against the general tensor-core kernel this one has no
// operand-split launch before it, no tensor maps to fetch, no runs of ids to
// plan and no operand that is read again for every tile:
//
//   B   the hidden states of all rows, loaded once per CTA as fp32, split in
//       registers into bf16 hi + lo (h = hi + lo + O(2^-18 |h|)) and kept in
//       shared memory for every tile the CTA takes
//   A   the tile's weight rows by 16-byte cp.async with per-thread row
//       pointers: any id pattern costs the same, and the first copies go out
//       as soon as the ids are there (where kernels of the same call ran
//       before this one: before it waits for them).  Rows past the tile hold
//       stale bytes and land in accumulator lanes that are never read.
//   D   fp32 in TMEM, two tiles' accumulators.  Every 64 columns multiply hi,
//       then lo, in the order of the general kernel, so z has the same bits.
//
// Warps 0-7 copy and run the epilogue; warp 8 owns TMEM and issues the MMAs
// (one elected lane).  The copies of the next tiles are in flight while a tile's
// epilogue runs.  Every wait is bounded; a wait that gives up sets the
// context's error word, and the CTA winds down after its copies and MMAs have
// landed.
//
// What bounds it: launch, set-up and one round trip each for ids, weights and
// payload (4 rows x 700 ids x 48 columns with its draw: 7.9 us, general
// kernel 10.9); past that the epilogues (32 rows x 60000 ids x 96: 15.4 us,
// 22.3) and, at 512 columns, the copies: they arrive on a stage's barrier
// thread by thread, about 600 cycles a stage (12 rows x 44999 ids x 512: 21.0
// us, 23.9).  A long hidden dimension would pay that at every stage, so the
// general kernel's tensor copies keep those (an earlier form of this kernel
// for 3840 columns: 35 us against 28).
#include <atomic>

#include "sm100_ptx.cuh"
#include "sph_common.cuh"
#include "sph_internal.h"

namespace sph {
namespace {

constexpr int kWorkWarps = 8;
constexpr int kWorkers = kWorkWarps * 32;
constexpr int kThreads = kWorkers + 32;
constexpr int kTileIds = 128;          // M of one MMA
constexpr int kAtomCols = 64;          // bf16 columns of one 128-byte swizzled row
constexpr int kMaxStages = 12;
constexpr size_t kSmemBudget = 220 * 1024;
constexpr size_t kMaxHidden = 128 * 1024;   // bytes of the resident hi + lo planes
constexpr long long kDrainLimit = 1ll << 31;
constexpr float kLog2eF = 1.4426950408889634f;
constexpr int kMaxDevices = 64;

struct FewParams {
  const float* h;
  int64_t ld_h;
  int R, K, n;
  const uint16_t* W;
  int64_t ld_w;
  const int32_t* ids;
  int pitch;                 // ids of a tile, a multiple of 32
  int na, KB;                // 64-column atoms of a stage, stages of a tile
  int tiles, stages, lag;    // lag: stages copied before a tile's epilogue waits
  int h16;                   // h and its rows are 16-byte aligned
  int early;                 // ids and weights may be read before the wait (after_own)
  float* Z;                  // fused logits, row stride ldz, or nullptr
  int64_t ldz;
  const int8_t* codes;       // payload [R][n], or nullptr (none, or fused)
  const float* row_scale;
  float inv_tau;
  float2* seg_stats;         // [R][nseg], or nullptr
  int nseg;
  // fused: the cloud's clipped partials in, the payload out
  const float* yc;
  const unsigned* rowmax_in;
  int8_t* codes_out;
  float* scale_out;
  unsigned* status;
  long long spin_limit;
};

// 16 bytes to shared memory, the bytes past `valid` as zeros
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, int valid) {
  asm volatile("cp.async.cg.shared.global.L2::256B [%0], [%1], 16, %2;" ::"r"(dst), "l"(src),
               "r"(valid)
               : "memory");
}
// Arrive on `bar` (which counts this arrival) once all of this thread's
// copies so far have landed.
__device__ __forceinline__ void cp_arrive(uint64_t* bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(ptx::smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void cp_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }
// Generic-proxy writes (copies, stores) before async-proxy reads (MMAs).
__device__ __forceinline__ void fence_proxy_async() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void st_shared16(uint32_t addr, uint4 v) {
  asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z),
               "r"(v.w)
               : "memory");
}
__device__ __forceinline__ uint32_t pack2(float x0, float x1) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(x0, x1);
  return *reinterpret_cast<const uint32_t*>(&v);
}
// offset of 16-byte column ch of row r in a 128-byte-swizzled atom
__device__ __forceinline__ uint32_t swizzled(int r, int ch) {
  return (uint32_t)((r >> 3) * 1024 + (r & 7) * 128 + ((ch ^ (r & 7)) << 4));
}

// NR = MMA columns (rows of hidden states): 16 or 32.
template <int NR, int EPI>
__global__ void __launch_bounds__(kThreads, 1) few_kernel(const FewParams p) {
  constexpr uint32_t kCols = 2 * NR;           // two tiles' accumulators
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint64_t s_full[kMaxStages], s_empty[kMaxStages], s_tfull[2], s_tempty[2], s_hready,
      s_drain;
  __shared__ uint32_t s_tmem;
  __shared__ volatile int s_abort;
  __shared__ RowQuant s_rq[NR];                // fused: the quantizer; else s alone
  const uint32_t base = (ptx::smem_u32(smem_raw) + 1023) & ~1023u;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int S = p.stages, KB = p.KB, na = p.na;
  // hidden states: per 64 columns a hi and a lo atom of NR rows; then the
  // stages, na atoms of the tile's rows each
  constexpr uint32_t kHAtom = NR * 128;
  const uint32_t a_atom = (uint32_t)(p.pitch >> 3) * 1024u;
  const uint32_t stage_bytes = (uint32_t)na * a_atom;
  const uint32_t a_base = base + (uint32_t)(KB * na) * 2 * kHAtom;
  const int my_tiles = (p.tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
  const int total = my_tiles * KB;             // this CTA's stages

  // ---- copy state of a worker thread: rows row0 + 32 i, 16-byte column ch
  const int row0 = (threadIdx.x & (kWorkers - 1)) >> 3, ch = threadIdx.x & 7;
  int nid[4];                                  // the next tile's ids (-1: none)
  auto load_ids = [&](int tl) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = row0 + 32 * i, j = tl * p.pitch + r;
      nid[i] = (tl < p.tiles && r < p.pitch && j < p.n) ? (p.ids ? p.ids[j] : j) : -1;
    }
  };
  if (warp == kWorkWarps) ptx::tmem_alloc(&s_tmem, kCols);
  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      ptx::mbar_init(&s_full[s], kWorkers);
      ptx::mbar_init(&s_empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      ptx::mbar_init(&s_tfull[a], 1);
      ptx::mbar_init(&s_tempty[a], kWorkWarps);
    }
    ptx::mbar_init(&s_hready, kWorkWarps);
    ptx::mbar_init(&s_drain, 1);
    s_abort = 0;
    ptx::fence_mbar_init();
  }
  // As the first kernel of its call on the stream it follows the caller's
  // work, which may be writing the ids and the weights: nothing is read, and
  // no dependent kernel is let go, before the wait.  Behind kernels of its
  // own call it started after the caller's work had completed (the first of
  // them waited for that before it let anything start).
  if (warp < kWorkWarps) {
    if (!p.early) {
      ptx::griddep_wait();
      ptx::griddep_launch_dependents();
    }
    load_ids((int)blockIdx.x);
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = s_tmem;
  const long long limit = p.spin_limit;
  auto give_up = [&]() {
    atomicOr(p.status, ERR_TIMEOUT);
    s_abort = 1;
  };

  // (a poll may suspend the thread for longer than this kernel's waits take,
  // so the limit is looked at before each)
  auto wait = [&](uint64_t* bar, uint32_t parity) {
    if (ptx::mbar_test(bar, parity)) return true;
    const long long t0 = clock64();
    while (clock64() - t0 < limit)
      if (ptx::mbar_try_wait(bar, parity)) return true;
    return false;
  };
  auto warp_wait = [&](uint64_t* bar, uint32_t parity) {
    const bool ok = __all_sync(0xFFFFFFFFu, !s_abort && wait(bar, parity));
    if (!ok && lane == 0 && !s_abort) give_up();
    return ok;
  };

  if (warp == kWorkWarps) {
    // ---------------------------------------------------------- MMA issuer
    // (the whole warp runs the loop, one elected lane issues: see the PTX
    // wrappers)
    if (p.early) ptx::griddep_launch_dependents();
    constexpr uint32_t idesc = ptx::idesc_bf16_f32(kTileIds, NR);
    int stage = 0;
    uint32_t phase = 0;
    bool stop = !warp_wait(&s_hready, 0);
    for (int x = 0; x < my_tiles && !stop; ++x) {
      const int acc = x & 1;
      // (the accumulator's previous tile, x - 2, has been read)
      if (x >= 2 && !warp_wait(&s_tempty[acc], (uint32_t)((x >> 1) - 1) & 1u)) break;
      const uint32_t d = tmem + (uint32_t)(acc * NR);
      uint32_t hd = ptx::sdesc_k128(base);
      uint32_t accum = 0;                      // the tile's first MMA overwrites
      for (int kb = 0; kb < KB; ++kb) {
        if (!warp_wait(&s_full[stage], phase)) {
          stop = true;
          break;
        }
        fence_proxy_async();
        ptx::tc_fence_after();
        uint32_t wd = ptx::sdesc_k128(a_base + (uint32_t)stage * stage_bytes);
        for (int at = 0; at < na; ++at) {
#pragma unroll
          for (int hl = 0; hl < 2; ++hl)
#pragma unroll
            for (int kk = 0; kk < kAtomCols / 16; ++kk) {
              ptx::umma_f16(d, wd + (uint32_t)(kk * 32 >> 4),
                            hd + (uint32_t)((hl * kHAtom + kk * 32) >> 4), idesc, accum);
              accum = 1;
            }
          wd += a_atom >> 4;
          hd += 2 * kHAtom >> 4;
        }
        ptx::umma_commit(&s_empty[stage]);
        if (++stage == S) { stage = 0; phase ^= 1; }
      }
      if (!stop) ptx::umma_commit(&s_tfull[acc]);
    }
    ptx::umma_commit(&s_drain);
    ptx::mbar_wait(&s_drain, 0, kDrainLimit);
    __syncwarp();
  } else {
    // ---------------------------------------------------- copy and epilogue
    const uint32_t off0 = swizzled(row0, ch);
    const uint16_t* wp[4];                     // this tile's weight rows
    int ltile = blockIdx.x, lkb = 0, lstage = 0;
    uint32_t lphase = 0;
    unsigned rows_ok = 0;                      // which of the four rows hold an id
    // the weights of the next stage; moves the position on
    auto copy_a = [&]() {
      if (lkb == 0) {
        rows_ok = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          wp[i] = p.W + (int64_t)max(nid[i], 0) * p.ld_w;
          rows_ok |= (nid[i] >= 0 ? 1u : 0u) << i;
        }
        load_ids(ltile + (int)gridDim.x);
      }
      for (int at = 0; at < na; ++at) {
        const int k = (lkb * na + at) * kAtomCols + ch * 8;
        const int valid = min(max((p.K - k) * 2, 0), 16);
        const int ka = valid > 0 ? k : 0;      // (past K nothing is read)
        const uint32_t dst =
            a_base + (uint32_t)lstage * stage_bytes + (uint32_t)at * a_atom + off0;
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (row0 + 32 * i < p.pitch)
            cp_async16(dst + i * 4096, wp[i] + ka, ((rows_ok >> i) & 1u) ? valid : 0);
      }
      cp_arrive(&s_full[lstage]);
      if (++lkb == KB) { lkb = 0; ltile += gridDim.x; }
      if (++lstage == S) { lstage = 0; lphase ^= 1; }
    };
    // The weights and ids come from the caller: the first stages' weights go
    // out before the wait for this call's earlier kernels (whose payload the
    // epilogue reads).
    const int ahead = min(total, p.lag + 1);
    for (int i = 0; i < ahead; ++i) copy_a();
    ptx::griddep_wait();

    // epilogue: a warp reads the TMEM lanes of its quadrant (ids quad * 32 +
    // lane of the tile) and rows erow0 .. erow0 + 15
    const int quad = warp & 3, erow0 = (warp >> 2) * 16;
    const bool epi_on = quad * 32 < p.pitch && erow0 < p.R;
    // the payload of this lane's id, loaded a tile ahead: codes, or (fused)
    // the clipped partials
    float pay_f[16];
    int pay_c[16];
    auto load_payload = [&](int tile) {
      if (!epi_on || tile >= p.tiles) return;
      const int j = min(tile * p.pitch + quad * 32 + lane, p.n - 1);
      if constexpr (EPI == EPI_FUSED) {
#pragma unroll
        for (int q = 0; q < 16; ++q)
          pay_f[q] = __ldcg(p.yc + (int64_t)min(erow0 + q, p.R - 1) * p.n + j);
      } else if (p.codes) {
        const int8_t* cp = p.codes + (int64_t)erow0 * p.n + j;
#pragma unroll
        for (int q = 0; q < 16; ++q, cp += p.n)
          if (erow0 + q < p.R) pay_c[q] = *cp;
      }
    };
#pragma unroll
    for (int q = 0; q < 16; ++q) { pay_c[q] = 0; pay_f[q] = 0.f; }
    load_payload((int)blockIdx.x);
    // the row's scale (and, fused, its quantizer)
    if constexpr (EPI == EPI_FUSED) {
      if (threadIdx.x < p.R) {
        const RowQuant rq = row_quant(__ldcg(p.rowmax_in + threadIdx.x));
        s_rq[threadIdx.x] = rq;
        if (blockIdx.x == 0) p.scale_out[threadIdx.x] = rq.s;
      }
    } else {
      if (threadIdx.x < p.R)
        s_rq[threadIdx.x].s = p.codes ? p.row_scale[threadIdx.x] : 0.f;
    }
    // the hidden states: 8-column pieces (row, column c) of every atom, four
    // pieces a thread requested before the first is converted
    constexpr int kU = 4;
    const int pieces = KB * na * NR * 8;
    for (int q0 = threadIdx.x; q0 < pieces; q0 += kU * kWorkers) {
      float x[kU][8];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int q = q0 + u * kWorkers;
        const int c = q & 7, r = (q >> 3) & (NR - 1), atom = q / (NR * 8);
        const int k = atom * kAtomCols + c * 8, left = (q < pieces && r < p.R) ? p.K - k : 0;
        const float* hp = p.h + (int64_t)r * p.ld_h + k;
        if (p.h16 && left >= 8) {
          const float4 a = *reinterpret_cast<const float4*>(hp);
          const float4 b = *(reinterpret_cast<const float4*>(hp) + 1);
          x[u][0] = a.x; x[u][1] = a.y; x[u][2] = a.z; x[u][3] = a.w;
          x[u][4] = b.x; x[u][5] = b.y; x[u][6] = b.z; x[u][7] = b.w;
        } else {
#pragma unroll
          for (int e = 0; e < 8; ++e) x[u][e] = e < left ? hp[e] : 0.f;
        }
      }
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int q = q0 + u * kWorkers;
        if (q >= pieces) break;
        const int c = q & 7, r = (q >> 3) & (NR - 1), atom = q / (NR * 8);
        float hi[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) hi[e] = __bfloat162float(__float2bfloat16_rn(x[u][e]));
        const uint32_t dst = base + (uint32_t)atom * 2 * kHAtom + swizzled(r, c);
        st_shared16(dst, make_uint4(pack2(hi[0], hi[1]), pack2(hi[2], hi[3]),
                                    pack2(hi[4], hi[5]), pack2(hi[6], hi[7])));
        st_shared16(dst + kHAtom,
                    make_uint4(pack2(x[u][0] - hi[0], x[u][1] - hi[1]),
                               pack2(x[u][2] - hi[2], x[u][3] - hi[3]),
                               pack2(x[u][4] - hi[4], x[u][5] - hi[5]),
                               pack2(x[u][6] - hi[6], x[u][7] - hi[7])));
      }
    }
    __syncwarp();
    if (lane == 0) ptx::mbar_arrive(&s_hready);
    ptx::named_bar_sync(1, kWorkers);          // (s_rq)

    auto epilogue = [&](int x, int tile) -> bool {
      const int acc = x & 1;
      if (!warp_wait(&s_tfull[acc], (uint32_t)(x >> 1) & 1u)) return false;
      ptx::tc_fence_after();
      float z[16];
      if (epi_on)
        ptx::tmem_ld16(tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(acc * NR + erow0), z);
      ptx::tc_fence_before();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(&s_tempty[acc]);
      if (!epi_on) return true;
      const int j = tile * p.pitch + quad * 32 + lane;
      const bool vj = j < p.n;
      const int kr = (lane >> 1) & 15;         // the row this lane reduces
      if constexpr (EPI == EPI_ENDPOINT) {
        // all 32 ids exist (nearly always): no lane predicate and no address
        // product per value (an epilogue's length is its instructions'
        // latency)
        if (__all_sync(0xFFFFFFFFu, vj)) {
          const int nr = p.R - erow0;
          if (p.codes) {
#pragma unroll
            for (int q = 0; q < 16; ++q)
              z[q] = z[q] + (float)pay_c[q] * s_rq[min(erow0 + q, NR - 1)].s;
          }
          if (p.Z) {
            float* zp = p.Z + (int64_t)erow0 * p.ldz + j;
#pragma unroll
            for (int q = 0; q < 16; ++q, zp += p.ldz)
              if (q < nr) *zp = z[q];
          }
          load_payload(tile + (int)gridDim.x);
          if (p.seg_stats) {
            const float mk = warp_reduce_scatter16(z, MaxOp{}, lane);
            float e[16];
            const float l2t = p.inv_tau * kLog2eF;
#pragma unroll
            for (int q = 0; q < 16; ++q)
              e[q] = ex2_approx((z[q] - __shfl_sync(0xFFFFFFFFu, mk, 2 * q)) * l2t);
            const float sk = warp_reduce_scatter16(e, SumOp{}, lane);
            if (!(lane & 1) && kr < nr)
              p.seg_stats[(int64_t)(erow0 + kr) * p.nseg + ((tile * p.pitch) >> 5) + quad] =
                  make_float2(mk, sk);
          }
          return true;
        }
      }
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        const int r = min(erow0 + q, p.R - 1);
        if constexpr (EPI == EPI_FUSED) {
          // quantize the cloud's clipped partial (Eq. 18) exactly as the
          // quantize kernel does, emit the code, and dequantize it (Eq. 13)
          const RowQuant rq = s_rq[r];
          const int code = quantize_one(pay_f[q], rq.k, rq.inv);
          if (vj && erow0 + q < p.R) p.codes_out[(int64_t)r * p.n + j] = (int8_t)code;
          z[q] = z[q] + (float)code * rq.s;
        } else {
          z[q] = z[q] + (float)pay_c[q] * s_rq[r].s;
        }
        if (!vj || erow0 + q >= p.R) z[q] = -INFINITY;
        else if (p.Z) p.Z[(int64_t)r * p.ldz + j] = z[q];
      }
      load_payload(tile + (int)gridDim.x);
      if (p.seg_stats) {
        const float mk = warp_reduce_scatter16(z, MaxOp{}, lane);
        float e[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) {
          const float mq = __shfl_sync(0xFFFFFFFFu, mk, 2 * q);
          e[q] = z[q] > -INFINITY ? ex2_approx((z[q] - mq) * (p.inv_tau * kLog2eF)) : 0.f;
        }
        const float sk = warp_reduce_scatter16(e, SumOp{}, lane);
        if (!(lane & 1) && erow0 + kr < p.R && tile * p.pitch + quad * 32 < p.n)
          p.seg_stats[(int64_t)(erow0 + kr) * p.nseg + ((tile * p.pitch) >> 5) + quad] =
              make_float2(mk, sk);
      }
      return true;
    };

    // Position i: the stage's copies go out.  A tile's epilogue runs lag
    // positions after its last stage, when its MMAs are nearly done and the
    // next tiles' copies are on their way.
    const int lag = p.lag;
    int qkb = 0, qx = 0, qtile = blockIdx.x;
    for (int i = 0; i < total + lag; ++i) {
      if (i >= ahead && i < total) {
        // (position i reuses the stage of position i - S)
        if (i >= S && !warp_wait(&s_empty[lstage], lphase ^ 1)) break;
        copy_a();
      }
      if (i >= lag && ++qkb == KB) {
        qkb = 0;
        if (!epilogue(qx, qtile)) break;
        ++qx;
        qtile += gridDim.x;
      }
    }
    cp_wait_all();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  if (warp == kWorkWarps) {
    __syncwarp();
    ptx::tmem_dealloc(tmem, kCols);
  }
}

template <int NR, int EPI>
cudaError_t launch_inst(const FewParams& p, const FewPlan& pl, cudaStream_t st) {
  auto kern = few_kernel<NR, EPI>;
  static std::atomic<bool> opted[kMaxDevices];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const bool cacheable = dev >= 0 && dev < kMaxDevices;
  if (!cacheable || !opted[dev].load()) {
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(kSmemBudget + 1024));
    if (e != cudaSuccess) return e;
    if (cacheable) opted[dev].store(true);
  }
  return launch_pdl(kern, dim3(pl.grid), dim3(kThreads), pl.smem_bytes, st, p);
}

int rows_padded(int rows) { return rows <= 16 ? 16 : 32; }

}  // namespace

FewPlan few_plan(int rows, int n, int K, int sm_count) {
  FewPlan pl{};
  if (rows < 1 || rows > kFewMaxRows || n < 1 || K < 1) return pl;
  pl.na = K > kAtomCols ? 2 : 1;
  pl.KB = (K + pl.na * kAtomCols - 1) / (pl.na * kAtomCols);
  const size_t hidden = (size_t)pl.KB * pl.na * 2 * rows_padded(rows) * 128;
  if (hidden > kMaxHidden) return pl;
  // the fewest turns per SM of at most 128 ids, and then the shortest tile
  // (whole 32-id segments) that needs no more
  const auto turns = [&](int pitch) {
    const long long tiles = ((long long)n + pitch - 1) / pitch;
    return (tiles + sm_count - 1) / sm_count;
  };
  pl.pitch = kTileIds;
  while (pl.pitch > 32 && turns(pl.pitch - 32) == turns(kTileIds)) pl.pitch -= 32;
  pl.tiles = (n + pl.pitch - 1) / pl.pitch;
  pl.grid = pl.tiles < sm_count ? pl.tiles : sm_count;
  const size_t stage = (size_t)pl.na * pl.pitch * 128;
  // (an MMA reads 128 weight rows, past the last stage too)
  const size_t tail = (size_t)kTileIds * 128;
  pl.stages = (int)((kSmemBudget - hidden - tail) / stage);
  if (pl.stages > kMaxStages) pl.stages = kMaxStages;
  pl.lag = pl.stages - 1 < 4 ? pl.stages - 1 : 4;
  pl.smem_bytes = 1024 + hidden + pl.stages * stage + tail;
  pl.nseg = (n + 31) / 32;
  pl.ok = pl.stages >= 2;
  return pl;
}

bool few_operands(const GatherGemm& g) {
  return g.epilogue != EPI_CLOUD && g.w_dtype == W_BF16 &&
         (reinterpret_cast<uintptr_t>(g.W) & 15) == 0 && g.ld_w % 8 == 0;
}

cudaError_t launch_few(const GatherGemm& g, const FewPlan& pl, float2* seg_stats,
                       long long spin_limit, cudaStream_t st) {
  if (!pl.ok || !few_operands(g) || g.rows > kFewMaxRows || !g.status)
    return cudaErrorNotSupported;
  FewParams p{};
  p.h = g.h; p.ld_h = g.ld_h; p.R = g.rows; p.K = g.K; p.n = g.n;
  p.W = static_cast<const uint16_t*>(g.W); p.ld_w = g.ld_w; p.ids = g.ids;
  p.pitch = pl.pitch; p.na = pl.na; p.KB = pl.KB; p.tiles = pl.tiles;
  p.stages = pl.stages; p.lag = pl.lag;
  p.early = g.after_own;
  p.h16 = (reinterpret_cast<uintptr_t>(g.h) & 15) == 0 && g.ld_h % 4 == 0;
  p.Z = g.Y; p.ldz = g.ldy ? g.ldy : g.n;
  p.codes = g.codes; p.row_scale = g.row_scale; p.inv_tau = g.inv_tau;
  p.seg_stats = g.no_stats ? nullptr : seg_stats; p.nseg = pl.nseg;
  p.yc = g.yc; p.rowmax_in = g.rowmax_in; p.codes_out = g.codes_out; p.scale_out = g.scale_out;
  p.status = g.status; p.spin_limit = spin_limit;
  const bool r16 = rows_padded(g.rows) == 16;
  if (g.epilogue == EPI_FUSED) {
    if (!g.yc || !g.rowmax_in || !g.codes_out || !g.scale_out) return cudaErrorInvalidValue;
    return r16 ? launch_inst<16, EPI_FUSED>(p, pl, st) : launch_inst<32, EPI_FUSED>(p, pl, st);
  }
  return r16 ? launch_inst<16, EPI_ENDPOINT>(p, pl, st) : launch_inst<32, EPI_ENDPOINT>(p, pl, st);
}

}  // namespace sph

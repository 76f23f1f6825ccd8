// dC and C^L of every (sample pair, tau point) of a chunk, with the operands of
// the chain's later stages as the only outputs.
//
// The chain at N = 200 is bound by what its stages move through memory.  As two
// separate products, dC and C^L went out in fp32 and in bf16, and a fold read
// the fp32 copies back to form (C^L + dC)^T and dC^T.  Here both accumulators of
// a tile stand in tensor memory together, so the sum is formed in fp32 registers
// and every later operand is written once, in its final type and order.
//
// Persistent: one CTA per SM walks the 128 x 128 output tiles of all pairs and
// tau points, the tau points of a pair next to each other so that its R', R'^S
// and R'^L are read from HBM once.  Per CTA, as in tc_group.cu:
//   warp 0 lane 0  TMA producer: the K slabs (128 bytes per row, 128-byte
//                  swizzle) of three segments, P_S R', P_L R'^S, P_L R'^L;
//   warp 1 lane 0  MMA issuer: the first two segments into accumulator 0, the
//                  third into accumulator 1, of one of two accumulator pairs
//                  (2 x 2 x 128 columns of tensor memory);
//   warps 2-5      epilogue: CW columns of both accumulators at a time, rounded
//                  to the operand type and staged as dense boxes (rows i for
//                  dC and C^L, transposed for the others; swizzled, so that
//                  neither the writes nor the copies conflict on banks), each
//                  written by one TMA bulk store.
// Sums run over K in the same order as in tc_group_kernel, bit for bit.  At N =
// 200, 300 pairs, 64 tau points a bf16 sampling call took 15.5 ms with this and
// the fold that only needs the traces, 22.4 ms with the two products and the
// fold that rewrote their fp32 results.
// Every mbarrier wait is bounded, as there.
#include <algorithm>
#include <cstring>
#include <mutex>

#include "tc_dual.cuh"
#include "tc_ptx.cuh"

namespace rssri {
namespace {

using namespace tcx;

constexpr int DTHREADS = 192, DBN = 128, DSTAGES = 4;
constexpr int ACC = 128;          // columns per accumulator
constexpr int BOX = 2048;         // bytes of a staged box: 32 rows x 64 bytes, or 16 x 128
constexpr int NOUT = 5;           // dC, C^L, C^T, dC^T, (C^L)^T
constexpr int STG = NOUT * BOX;   // one warp's boxes of one chunk of columns
constexpr size_t DSMEM = 1024 + (size_t)DSTAGES * 2 * A_STAGE + 1024 + 4 * 2 * STG;

struct DParams {
  CUtensorMap ta, tb, tdcl, tct, tdct, tclt;
  int n, ns, c, mtiles, ntiles, tiles, wait_polls, has_clt;
  int *err;
};

struct DTile {
  int x, j, m0, n0;
};
__device__ __forceinline__ DTile dtile(const DParams &p, int q) {
  DTile t;
  t.n0 = q % p.ntiles * DBN;
  q /= p.ntiles;
  t.m0 = q % p.mtiles * TBM;
  q /= p.mtiles;
  t.j = q % p.c;
  t.x = q / p.c;
  return t;
}

// A box of 32 rows (i = lane) x CW columns with 64-byte rows, 64-byte swizzle.
template <int KIND>
__device__ __forceinline__ void stage_rows(uint8_t *box, int lane, const float *v) {
  const int sw = (lane >> 1) & 3;
#pragma unroll
  for (int ch = 0; ch < 4; ++ch) {
    uint4 q;
    if (KIND == TC_BF16) {
      uint32_t w[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(v[8 * ch + 2 * u], v[8 * ch + 2 * u + 1]);
        w[u] = *reinterpret_cast<const uint32_t *>(&h);
      }
      q = make_uint4(w[0], w[1], w[2], w[3]);
    } else {
      q = make_uint4(__float_as_uint(round_tf32(v[4 * ch])),
                     __float_as_uint(round_tf32(v[4 * ch + 1])),
                     __float_as_uint(round_tf32(v[4 * ch + 2])),
                     __float_as_uint(round_tf32(v[4 * ch + 3])));
    }
    *reinterpret_cast<uint4 *>(box + lane * 64 + 16 * (ch ^ sw)) = q;
  }
}
// The transposed box: CW rows (columns j of the tile) x 32 columns (i = lane): 64-byte
// rows for bf16, 128-byte rows (128-byte swizzle) for tf32.
template <int KIND>
__device__ __forceinline__ void stage_cols(uint8_t *box, int lane, const float *v) {
  if (KIND == TC_BF16) {
#pragma unroll
    for (int j = 0; j < 32; ++j)
      *reinterpret_cast<__nv_bfloat16 *>(box + j * 64 + 16 * ((lane >> 3) ^ ((j >> 1) & 3)) +
                                         2 * (lane & 7)) = __float2bfloat16_rn(v[j]);
  } else {
#pragma unroll
    for (int j = 0; j < 16; ++j)
      *reinterpret_cast<float *>(box + j * 128 + 16 * ((lane >> 2) ^ (j & 7)) + 4 * (lane & 3)) =
          round_tf32(v[j]);
  }
}

template <int CW> __device__ __forceinline__ void tmem_cols(uint32_t addr, float *v) {
#pragma unroll
  for (int h = 0; h < CW; h += 16) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,"
        "%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
          "=r"(r[14]), "=r"(r[15])
        : "r"(addr + h));
#pragma unroll
    for (int u = 0; u < 16; ++u) v[h + u] = __uint_as_float(r[u]);
  }
}

__device__ __forceinline__ void commit_to(uint64_t *bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(s_u32(bar))
      : "memory");
}

template <int KIND>
__global__ void __launch_bounds__(DTHREADS, 1) tc_dual_kernel(const __grid_constant__ DParams p) {
  constexpr int TBK = KindT<KIND>::TBK, KMMA = KindT<KIND>::KMMA;
  constexpr int CW = KIND == TC_BF16 ? 32 : 16;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t *sA = smem, *sB = smem + DSTAGES * A_STAGE;
  uint64_t *full = (uint64_t *)(sB + DSTAGES * A_STAGE);
  uint64_t *empty = full + DSTAGES;
  uint64_t *accf = empty + DSTAGES;  // [2] accumulator pair complete
  uint64_t *acce = accf + 2;         // [2] accumulator pair drained
  uint64_t *done = acce + 2;
  uint32_t *tslot = (uint32_t *)(done + 1);
  uint8_t *stg = sB + DSTAGES * A_STAGE + 1024;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < DSTAGES; ++s) {
      bar_init(&full[s], 1);
      bar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      bar_init(&accf[b], 1);
      bar_init(&acce[b], 4);
    }
    bar_init(done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     s_u32(tslot)),
                 "r"(4 * ACC));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = *tslot;

  if (warp == 0) {
    if (lane == 0) {
      bool ok = test_mode_gate(p.wait_polls, p.err);
      int it = 0;
      for (int q = blockIdx.x; q < p.tiles && ok; q += gridDim.x) {
        const DTile t = dtile(p, q);
        for (int sg = 0; sg < 3 && ok; ++sg) {
          const int az = t.j * 2 * p.ns + (sg ? p.ns : 0) + t.x, bz = sg * p.ns + t.x;
          for (int k0 = 0; k0 < p.n; k0 += TBK, ++it) {
            const int st = it % DSTAGES;
            if (it >= DSTAGES &&
                !bar_wait(&empty[st], ((it / DSTAGES) - 1) & 1, p.err, 1, p.wait_polls)) {
              ok = false;
              break;
            }
            bar_expect(&full[st], 2 * A_STAGE);
            tma_load3(sA + st * A_STAGE, &p.ta, &full[st], k0, t.m0, az);
            tma_load3(sB + st * A_STAGE, &p.tb, &full[st], k0, t.n0, bz);
          }
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      bool ok = true;
      int it = 0, lt = 0;
      for (int q = blockIdx.x; q < p.tiles && ok; q += gridDim.x, ++lt) {
        const DTile t = dtile(p, q);
        const int buf = lt & 1;
        if (lt >= 2) {
          if (!bar_wait(&acce[buf], ((lt >> 1) - 1) & 1, p.err, 2, p.wait_polls)) {
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;");
        }
        // the columns of the tile that exist, rounded up to 16
        const uint32_t idesc = instr_desc<KIND>(min(DBN, (p.n - t.n0 + 15) & ~15));
        for (int sg = 0; sg < 3 && ok; ++sg) {
          const uint32_t acc_addr = tmem + (uint32_t)(buf * 2 * ACC + (sg == 2 ? ACC : 0));
          for (int k0 = 0; k0 < p.n; k0 += TBK, ++it) {
            const int st = it % DSTAGES;
            if (!bar_wait(&full[st], (it / DSTAGES) & 1, p.err, 3, p.wait_polls)) {
              ok = false;
              break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;");
            const uint64_t da = smem_desc(s_u32(sA + st * A_STAGE));
            const uint64_t db = smem_desc(s_u32(sB + st * A_STAGE));
            const int nk = min(TBK / KMMA, (p.n - k0 + KMMA - 1) / KMMA);
            for (int kk = 0; kk < nk; ++kk) {
              const uint32_t acc = (sg != 1 && k0 == 0 && kk == 0) ? 0u : 1u;
              if (KIND == TC_BF16)
                asm volatile(
                    "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %4, 0;\n\t"
                    "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, q;\n}" ::"r"(acc_addr),
                    "l"(da + 2 * kk), "l"(db + 2 * kk), "r"(idesc), "r"(acc));
              else
                asm volatile(
                    "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %4, 0;\n\t"
                    "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, q;\n}" ::"r"(acc_addr),
                    "l"(da + 2 * kk), "l"(db + 2 * kk), "r"(idesc), "r"(acc));
            }
            commit_to(&empty[st]);
          }
        }
        if (ok) commit_to(&accf[buf]);
      }
      commit_to(done);  // arrives once every product issued above has completed
    }
  } else {
    const int lq = warp & 3;
    uint8_t *wst = stg + (warp - 2) * 2 * STG;
    bool ok = true;
    int lt = 0, sc = 0;
    for (int q = blockIdx.x; q < p.tiles && ok; q += gridDim.x, ++lt) {
      const DTile t = dtile(p, q);
      const int buf = lt & 1;
      if (!bar_wait(&accf[buf], (lt >> 1) & 1, p.err, 4, p.wait_polls)) {
        ok = false;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;");
      const int row0 = t.m0 + lq * 32;
      const int cend = min(DBN, p.n - t.n0);
      const uint32_t ta = tmem + ((uint32_t)(lq * 32) << 16) + (uint32_t)(buf * 2 * ACC);
      // the next columns are read from tensor memory while these are staged
      float d0[CW], l0[CW], d1[CW], l1[CW];
      auto fetch = [&](int c0, float *d, float *l) {
        tmem_cols<CW>(ta + c0, d);
        tmem_cols<CW>(ta + ACC + c0, l);
      };
      auto step = [&](int c0, float *d, float *l) {
        uint8_t *b = wst + (sc & 1) * STG;
        if (sc >= 2) {
          if (lane == 0) bulk_wait_read1();  // the boxes two steps back have been read
          __syncwarp();
        }
        stage_rows<KIND>(b, lane, d);
        stage_rows<KIND>(b + BOX, lane, l);
        stage_cols<KIND>(b + 3 * BOX, lane, d);
        if (p.has_clt) stage_cols<KIND>(b + 4 * BOX, lane, l);
#pragma unroll
        for (int u = 0; u < CW; ++u) l[u] = l[u] + d[u];
        stage_cols<KIND>(b + 2 * BOX, lane, l);
        fence_async_smem();
        __syncwarp();
        if (lane == 0) {
          const int z2 = t.j * 2 * p.ns + t.x, z1 = t.j * p.ns + t.x;
          tma_store3(&p.tdcl, b, t.n0 + c0, row0, z2);
          tma_store3(&p.tdcl, b + BOX, t.n0 + c0, row0, z2 + p.ns);
          tma_store3(&p.tct, b + 2 * BOX, row0, t.n0 + c0, z1);
          tma_store3(&p.tdct, b + 3 * BOX, row0, t.n0 + c0, z1);
          if (p.has_clt) tma_store3(&p.tclt, b + 4 * BOX, row0, t.n0 + c0, z1);
          bulk_commit();
        }
        ++sc;
      };
      if (row0 < p.n) {
        fetch(0, d0, l0);
        for (int c0 = 0; c0 < cend; c0 += 2 * CW) {
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          if (c0 + CW < cend) fetch(c0 + CW, d1, l1);
          step(c0, d0, l0);
          if (c0 + CW >= cend) break;
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          if (c0 + 2 * CW < cend) fetch(c0 + 2 * CW, d0, l0);
          step(c0 + CW, d1, l1);
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;");
      __syncwarp();
      if (lane == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(s_u32(&acce[buf])) : "memory");
    }
    if (lane == 0) bulk_wait_all();
    __syncwarp();
    bar_wait(done, 0, p.err, 5, p.wait_polls);
    asm volatile("tcgen05.fence::after_thread_sync;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(4 * ACC));
}

}  // namespace

cudaError_t tc_dual_prepare() {
  static std::mutex mu;
  static bool done[64] = {};
  int dev = 0;
  RS_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(mu);
  if (!done[dev]) {
    RS_TRY(cudaFuncSetAttribute(tc_dual_kernel<TC_BF16>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DSMEM));
    RS_TRY(cudaFuncSetAttribute(tc_dual_kernel<TC_TF32>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DSMEM));
    done[dev] = true;
  }
  return cudaSuccess;
}

cudaError_t tc_dual(int kind, const TcDual &g, cudaStream_t s) {
  if (!tc_available()) return cudaErrorNotSupported;
  if ((kind != TC_BF16 && kind != TC_TF32) || g.n <= 0 || g.ns <= 0 || g.c <= 0)
    return cudaErrorInvalidValue;
  const int es = kind == TC_BF16 ? 2 : 4;
  const long long mat = (long long)g.n * g.ld;
  DParams p;
  std::memset(&p, 0, sizeof(p));
  TcOperand a, b;
  a.ptr = g.P; a.ld = g.ld; a.sb = mat; a.rows = g.n;
  b.ptr = g.y3; b.ld = g.ld; b.sb = mat; b.rows = g.n;
  RS_TRY(tc_make_map(&p.ta, kind, a, g.n, g.c * 2 * g.ns, TBM));
  RS_TRY(tc_make_map(&p.tb, kind, b, g.n, 3 * g.ns, DBN));
  // boxes: 64-byte rows of CW columns x 32 rows; transposed, 32 columns x CW rows
  const int cw = 64 / es;
  RS_TRY(tc_make_box_map(&p.tdcl, g.dcl, es, g.n, g.n, 2LL * g.c * g.ns, g.ld, cw, 32));
  RS_TRY(tc_make_box_map(&p.tct, g.ct, es, g.n, g.n, (long long)g.c * g.ns, g.ld, 32, cw));
  RS_TRY(tc_make_box_map(&p.tdct, g.dct, es, g.n, g.n, (long long)g.c * g.ns, g.ld, 32, cw));
  p.has_clt = g.clt != nullptr;
  if (g.clt) RS_TRY(tc_make_box_map(&p.tclt, g.clt, es, g.n, g.n, (long long)g.c * g.ns, g.ld, 32, cw));
  p.n = g.n;
  p.ns = g.ns;
  p.c = g.c;
  p.mtiles = ceil_div(g.n, TBM);
  p.ntiles = ceil_div(g.n, DBN);
  const long long tiles = (long long)p.mtiles * p.ntiles * g.ns * g.c;
  if (tiles > (1LL << 30)) return cudaErrorInvalidValue;
  p.tiles = (int)tiles;
  p.wait_polls = g.wait_polls;
  p.err = g.err;
  RS_TRY(tc_dual_prepare());
  int dev = 0, sms = 152;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int grid = (int)std::min<long long>(tiles, sms);
  if (kind == TC_BF16) tc_dual_kernel<TC_BF16><<<grid, DTHREADS, DSMEM, s>>>(p);
  else tc_dual_kernel<TC_TF32><<<grid, DTHREADS, DSMEM, s>>>(p);
  ++launch_counter();
  return cudaGetLastError();
}

}  // namespace rssri

// conv.cu -- 3^3 convolutions of the warm-start network as implicit GEMMs on the 5th-generation tensor
// cores (sm_103a): the forward pass, the input gradient (the same kernel with the flipped, transposed
// weights) and the weight gradient, without im2col rows in memory.
//
// Layouts: activations are channel-last BF16, x[v][c], voxel v = x + W (y + H z).  The input may be given
// as two parts along the channels, the first optionally on the 2x coarser grid (nearest upsampling), which
// is the decoder's concatenation.
//
// What the im2col form spent its time on (one 128^3 training step, 25.5 ms on a GB300): writing and reading
// back columns of 27 C values per voxel (4.3 GB per level-0 convolution at C = 16), and transposed copies for the
// weight gradient.  Here a CTA keeps the voxels of a tile and their one-voxel halo in shared memory, and each
// of the 27 taps is the same shared memory read from another start address:
//   - a plane of the tile is 8 x 16 voxels plus halo, 10 x 18, held as [8-channel chunk][voxel][16 bytes], the
//     unswizzled K-major operand layout: rows (voxels) 16 bytes apart, 8-row groups (voxel rows of the tile)
//     one halo row (160 bytes) apart, channel chunks one plane (2880 bytes) apart.  A tap (dy, dx) moves the
//     start address by dy * 160 + dx * 16 bytes;
//   - the CTA walks along z with a ring of planes, so a plane is loaded once for the three taps dz;
//   - accumulation runs over taps, then channels, 16 at a time: the order of the im2col GEMM, whose
//     results it repeats bit for bit.
// The weight gradient contracts over voxels: its operands are the im2col rows of 64 voxels at a time, put
// together in shared memory, MN-major; see k_wgrad.
// A 128^3 training step of the three-level network takes 6.5 ms with these kernels (weight gradients 4.0 ms, the
// other convolutions 1.8 ms), a prediction at 128 x 64 x 96 0.56 ms (3.8 ms from im2col rows).
//
// Every wait on an mbarrier is bounded; a wait that runs out sets the error word (lbm_nn_status then returns
// LBM_ERR_TIMEOUT) and the kernel still releases its TMEM before it returns.
#include <algorithm>
#include <initializer_list>
#include <type_traits>

#include "../../include/lbm_nn.h"
#include "tc.cuh"

namespace lbmnn {

constexpr int TX = 8, TY = 16;                 // tile: 128 voxels of one z plane
constexpr int HX = TX + 2, HY = TY + 2;        // with halo
constexpr int PV = HX * HY;                    // voxels of a halo plane
constexpr int ROW16 = 16;                      // bytes of one voxel in an 8-channel chunk
constexpr int CHUNK = PV * ROW16;              // bytes of an 8-channel chunk of a plane

struct ConvSrc {
  const bf16* a;   // channels [0, ca), on the coarse grid (W/2, H/2, D/2) if up
  const bf16* b;   // channels [ca, ca + cb)
  int ca, cb, up;
};

// 16 bytes (8 channels from c) of voxel (x, y, z)
__device__ __forceinline__ const bf16* src_at(const ConvSrc& s, int c, int x, int y, int z, int H, int W) {
  if (c < s.ca) {
    if (s.up) return s.a + ((long long)((z >> 1) * (H >> 1) + (y >> 1)) * (W >> 1) + (x >> 1)) * s.ca + c;
    return s.a + ((long long)(z * H + y) * W + x) * s.ca + c;
  }
  return s.b + ((long long)(z * H + y) * W + x) * s.cb + (c - s.ca);
}

// 16-byte asynchronous copy to shared memory, zero-filled when !in
__device__ __forceinline__ void cp16(void* dst, const void* src, bool in) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(saddr(dst)), "l"(src), "r"(in ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }
// makes this thread's shared-memory writes visible to the tensor core's (async) reads
__device__ __forceinline__ void fence_async() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }
__device__ __forceinline__ void mbar_arrive(uint64_t* b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(saddr(b)) : "memory");
}
// bulk copy of contiguous bytes (a multiple of 16) into shared memory, counted on bar
__device__ __forceinline__ void bulk_load(void* dst, const void* src, unsigned bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(saddr(dst)),
               "l"(src), "r"(bytes), "r"(saddr(bar))
               : "memory");
}

// Unswizzled shared-memory descriptor: start address, leading (lbo) and stride (sbo) byte offsets, all in
// 16-byte units; descriptor version 1, layout 0.  K-major: rows 16 bytes apart, 8-row groups sbo, 8-element
// K chunks lbo apart.  MN-major: K rows 16 bytes apart, 8-element MN chunks sbo, 8-row K groups lbo apart.
__device__ __forceinline__ uint64_t desc_plain(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(sbo >> 4) << 32) |
         ((uint64_t)1 << 46);
}

__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(saddr(slot)), "r"(cols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void tmem_free(uint32_t tmem, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(cols) : "memory");
}

// mbar_wait by a whole warp, with one answer for its lanes (tensor-memory loads need them together)
__device__ __forceinline__ bool warp_wait(uint64_t* b, unsigned parity) {
  const bool r = mbar_wait(b, parity);
  return __all_sync(0xffffffffu, r);
}

struct ConvOut {
  bf16* y0;            // columns [0, n0)
  bf16* y1;            // columns [n0, N)
  const float* bias;   // [N] or null
  int n0, relu;
};

// one row (voxel) of the output tile from its TMEM lane; every lane of the warp takes part in the loads
__device__ __forceinline__ void store_row(uint32_t taddr, const ConvOut& o, int N, long long v, bool in) {
#pragma unroll 1
  for (int c = 0; c < N; c += 16) {
    float r[16], b[16];
#pragma unroll
    for (int i = 0; i < 16; i += 4)
      *reinterpret_cast<float4*>(b + i) = o.bias ? __ldg(reinterpret_cast<const float4*>(o.bias + c + i)) : make_float4(0.f, 0.f, 0.f, 0.f);
    tmem_ld16(taddr + (uint32_t)c, r);
    if (!in) continue;
    __align__(16) bf16 w[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      float x = r[i] + b[i];
      if (o.relu) x = fmaxf(x, 0.f);
      w[i] = __float2bfloat16_rn(x);
    }
    bf16* dst = c < o.n0 ? o.y0 + v * o.n0 + c : o.y1 + v * (N - o.n0) + (c - o.n0);
    *reinterpret_cast<uint4*>(dst) = *reinterpret_cast<const uint4*>(w);
    *reinterpret_cast<uint4*>(dst + 8) = *reinterpret_cast<const uint4*>(w + 8);
  }
}

// ------------------------------------------------------------------ forward / input gradient

struct ConvPlan {
  int C, N, nz;        // channels, outputs, z planes per CTA
  int planes;          // ring of halo planes
  int seq;             // 1: three plane loads per output (nz == 1), 0: planes roll along z
  int sc, stages;      // channels and number of the weight stages; stages == 0: all weights resident
  int accs, cols;      // accumulators and TMEM columns
  unsigned smem;
};

// Warps 0-3 load planes (cp.async) and write results, warp 4 issues the MMAs, warp 5 the weight copies.
// Bound by the tensor core's operand reads: an MMA of 128 x N x 16 from unswizzled planes takes 64 cycles at any N up
// to 32, so the 27 taps of 16 channels at 128^3 (16,384 tiles) need 90 us of the 152 us the layer takes (378 us when the
// issuing thread built every descriptor anew).
__global__ void __launch_bounds__(192, 4) k_conv3(const ConvSrc src, const bf16* __restrict__ wp, const ConvOut out,
                                               const ConvPlan p, int D, int H, int W, int* err) {
  extern __shared__ unsigned char raw[];
  unsigned char* base = raw + ((128u - (saddr(raw) & 127u)) & 127u);
  const int C = p.C, N = p.N, P = p.planes;
  const uint32_t plane_bytes = (uint32_t)(C / 8) * CHUNK;
  const uint32_t tap_bytes = (uint32_t)C * N * 2, stage_bytes = (uint32_t)p.sc * N * 2;
  const int nch = p.stages ? C / p.sc : 1;
  unsigned char* sA = base;
  unsigned char* sB = sA + (size_t)P * plane_bytes;
  unsigned char* end = sB + (p.stages ? (size_t)p.stages * stage_bytes : (size_t)27 * tap_bytes);
  uint64_t* fullA = reinterpret_cast<uint64_t*>(end);   // [4]
  uint64_t* emptyA = fullA + 4;
  uint64_t* fullB = emptyA + 4;                         // [8]
  uint64_t* emptyB = fullB + 8;
  uint64_t* done = emptyB + 8;                          // [2]
  uint64_t* accfree = done + 2;
  uint32_t* slot = reinterpret_cast<uint32_t*>(accfree + 2);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // one index for all tiles: any proportions of the domain, where the y and z of a grid end at 65535
  const unsigned tiles_x = (unsigned)(W + TX - 1) / TX, tiles_y = (unsigned)(H + TY - 1) / TY;
  const unsigned row = blockIdx.x / tiles_x;
  const int x0 = (int)(blockIdx.x - row * tiles_x) * TX, y0 = (int)(row % tiles_y) * TY, z0 = (int)(row / tiles_y) * p.nz;
  const int nz = min(p.nz, D - z0);
  if (threadIdx.x == 0) {
    for (int i = 0; i < 4; ++i) {
      mbar_init(&fullA[i], 128);
      mbar_init(&emptyA[i], 1);
    }
    for (int i = 0; i < 8; ++i) {
      mbar_init(&fullB[i], 1);
      mbar_init(&emptyB[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&done[i], 1);
      mbar_init(&accfree[i], 128);
    }
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 0) tmem_alloc(slot, (uint32_t)p.cols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *slot;
  bool ok = true;

  if (warp < 4) {
    const int C8 = C / 8;
    const int v_first = threadIdx.x / C8, c8_first = threadIdx.x % C8, v_step = 128 / C8, c8_step = 128 % C8;
    // plane q of the sequence: z index
    auto plane_z = [&](int q) { return p.seq ? z0 + q / 3 + q % 3 - 1 : z0 - 1 + q; };
    const int nq = p.seq ? 3 * nz : nz + 2;
    auto issue = [&](int q) {
      // item i = v C8 + c8 of the plane, 128 apart: v and c8 advance by fixed steps
      const int z = plane_z(q);
      unsigned char* dst = sA + (size_t)(q % P) * plane_bytes;
      const bool zin = z >= 0 && z < D;
      int v = v_first, c8 = c8_first;
#pragma unroll 4
      for (; v < PV;) {
        const int vy = v / HX, xx = x0 - 1 + v - vy * HX, yy = y0 - 1 + vy;
        const bool in = zin && (unsigned)xx < (unsigned)W && (unsigned)yy < (unsigned)H;
        cp16(dst + c8 * CHUNK + v * ROW16, in ? src_at(src, c8 * 8, xx, yy, z, H, W) : src.a, in);
        c8 += c8_step;
        v += v_step;
        if (c8 >= C8) {
          c8 -= C8;
          ++v;
        }
      }
      cp_commit();
    };
    auto publish = [&](int q) { mbar_arrive(&fullA[q % P]); };
    int q = 0;
    for (; q < nq && q < P; ++q) issue(q);
    cp_wait_all();
    fence_async();
    for (int i = 0; i < q; ++i) publish(i);
    if (p.seq)
      for (; q < nq && ok; ++q) {
        if (!warp_wait(&emptyA[q % P], (unsigned)(q / P - 1) & 1u)) ok = false;
        issue(q);
        cp_wait_all();
        fence_async();
        publish(q);
      }
    const int m = threadIdx.x;
    const int xx = x0 + m % TX, yy = y0 + m / TX;
    for (int t = 0; t < nz && ok; ++t) {
      const int ac = t % p.accs;
      if (!warp_wait(&done[ac], (unsigned)(t / p.accs) & 1u)) ok = false;
      tc_fence_after();
      const bool more = !p.seq && q < nq;   // the first plane of output t is free: refill its slot
      if (more) issue(q);
      store_row(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(ac * N), out, N,
                ((long long)(z0 + t) * H + yy) * W + xx, ok && xx < W && yy < H);
      tc_fence_before();
      mbar_arrive(&accfree[ac]);
      if (more) {
        cp_wait_all();
        fence_async();
        publish(q);
        ++q;
      }
    }
  } else if (warp == 4) {
    if (lane == 0) {
      // one thread issues 27 C / 16 MMAs per output, so the loop is kept to a few instructions each: descriptors
      // differ in their start address only, in 16-byte units
      const uint32_t idesc = idesc_bf16(128, N);
      const uint64_t a_desc = desc_plain(saddr(sA), CHUNK, HX * ROW16), b_desc = desc_plain(saddr(sB), (uint32_t)N * 16, 128);
      const uint32_t a_step = 2 * CHUNK / 16, b_step = 2 * (uint32_t)N, plane16 = plane_bytes / 16, stage16 = stage_bytes / 16;
      const int n16 = (p.stages ? p.sc : C) / 16;
      int st = 0;              // weight stage and the parity of its current fill
      unsigned st_ph = 0;
      if (!p.stages && !mbar_wait(&fullB[0], 0)) ok = false;
      for (int t = 0; t < nz && ok; ++t) {
        const int ac = t % p.accs;
        if (t >= p.accs && !mbar_wait(&accfree[ac], (unsigned)(t / p.accs - 1) & 1u)) ok = false;
        tc_fence_after();
        const uint32_t d = tmem + (uint32_t)(ac * N);
        uint32_t acc = 0;
        uint64_t bd = b_desc;
#pragma unroll 1
        for (int dz = 0; dz < 3 && ok; ++dz) {
          const int q = p.seq ? 3 * t + dz : t + dz;
          if ((p.seq || t == 0 || dz == 2) && !mbar_wait(&fullA[q % P], (unsigned)(q / P) & 1u)) {
            ok = false;
            break;
          }
          uint64_t ad = a_desc + (uint64_t)((uint32_t)(q % P) * plane16);
#pragma unroll 1
          for (int dy = 0; dy < 3 && ok; ++dy, ad += HX) {
#pragma unroll
            for (int dx = 0; dx < 3; ++dx) {
              uint64_t a = ad + dx;
              if (!p.stages) {
#pragma unroll 2
                for (int kk = 0; kk < n16; ++kk, a += a_step, bd += b_step) {
                  mma_bf16(d, a, bd, idesc, acc);
                  acc = 1;
                }
              } else {
                for (int ch = 0; ch < nch && ok; ++ch) {
                  if (!mbar_wait(&fullB[st], st_ph)) ok = false;
                  bd = b_desc + (uint64_t)((uint32_t)st * stage16);
#pragma unroll 2
                  for (int kk = 0; kk < n16; ++kk, a += a_step, bd += b_step) {
                    mma_bf16(d, a, bd, idesc, acc);
                    acc = 1;
                  }
                  mma_commit(&emptyB[st]);
                  if (++st == p.stages) {
                    st = 0;
                    st_ph ^= 1u;
                  }
                }
              }
            }
          }
          if (p.seq) mma_commit(&emptyA[q % P]);
        }
        mma_commit(&done[ac]);
      }
    }
  } else if (lane == 0) {
    if (!p.stages) {
      mbar_expect_tx(&fullB[0], 27 * tap_bytes);
      // one request per tap, so that no single copy is very long
      for (int t = 0; t < 27; ++t) bulk_load(sB + (size_t)t * tap_bytes, wp + (size_t)t * C * N, tap_bytes, &fullB[0]);
      if (!mbar_wait(&fullB[0], 0)) ok = false;   // nothing of this CTA is in flight when it returns
    } else {
      const int total = nz * 27 * nch, per = 27 * nch;
      int b = 0;
      for (; b < total; ++b) {
        const int st = b % p.stages;
        if (b >= p.stages && !mbar_wait(&emptyB[st], (unsigned)(b / p.stages - 1) & 1u)) {
          ok = false;
          break;
        }
        mbar_expect_tx(&fullB[st], stage_bytes);
        bulk_load(sB + (size_t)st * stage_bytes, wp + (size_t)(b % per) * p.sc * N, stage_bytes, &fullB[st]);
      }
      for (int i = max(0, b - p.stages); i < b; ++i)
        if (!mbar_wait(&fullB[i % p.stages], (unsigned)(i / p.stages) & 1u)) ok = false;
    }
  }
  if (!ok) atomicOr(err, 1);
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_free(tmem, (uint32_t)p.cols);
}

// The first layer: C <= 8 channels in rows of 8 (lbm_nn_pad8).  K runs over tap * C + c as in the im2col GEMM (in 16s
// across taps), so a row of the operand is put together from the 27 neighbours' 16-byte rows in registers: chunk q
// holds the values k = 8 q .. 8 q + 7, all positions known at compile time.
template <int C>
struct FirstRow {
  static constexpr int K16 = (27 * C + 15) / 16, CHUNKS = 2 * K16, USED = (27 * C + 7) / 8;
  uint4 t[27];
  __device__ __forceinline__ void load(const bf16* __restrict__ x8, long long v, int x, int y, int z, int D, int H, int W, bool in) {
#pragma unroll
    for (int i = 0; i < 27; ++i) {
      const int dz = i / 9 - 1, dy = (i / 3) % 3 - 1, dx = i % 3 - 1;
      const bool ok = in && (unsigned)(x + dx) < (unsigned)W && (unsigned)(y + dy) < (unsigned)H && (unsigned)(z + dz) < (unsigned)D;
      t[i] = ok ? __ldg(reinterpret_cast<const uint4*>(x8 + (v + (long long)(dz * H + dy) * W + dx) * 8)) : make_uint4(0u, 0u, 0u, 0u);
    }
  }
  __device__ __forceinline__ uint32_t half_at(int k) const {   // 16-bit value k
    if (k >= 27 * C) return 0u;
    const int tap = k / C, c = k % C;
    const uint32_t w = c / 2 == 0 ? t[tap].x : (c / 2 == 1 ? t[tap].y : (c / 2 == 2 ? t[tap].z : t[tap].w));
    return c % 2 ? w >> 16 : w & 0xffffu;
  }
  __device__ __forceinline__ uint4 chunk(int q) const {
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) w[i] = half_at(8 * q + 2 * i) | half_at(8 * q + 2 * i + 1) << 16;
    return make_uint4(w[0], w[1], w[2], w[3]);
  }
};

// x [V][C] -> x8 [V][8], zero padded
__global__ void __launch_bounds__(256) k_pad8(const bf16* __restrict__ x, bf16* __restrict__ x8, long long V, int C) {
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < V; v += (long long)gridDim.x * blockDim.x) {
    __align__(16) bf16 w[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) w[c] = c < C ? x[v * C + c] : __float2bfloat16_rn(0.f);
    *reinterpret_cast<uint4*>(x8 + v * 8) = *reinterpret_cast<const uint4*>(w);
  }
}

// Tiles of 128 consecutive voxels, one thread per voxel; the CTAs of an SM hide one another's phases.  Bound by the
// 27 row loads per voxel, L1 hits mostly: 82 us at 128^3 with 5 channels (311 us with the input's unpadded rows).
template <int C>
__global__ void __launch_bounds__(128, 3) k_conv3_first(const bf16* __restrict__ x8, const bf16* __restrict__ wp, const ConvOut out,
                                                        int N, int D, int H, int W, int cols, int* err) {
  using F = FirstRow<C>;
  extern __shared__ unsigned char raw[];
  unsigned char* base = raw + ((128u - (saddr(raw) & 127u)) & 127u);
  unsigned char* sA = base;                                        // [CHUNKS][128 rows][16 bytes]
  unsigned char* sB = sA + F::CHUNKS * 2048;                       // [K16][2][N][16 bytes]
  __shared__ uint64_t full, done;
  __shared__ uint32_t slot;
  const int warp = threadIdx.x >> 5;
  const long long V = (long long)D * H * W;
  if (threadIdx.x == 0) {
    mbar_init(&full, 1);
    mbar_init(&done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    mbar_expect_tx(&full, (unsigned)(F::K16 * N * 32));
    bulk_load(sB, wp, (unsigned)(F::K16 * N * 32), &full);
  }
  if (warp == 0) tmem_alloc(&slot, (uint32_t)cols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = slot;
  bool ok = warp_wait(&full, 0);
  unsigned ph = 0;
  for (long long v0 = (long long)blockIdx.x * 128; v0 < V; v0 += (long long)gridDim.x * 128, ph ^= 1u) {
    const long long v = v0 + threadIdx.x;
    {
      F row;
      const int r = (int)(v / W);
      row.load(x8, v, (int)(v - (long long)r * W), r % H, r / H, D, H, W, v < V);
#pragma unroll
      for (int q = 0; q < F::CHUNKS; ++q) *reinterpret_cast<uint4*>(sA + q * 2048 + threadIdx.x * 16) = row.chunk(q);
    }
    fence_async();
    __syncthreads();
    if (threadIdx.x == 0 && ok) {
      const uint32_t idesc = idesc_bf16(128, N);
      const uint64_t ad = desc_plain(saddr(sA), 2048, 128), bd = desc_plain(saddr(sB), (uint32_t)N * 16, 128);
      for (int kk = 0; kk < F::K16; ++kk) mma_bf16(tmem, ad + kk * 256, bd + (uint64_t)(kk * 2 * N), idesc, kk > 0 ? 1u : 0u);
      mma_commit(&done);
    }
    if (ok && !warp_wait(&done, ph)) ok = false;
    tc_fence_after();
    store_row(tmem + ((uint32_t)(warp * 32) << 16), out, N, v, ok && v < V);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
  }
  if (!ok) atomicOr(err, 1);
  __syncwarp();
  __syncthreads();
  if (warp == 0) tmem_free(tmem, (uint32_t)cols);
}

// ------------------------------------------------------------------ weight gradient

// dW[k][o] = sum_v col[v][k] dy[v][o], k = tap C + c: a GEMM over voxels, in blocks of 64, with the 128 x 64 tiles of
// the transposed im2col gathered straight from x into shared memory (16-byte copies, 8 channels of one voxel and
// tap each).  Both operands are MN-major: [k / 8][64 voxels][8] and [o / 8][64 voxels][8], 8-element MN chunks 1 KB
// and 8-voxel K groups 128 bytes apart.  A CTA owns some of the 128-row tiles and one of the voxel ranges that the
// split-K GEMM over im2col rows would take, adds the voxels in the same order, and writes FP32 partial sums
// that k_wgrad_sum adds in split order: the same result bit for bit.
// Bound by the gather, not by a bandwidth: a 16 KB tile per 0.6 us and SM is 13 bytes per clock, and no order of the
// tiles changed it.  A tile is 32 copy instructions of a warp, each of sixteen 32-byte pieces from different rows with
// their tap's test and address, with the copies of WLAG tiles in flight behind the one being issued (128^3: 48 -> 16
// channels 1514 us, 16 -> 16 channels 621 us, the 5-channel input 534 us, from 3597 us with unpadded rows).
struct WgradPlan {
  int C, Co;
  int tiles, tj, jobs;       // 128-row tiles of k, tiles per CTA, CTAs along k
  int nkb, kbs, splits;      // 64-voxel blocks, blocks per split, splits
  int ws, nb, cols;          // im2col tiles in the ring, dy buffers, TMEM columns
  unsigned smem;
};
constexpr int WSTAGES = 6;                 // ring of 16 KB im2col tiles, fewer (more than WLAG) for wide layers
constexpr int WLAG = 3;                    // tiles whose copies are in flight behind the one being issued
constexpr int WBLOCK = 64 * 16;            // bytes of an 8-row chunk of 64 voxels

__device__ __forceinline__ void cp16_ca(void* dst, const void* src, bool in) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;\n" ::"r"(saddr(dst)), "l"(src), "r"(in ? 16 : 0) : "memory");
}

template <int FIRST>   // 0: channels in 16s; else the narrow input of FIRST channels in rows of 8
__global__ void __launch_bounds__(288, FIRST ? 1 : 2) k_wgrad(const ConvSrc src, const bf16* __restrict__ dy, float* __restrict__ part,
                                               const WgradPlan p, int D, int H, int W, int* err) {
  extern __shared__ unsigned char raw[];
  unsigned char* base = raw + ((128u - (saddr(raw) & 127u)) & 127u);
  __shared__ uint64_t full[WSTAGES], empty[WSTAGES], done;
  __shared__ uint32_t slot;
  unsigned char* sA = base;
  unsigned char* sB = base + (size_t)p.ws * 16 * WBLOCK;
  const uint32_t bbytes = (uint32_t)(p.Co / 8) * WBLOCK;
  // per pair of 8-row chunks (16 channels of a tap): tap, part of the input (0 a, 1 a on the coarse grid, 2 b, -1 past
  // 27 C), element offset from the voxel's own row (channel alone on the coarse grid) in 64 bits: a plane of H W C
  // elements may pass 2^31
  int4* table = reinterpret_cast<int4*>(sB + (size_t)p.nb * bbytes);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int C = p.C, Co = p.Co, ws = p.ws;
  const int t0 = blockIdx.y * p.tj, nt = min(p.tj, p.tiles - t0);
  const int kb0 = blockIdx.x * p.kbs, kb1 = min(p.nkb, kb0 + p.kbs);
  if (threadIdx.x == 0) {
    for (int i = 0; i < WSTAGES; ++i) {
      mbar_init(&full[i], 256);
      mbar_init(&empty[i], 1);
    }
    mbar_init(&done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  for (int i = threadIdx.x; i < 8 * nt; i += 288) {
    const int k = (t0 * 8 + i) * 16, tap = k / C, c = k % C;
    const long long shift = ((long long)(tap / 9 - 1) * H + (tap / 3) % 3 - 1) * W + tap % 3 - 1;
    const int part = k >= 27 * C ? -1 : c >= src.ca ? 2 : src.up ? 1 : 0;
    const long long off = part == 2 ? shift * src.cb + c - src.ca : part == 1 ? c : shift * src.ca + c;
    table[i] = make_int4(part < 0 ? 0 : tap, part, (int)(unsigned)off, (int)(off >> 32));
  }
  if (warp == 0) tmem_alloc(&slot, (uint32_t)p.cols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = slot;
  bool ok = true;
  const int total = (kb1 - kb0) * nt;

  if (warp < 8) {
    int a = 0;
    auto publish_behind = [&]() {
      cp_commit();
      asm volatile("cp.async.wait_group %0;\n" ::"n"(WLAG) : "memory");
      if (a >= WLAG) {
        fence_async();
        mbar_arrive(&full[(a - WLAG) % ws]);
      }
    };
    if constexpr (FIRST > 0) {
      // a warp pair per 64-voxel block, four blocks at a time: every thread puts one voxel's row together, then the
      // blocks' tiles are written in order
      using F = FirstRow<FIRST>;
      const int vox = threadIdx.x & 63, grp = threadIdx.x >> 6;
      for (int kb = kb0; kb < kb1 && ok; kb += 4) {
        const bool mine = kb + grp < kb1;
        const int v = (kb + grp) * 64 + vox;
        const int r = v / W;
        F row;
        row.load(src.a, v, v - r * W, r % H, r / H, D, H, W, mine);
        for (int g = 0; g < 4 && kb + g < kb1 && ok; ++g)
          for (int ti = 0; ti < nt && ok; ++ti, ++a) {
            const int s = a % ws;
            if (a >= ws && !warp_wait(&empty[s], (unsigned)(a / ws - 1) & 1u)) ok = false;
            if (g == grp) {
              unsigned char* d = sA + (size_t)s * 16 * WBLOCK + vox * 16;
              if (ti == 0)
                for (int o8 = 0; o8 < Co / 8; ++o8)
                  cp16_ca(sB + (size_t)((kb + g - kb0) % p.nb) * bbytes + vox * 16 + o8 * WBLOCK, dy + (long long)v * Co + o8 * 8, true);
#pragma unroll
              for (int q = 0; q < F::USED; ++q)
                if (q / 16 == t0 + ti) *reinterpret_cast<uint4*>(d + (q % 16) * WBLOCK) = row.chunk(q);
            }
            publish_behind();
          }
      }
    } else {
      // two lanes per voxel take the two chunks of a pair, so that they read 32 contiguous bytes
      const int sub = threadIdx.x & 1, vox = (threadIdx.x >> 1) & 63, half = threadIdx.x >> 7;
      int v = kb0 * 64 + vox;
      int x = v % W, y = (v / W) % H, z = v / (W * H);
      for (int kb = kb0; kb < kb1 && ok; ++kb) {
        // taps whose voxel is inside: bits tap = (dz + 1) 9 + (dy + 1) 3 + dx + 1
        const uint32_t mx = (x > 0 ? 1u : 0u) | 2u | (x < W - 1 ? 4u : 0u);
        const uint32_t my = (y > 0 ? mx : 0u) | mx << 3 | (y < H - 1 ? mx << 6 : 0u);
        const uint32_t mz = (z > 0 ? my : 0u) | my << 9 | (z < D - 1 ? my << 18 : 0u);
        const bf16* pa = src.a + (src.up ? 0 : (long long)v * src.ca) + sub * 8;
        const bf16* pb = src.b + (long long)v * src.cb + sub * 8;
        for (int ti = 0; ti < nt && ok; ++ti, ++a) {
          const int s = a % ws;
          if (a >= ws && !warp_wait(&empty[s], (unsigned)(a / ws - 1) & 1u)) ok = false;
          if (ti == 0) {   // the block's dy, for all of its tiles
            unsigned char* d = sB + (size_t)((kb - kb0) % p.nb) * bbytes + vox * 16;
            for (int o8 = 2 * half + sub; o8 < Co / 8; o8 += 4) cp16_ca(d + o8 * WBLOCK, dy + (long long)v * Co + o8 * 8, true);
          }
          unsigned char* d = sA + (size_t)s * 16 * WBLOCK + (8 * half + sub) * WBLOCK + vox * 16;
#pragma unroll
          for (int jj = 0; jj < 4; ++jj, d += 2 * WBLOCK) {
            const int4 e = table[ti * 8 + half * 4 + jj];
            const bool in = e.y >= 0 && ((mz >> e.x) & 1u);
            const bf16* q = src.a;
            if (in) {
              const long long off = (long long)e.w << 32 | (unsigned)e.z;
              if (e.y == 0) q = pa + off;
              else if (e.y == 2) q = pb + off;
              else
                q = pa + ((long long)(((z + e.x / 9 - 1) >> 1) * (H >> 1) + ((y + (e.x / 3) % 3 - 1) >> 1)) * (W >> 1) +
                          ((x + e.x % 3 - 1) >> 1)) * src.ca + e.z;
            }
            cp16_ca(d, q, in);
          }
          publish_behind();
        }
        v += 64;
        for (x += 64; x >= W; x -= W)
          if (++y == H) {
            y = 0;
            ++z;
          }
      }
    }
    cp_wait_all();
    fence_async();
    for (int i = max(0, a - WLAG); i < a; ++i) mbar_arrive(&full[i % ws]);
    if (warp >= 4) goto tail;
    if (!warp_wait(&done, 0)) ok = false;
    tc_fence_after();
    float* dst = part + (size_t)blockIdx.x * 27 * C * Co;
    for (int ti = 0; ti < nt; ++ti) {
      const int k = (t0 + ti) * 128 + warp * 32 + lane;
      const bool in = ok && k < 27 * C;
      for (int col = 0; col < Co; col += 16) {
        float r[16];
        tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(ti * Co + col), r);
        if (!in) continue;
        float* q = dst + (size_t)k * Co + col;
#pragma unroll
        for (int e = 0; e < 16; e += 4) *reinterpret_cast<float4*>(q + e) = make_float4(r[e], r[e + 1], r[e + 2], r[e + 3]);
      }
    }
  } else if (lane == 0) {
    // both operands MN-major (bits 15, 16)
    const uint32_t idesc = idesc_bf16(128, Co) | (1u << 15) | (1u << 16);
    for (int a = 0; a < total && ok; ++a) {
      const int s = a % ws, kb = a / nt, ti = a - kb * nt;
      if (!mbar_wait(&full[s], (unsigned)(a / ws) & 1u)) {
        ok = false;
        break;
      }
      const uint64_t ad = desc_plain(saddr(sA) + (uint32_t)s * 16 * WBLOCK, 128, WBLOCK);
      const uint64_t bd = desc_plain(saddr(sB) + (uint32_t)(kb % p.nb) * bbytes, 128, WBLOCK);
#pragma unroll
      for (int r = 0; r < 4; ++r)   // 16 voxels: 256 bytes further, 16 in descriptor units
        mma_bf16(tmem + (uint32_t)(ti * Co), ad + 16 * r, bd + 16 * r, idesc, (kb > 0 || r > 0) ? 1u : 0u);
      mma_commit(&empty[s]);
    }
    mma_commit(&done);
  }
tail:
  if (!ok) atomicOr(err, 1);
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_free(tmem, (uint32_t)p.cols);
}

// dw[o][c][tap] = sum over the splits of part[split][tap][c][o], in split order
__global__ void k_wgrad_sum(const float* __restrict__ part, float* __restrict__ dw, int splits, int C, int Co) {
  const int n = 27 * C * Co;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    float s = 0.f;
#pragma unroll 8
    for (int z = 0; z < splits; ++z) s += part[(size_t)z * n + i];
    const int o = i % Co, r = i / Co, c = r % C, tap = r / C;
    dw[((size_t)o * C + c) * 27 + tap] = s;
  }
}

// ------------------------------------------------------------------ weights

// w [Co][Ci][27] (FP32) -> wp [k / 16][(k / 8) % 2][o][k % 8] (k = tap Ci + c, zero past 27 Ci) and, if wtp is not
// null, the flipped transpose [k' / 16][(k' / 8) % 2][c][k' % 8] (k' = tap' Co + o holds w[o][c][26 - tap'])
__global__ void k_conv3_pack(const float* __restrict__ w, bf16* __restrict__ wp, bf16* __restrict__ wtp, int Co, int Ci) {
  const int K = (27 * Ci + 15) / 16 * 16, Kt = (27 * Co + 15) / 16 * 16;
  const int n1 = Co * K, n2 = wtp ? Ci * Kt : 0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n1 + n2; i += gridDim.x * blockDim.x) {
    const bool fw = i < n1;
    const int j = fw ? i : i - n1, rows = fw ? Co : Ci;
    const int e = j % 8, r = (j / 8) % rows, k = j / (8 * rows) * 8 + e;
    float val = 0.f;
    if (fw) {
      if (k < 27 * Ci) val = w[((size_t)r * Ci + k % Ci) * 27 + k / Ci];
      wp[j] = __float2bfloat16_rn(val);
    } else {
      if (k < 27 * Co) val = w[((size_t)(k % Co) * Ci + r) * 27 + (26 - k / Co)];
      wtp[j] = __float2bfloat16_rn(val);
    }
  }
}

// ------------------------------------------------------------------ host side

static int sm_count() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms > 0 ? sms : 1;
}
static int pow2_cols(int c) {
  int p = 32;
  while (p < c) p *= 2;
  return p;
}
constexpr unsigned kSmemTwo = 113 * 1024, kSmemOne = 226 * 1024;   // shared memory of a CTA for two and one per SM

// Ring, weight staging and z range for a layer.  Two CTAs per SM hide one another's loads and epilogues, so a
// layout that leaves room for them comes first; weights stay resident where they fit (up to C = N = 32).
static bool conv_plan(ConvPlan* p, int C, int N, int D, int H, int W) {
  const unsigned plane = (unsigned)(C / 8) * CHUNK, btot = 27u * C * N * 2, extra = 128 + 28 * 8 + 16;
  struct Opt { int planes, seq, res; };
  const Opt opts[] = {{4, 0, 1}, {4, 0, 0}, {3, 0, 1}, {3, 0, 0}, {2, 1, 0}};
  p->C = C;
  p->N = N;
  for (unsigned limit : {kSmemTwo, kSmemOne})
    for (const Opt& o : opts) {
      p->planes = o.planes;
      p->seq = o.seq;
      unsigned b = btot;
      p->sc = C;
      p->stages = 0;
      if (!o.res) {
        p->sc = 16;
        for (int s = 16; s <= C; s += 16)
          if (C % s == 0 && (unsigned)s * N * 2 <= 20480u) p->sc = s;
        p->stages = 4;
        b = 4u * p->sc * N * 2;
      }
      p->smem = (unsigned)o.planes * plane + b + extra;
      if (p->smem > limit) continue;
      const long long tiles = (long long)((W + TX - 1) / TX) * ((H + TY - 1) / TY);
      int per_sm = (int)(kSmemOne / p->smem);
      if (per_sm > 4) per_sm = 4;   // registers
      // accumulators of the CTAs of an SM share 512 TMEM columns
      while (per_sm > 1 && per_sm * pow2_cols(2 * N) > 512) --per_sm;
      const int slots = sm_count() * per_sm;
      int zs = std::max(1, std::min(D, (int)(slots / tiles)));
      p->nz = o.seq ? 1 : (D + zs - 1) / zs;
      p->accs = p->nz > 1 ? 2 : 1;
      if (p->accs * N > 512) p->accs = 1;
      p->cols = pow2_cols(p->accs * N);
      return true;
    }
  return false;
}

// Voxel ranges of the weight gradient: those of the split-K GEMM over im2col rows (K padded to 128, at most 64
// splits, about four waves of tiles over 152 SMs: a constant of that rule, so that the boundaries of the partial sums, and
// with them the results, do not depend on the device).
static bool wgrad_plan(WgradPlan* p, int C, int Co, int D, int H, int W) {
  const long long V = (long long)D * H * W;
  if (Co % 16 || Co > 256 || V % 64 || V >= (1ll << 31) - 64) return false;
  p->C = C;
  p->Co = Co;
  p->tiles = (27 * C + 127) / 128;
  p->nkb = (int)(V / 64);
  const int mn = p->tiles * std::max(1, Co / 128);
  const int want = (int)std::max(1ll, std::min({64ll, (4 * 152ll) / mn, V / 64}));
  const int sp = std::min(want, p->nkb);
  p->kbs = (p->nkb + sp - 1) / sp;
  p->splits = (p->nkb + p->kbs - 1) / p->kbs;
  // tiles per CTA: all that fit into half of TMEM, fewer where that leaves SMs without a CTA
  p->tj = std::max(1, std::min(p->tiles, 256 / Co));
  while (C % 16 == 0 && p->tj > 1 && p->splits * ((p->tiles + p->tj - 1) / p->tj) < 2 * sm_count()) --p->tj;
  p->jobs = (p->tiles + p->tj - 1) / p->tj;
  p->tj = (p->tiles + p->jobs - 1) / p->jobs;
  // before a tile is written, the one ws back has been multiplied; the dy buffer of a block is written with the
  // block's first tile, so the last tile of the buffer's previous block has to lie that far back: (nb - 1) tiles + 1 >=
  // ws for the CTA with the fewest tiles per block
  const int fewest = p->tiles - (p->jobs - 1) * p->tj;
  p->cols = pow2_cols(p->tj * Co);
  for (p->ws = WSTAGES; p->ws > WLAG; --p->ws) {
    p->nb = (p->ws - 1 + fewest - 1) / fewest + 1;
    p->smem = p->ws * 16u * WBLOCK + (unsigned)p->nb * (Co / 8) * WBLOCK + 8u * p->tj * 16 + 128;
    if (p->smem <= kSmemOne) break;
  }
  return p->ws > WLAG && p->jobs <= 65535;
}

template <class K>
static cudaError_t allow_smem(K kernel, unsigned bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

}  // namespace lbmnn

using namespace lbmnn;

#define NN_CK(x)                                 \
  do {                                           \
    if ((x) != cudaSuccess) return LBM_ERR_CUDA; \
  } while (0)

// calls f with the narrow input's channel count as a constant
template <class F>
static bool by_narrow(int C, F&& f) {
  switch (C) {
    case 1: f(std::integral_constant<int, 1>()); return true;
    case 2: f(std::integral_constant<int, 2>()); return true;
    case 3: f(std::integral_constant<int, 3>()); return true;
    case 4: f(std::integral_constant<int, 4>()); return true;
    case 5: f(std::integral_constant<int, 5>()); return true;
    case 6: f(std::integral_constant<int, 6>()); return true;
    case 7: f(std::integral_constant<int, 7>()); return true;
    case 8: f(std::integral_constant<int, 8>()); return true;
  }
  return false;
}

static bool conv_args_ok(const void* xa, int Ca, int up, const void* xb, int Cb, int D, int H, int W) {
  if (!xa || Ca <= 0 || Cb < 0 || (Cb > 0 && !xb) || D <= 0 || H <= 0 || W <= 0) return false;
  if (up && ((D | H | W) & 1)) return false;
  if ((long long)D * H * W >= (1ll << 31)) return false;
  if (Ca % 16 == 0 && Cb % 16 == 0) return true;
  return Ca <= 8 && Cb == 0 && !up;   // the narrow first layer
}

// the kernels read and write 16 bytes at a time
static bool aligned16(std::initializer_list<const void*> ps) {
  uintptr_t u = 0;
  for (const void* q : ps) u |= reinterpret_cast<uintptr_t>(q);
  return (u & 15u) == 0;
}

extern "C" {

int64_t lbm_nn_conv3_packed(int32_t Co, int32_t Ci) { return (int64_t)Co * ((27 * (int64_t)Ci + 15) / 16 * 16); }

int32_t lbm_nn_conv3_fits(int32_t Ca, int32_t up, int32_t Cb, int32_t Co) {
  const char some = 0;
  if (!conv_args_ok(&some, Ca, up, Cb ? &some : nullptr, Cb, 8, 8, 8) || Co <= 0 || Co % 16 || Co > 256) return 0;
  const int C = Ca + Cb;
  ConvPlan p;
  WgradPlan w;
  if (C % 16 == 0 && (C > 256 || !conv_plan(&p, C, Co, 8, 8, 8) || !conv_plan(&p, Co, C, 8, 8, 8))) return 0;
  return wgrad_plan(&w, C, Co, 8, 8, 8) ? 1 : 0;
}

lbm_status lbm_nn_pad8(const void* x, void* x8, int64_t V, int32_t C, void* stream) {
  if (!x || !x8 || V <= 0 || C <= 0 || C > 8 || !aligned16({x8})) return LBM_ERR_INVALID_ARG;
  k_pad8<<<grid_for(V), 256, 0, static_cast<cudaStream_t>(stream)>>>(static_cast<const bf16*>(x), static_cast<bf16*>(x8), V, C);
  NN_CK(cudaGetLastError());
  return LBM_OK;
}

lbm_status lbm_nn_conv3_pack(const float* w, void* wp, void* wtp, int32_t Co, int32_t Ci, void* stream) {
  if (!w || !wp || Co <= 0 || Ci <= 0 || Co > 4096 || Ci > 4096) return LBM_ERR_INVALID_ARG;
  const long long n = lbm_nn_conv3_packed(Co, Ci) + (wtp ? lbm_nn_conv3_packed(Ci, Co) : 0);
  if (n >= (1ll << 31)) return LBM_ERR_INVALID_ARG;
  k_conv3_pack<<<grid_for(n), 256, 0, static_cast<cudaStream_t>(stream)>>>(w, static_cast<bf16*>(wp), static_cast<bf16*>(wtp),
                                                                          Co, Ci);
  NN_CK(cudaGetLastError());
  return LBM_OK;
}

lbm_status lbm_nn_conv3(const void* xa, int32_t Ca, int32_t up, const void* xb, int32_t Cb, int32_t D, int32_t H, int32_t W,
                        const void* wp, int32_t N, const float* bias, int32_t relu, void* y0, int32_t n0, void* y1,
                        void* stream) {
  if (!conv_args_ok(xa, Ca, up, xb, Cb, D, H, W) || !wp || !y0 || N <= 0 || N % 16 || N > 256 || n0 <= 0 || n0 > N ||
      n0 % 16 || (n0 < N && !y1) || !aligned16({xa, xb, wp, bias, y0, y1}))
    return LBM_ERR_INVALID_ARG;
  int* err = err_word();
  if (!err) return LBM_ERR_CUDA;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const ConvOut out{static_cast<bf16*>(y0), static_cast<bf16*>(y1), bias, n0, relu ? 1 : 0};
  const int tx = (W + TX - 1) / TX, ty = (H + TY - 1) / TY;
  if (Ca % 16) {
    const int k16 = (27 * Ca + 15) / 16;
    const unsigned smem = (unsigned)k16 * (4096 + N * 32) + 128;
    if (smem > kSmemOne) return LBM_ERR_INVALID_ARG;
    cudaError_t e = cudaSuccess;
    by_narrow(Ca, [&](auto c) {
      constexpr int C = decltype(c)::value;
      e = allow_smem(k_conv3_first<C>, smem);
      if (e != cudaSuccess) return;
      const long long need = ((long long)D * H * W + 127) / 128;
      const unsigned grid = (unsigned)std::min<long long>(need, sm_count() * std::max(1u, std::min(3u, kSmemOne / smem)));
      k_conv3_first<C><<<grid, 128, smem, st>>>(static_cast<const bf16*>(xa), static_cast<const bf16*>(wp), out, N, D, H, W,
                                               pow2_cols(N), err);
    });
    NN_CK(e);
  } else {
    ConvPlan p;
    if (!conv_plan(&p, Ca + Cb, N, D, H, W) || (long long)tx * ty * ((D + p.nz - 1) / p.nz) >= (1ll << 31)) return LBM_ERR_INVALID_ARG;
    NN_CK(allow_smem(k_conv3, p.smem));
    const ConvSrc src{static_cast<const bf16*>(xa), static_cast<const bf16*>(xb), Ca, Cb, up ? 1 : 0};
    k_conv3<<<(unsigned)tx * (unsigned)ty * (unsigned)((D + p.nz - 1) / p.nz), 192, p.smem, st>>>(src, static_cast<const bf16*>(wp), out, p, D, H, W, err);
  }
  NN_CK(cudaGetLastError());
  return LBM_OK;
}

int64_t lbm_nn_conv3_wgrad_scratch(int32_t D, int32_t H, int32_t W, int32_t C, int32_t Co) {
  WgradPlan p;
  if (D <= 0 || H <= 0 || W <= 0 || C <= 0 || Co <= 0 || !wgrad_plan(&p, C, Co, D, H, W)) return 0;
  return (int64_t)p.splits * 27 * C * Co;
}

lbm_status lbm_nn_conv3_wgrad(const void* xa, int32_t Ca, int32_t up, const void* xb, int32_t Cb, int32_t D, int32_t H,
                              int32_t W, const void* dy, int32_t Co, float* scratch, float* dw, void* stream) {
  if (!conv_args_ok(xa, Ca, up, xb, Cb, D, H, W) || !dy || Co <= 0 || Co % 16 || !scratch || !dw ||
      !aligned16({xa, xb, dy, scratch}))
    return LBM_ERR_INVALID_ARG;
  WgradPlan p;
  if (!wgrad_plan(&p, Ca + Cb, Co, D, H, W)) return LBM_ERR_INVALID_ARG;
  int* err = err_word();
  if (!err) return LBM_ERR_CUDA;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const ConvSrc src{static_cast<const bf16*>(xa), static_cast<const bf16*>(xb), Ca, Cb, up ? 1 : 0};
  auto launch = [&](auto* kern) {
    cudaError_t e = allow_smem(kern, p.smem);
    if (e != cudaSuccess) return e;
    kern<<<dim3(p.splits, p.jobs), 288, p.smem, st>>>(src, static_cast<const bf16*>(dy), scratch, p, D, H, W, err);
    return cudaGetLastError();
  };
  cudaError_t e = cudaSuccess;
  if (Ca % 16) by_narrow(Ca, [&](auto c) { e = launch(k_wgrad<decltype(c)::value>); });
  else e = launch(k_wgrad<0>);
  NN_CK(e);
  k_wgrad_sum<<<grid_for(27ll * (Ca + Cb) * Co), 256, 0, st>>>(scratch, dw, p.splits, Ca + Cb, Co);
  NN_CK(cudaGetLastError());
  return LBM_OK;
}

}  // extern "C"

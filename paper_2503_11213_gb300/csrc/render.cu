// Per-pixel DP rendering (supplement, "Local DP PSF convolution") on sm_103a.
//
// out_L[n,c,y,x] = sum_{u,v} Ipad[n,c,y+u,x+v] * K_L(y,x,c)[ks-1-u][ks-1-v]
// with Ipad the image replicate-padded by p = (ks-1)/2 (likewise R) and, in
// bank mode, K(y,x,c) = (1-t) B[f][z0][lam] + t B[f][z0+1][lam] selected per
// pixel from its radial image height and depth (linear in inverse depth);
// with a quadrant bank, from the nearest first-quadrant field point of
// (|X|, |Y|) and the PSF's flip symmetry about both axes (Sec. 5.3).
//
// The render is linear in the kernel, so a pixel's output is
// (1-t) (I * B[f][z0]) + t (I * B[f][z0+1]): a sum over bank slices with
// per-pixel weights.  Neighbouring pixels use different slices (field index
// and depth bracket both vary), so each thread block, for one image tile and
// one channel:
//   1. selects (slice key, t) per pixel in FP32 without contraction;
//   2. splits the tile into vertical segments of SEG pixels and marks, per
//      slice key, the segments that need it (a bitmask per key);
//   3. cuts every key's segment list into chunks of 32 (one lane per
//      segment, lanes in column order so shared-memory reads of the staged
//      tile are conflict-free);
//   4. each warp takes chunks; for a chunk it streams the key's taps
//      through a warp-private shared-memory buffer, VB columns at a time,
//      prefetching the next block into registers while computing, and each
//      lane slides a register window of SEG image rows down the staged
//      tile+halo: per tap one shared load of the image, one broadcast load of
//      the (L, R) tap pair and 2*SEG FMAs;
//   5. weighted segment results go to a shared accumulator.  Every pixel
//      receives at most two non-zero contributions (its two slices), so the
//      order of the additions cannot change the result: deterministic.
//
// That is the form for callers without a workspace; with one, the render goes
// through a re-laid bank (render_quad_kernel below).  Each is the faster over
// a part of the sizes: direct_is_faster.

#define SD_TU 2  // translation unit id of this file's SD_CHECK sites
#include <algorithm>
#include <type_traits>

#include "render_common.cuh"

namespace sd {

// Shared-memory layout of one block (sizes in 4-byte words).
template <int TX, int VB>
struct RenderSmem {
  static constexpr int NT = 4 * TX;          // threads = segments
  static constexpr int NW = NT / 32;         // warps
  static constexpr int NPX = TX * RT_Y;      // pixels per tile
  static constexpr int MW = NT / 32;         // mask words per key
  // tap rows padded to a multiple of SEG (zeros beyond ks): 2 buffers
  __host__ __device__ static int ku(int ks) { return (ks + SEG - 1) / SEG * SEG; }
  __host__ __device__ static size_t kbuf_words(int ks) { return (size_t)2 * (2 * ku(ks) * VB); }
  __host__ __device__ static size_t halo_words(int ks) { return (size_t)(TX + ks - 1) * (RT_Y + ks - 1 + SEG); }
  static size_t bytes(int ks) {
    size_t w = halo_words(ks) + NW * kbuf_words(ks) + 3 * (size_t)NPX  // halo, K, accL/R, t
               + (size_t)RK * MW + (RK + 1) + MAX_CHUNKS               // masks, prefix, chunks
               + NPX / 2;                                              // u16 keys
    return 4 * w;
  }
};

template <class TB>
__device__ __forceinline__ float ldk(const TB* p) { return to_f32<TB>(__ldg(p)); }

template <class TI, class TB, int TX, int VB, int KSMAX>
__global__ void __launch_bounds__(4 * TX, 1) render_fwd_kernel(const RenderParams P) {
  using SM = RenderSmem<TX, VB>;
  constexpr int NT = SM::NT, NW = SM::NW, NPX = SM::NPX, MW = SM::MW;
  constexpr int NR = (2 * ((KSMAX + SEG - 1) / SEG * SEG) * VB + 31) / 32;  // prefetch regs
  extern __shared__ __align__(16) unsigned char smem[];
  const int ks = P.ks, p = (ks - 1) >> 1, ks2 = ks * ks;
  const int S = P.halo_w;
  float* halo = reinterpret_cast<float*>(smem);
  float* kbuf = halo + SM::halo_words(ks);                   // NW x 2 x [ks][VB][2]
  float* accL = kbuf + NW * SM::kbuf_words(ks);
  float* accR = accL + NPX;
  float* pt = accR + NPX;
  unsigned* mask = reinterpret_cast<unsigned*>(pt + NPX);     // [RK][MW]
  int* kpre = reinterpret_cast<int*>(mask + RK * MW);         // [RK + 1]
  int* chunks = kpre + RK + 1;                                // [MAX_CHUNKS]
  unsigned short* prel = reinterpret_cast<unsigned short*>(chunks + MAX_CHUNKS);
  __shared__ int s_kmin, s_kmax, s_nchunks, s_next;

  const int tx0 = blockIdx.x * TX, ty0 = blockIdx.y * RT_Y;
  const int n = blockIdx.z / P.C, c = blockIdx.z - n * P.C;
  const int lam = (P.NL == P.C) ? c : 0;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int H = P.H, W = P.W;
  const bool two = (P.Z > 1);

  // ---- 1. per-pixel selection; stage the tile + halo -------------------------
  const int seg_col = tid % TX, seg_rb = tid / TX;
  int kmin_t = 0x7fffffff, kmax_t = -1;
  int key_j[SEG];
  float t_j[SEG];
#pragma unroll
  for (int j = 0; j < SEG; ++j) {
    int yy = ty0 + seg_rb * SEG + j, xx = tx0 + seg_col;
    key_j[j] = -1;
    t_j[j] = 0.f;
    if (yy < H && xx < W) {
      float d = P.depth[((size_t)n * H + yy) * W + xx];
      select_slice(P, yy, xx, d, &key_j[j], &t_j[j]);
      kmin_t = min(kmin_t, key_j[j]);
      kmax_t = max(kmax_t, key_j[j] + (two ? 1 : 0));
    }
    pt[(seg_rb * SEG + j) * TX + seg_col] = t_j[j];
  }
  if (tid == 0) {
    s_kmin = 0x7fffffff;
    s_kmax = -1;
  }
  // the tile and its halo, one warp per row: 16-byte loads of EPV columns
  // wherever such a group lies inside the image row at a 16-byte aligned
  // address, clamped single loads at the image edges (replicate padding)
  const TI* img = reinterpret_cast<const TI*>(P.aif) + ((size_t)n * P.C + c) * H * W;
  {
    constexpr int EPV = 16 / (int)sizeof(TI);
    const int x_lo = tx0 - p;  // image column of halo column 0
    for (int r = warp; r < P.halo_h; r += NW) {
      const size_t rowoff = (size_t)min(max(ty0 + r - p, 0), H - 1) * W;
      const TI* src = img + rowoff;
      // first column at or left of x_lo whose address is 16-byte aligned
      const int mis = (int)((reinterpret_cast<uintptr_t>(src) / sizeof(TI) + (size_t)(x_lo + 4 * EPV)) % EPV);
      const int xa = x_lo - mis;
      const int ng = (S + mis + EPV - 1) / EPV;
      for (int g = lane; g < ng; g += 32) {
        const int x = xa + g * EPV;
        float v[EPV];
        if (x >= 0 && x + EPV <= W) {
          const uint4 q = __ldg(reinterpret_cast<const uint4*>(src + x));
          const TI* e = reinterpret_cast<const TI*>(&q);
#pragma unroll
          for (int k = 0; k < EPV; ++k) v[k] = to_f32<TI>(e[k]);
        } else {
#pragma unroll
          for (int k = 0; k < EPV; ++k) v[k] = to_f32<TI>(src[min(max(x + k, 0), W - 1)]);
        }
#pragma unroll
        for (int k = 0; k < EPV; ++k) {
          const int cc = x + k - x_lo;
          if (cc >= 0 && cc < S) halo[r * S + cc] = v[k];
        }
      }
    }
  }
  for (int i = tid; i < NPX; i += NT) {
    accL[i] = 0.f;
    accR[i] = 0.f;
  }
  __syncthreads();
  atomicMin(&s_kmin, kmin_t);
  atomicMax(&s_kmax, kmax_t);
  __syncthreads();
  const int kmin = s_kmin, kmax = s_kmax;
#pragma unroll
  for (int j = 0; j < SEG; ++j)
    prel[(seg_rb * SEG + j) * TX + seg_col] =
        (unsigned short)(key_j[j] >= 0 ? key_j[j] - kmin : 0xffff);

  float* kb = kbuf + warp * SM::kbuf_words(ks);  // this warp's 2 x [ks][VB][side]
  const int nblk = (ks + VB - 1) / VB;
  const int KU = SM::ku(ks);
  const int kb_elems = 2 * KU * VB;

  for (int wbase = kmin; wbase <= kmax; wbase += RK) {
    // ---- 2. segment bitmask per key of the window ---------------------------
    for (int i = tid; i < RK * MW; i += NT) mask[i] = 0u;
    __syncthreads();
#pragma unroll
    for (int j = 0; j < SEG; ++j) {
      int k0 = key_j[j];
      if (k0 < 0) continue;
      float t = t_j[j];
      // slices with zero weight need no work
      if ((!two || t < 1.f) && k0 >= wbase && k0 < wbase + RK)
        atomicOr(&mask[(k0 - wbase) * MW + warp], 1u << lane);
      if (two && t > 0.f && k0 + 1 >= wbase && k0 + 1 < wbase + RK)
        atomicOr(&mask[(k0 + 1 - wbase) * MW + warp], 1u << lane);
    }
    __syncthreads();
    // ---- 3. chunks of 32 segments per key (warp 0 scans the key counts) -----
    if (warp == 0) {
      int carry = 0;
      for (int k0 = 0; k0 < RK; k0 += 32) {
        int k = k0 + lane;
        int cnt = 0;
        for (int w = 0; w < MW; ++w) cnt += __popc(mask[k * MW + w]);
        int nch = (cnt + 31) >> 5;
        int v = nch;
        for (int o = 1; o < 32; o <<= 1) {
          int u = __shfl_up_sync(0xffffffffu, v, o);
          if (lane >= o) v += u;
        }
        kpre[k] = carry + v - nch;
        carry += __shfl_sync(0xffffffffu, v, 31);
      }
      if (lane == 0) {
        kpre[RK] = carry;
        s_nchunks = carry;
      }
    }
    __syncthreads();
    const int nchunks = s_nchunks;  // <= NT * 2 * SEG / 32 + RK <= MAX_CHUNKS
    for (int k = tid; k < RK; k += NT)
      for (int q = kpre[k]; q < kpre[k + 1]; ++q) chunks[q] = (k << 8) | (q - kpre[k]);
    if (tid == 0) s_next = NW;
    __syncthreads();

    // ---- 4. warps take chunks (first one by index, then from a counter) -------
    for (int ch = warp; ch < nchunks;) {
      const int rel = chunks[ch] >> 8, sub = chunks[ch] & 0xff;
      const int key = wbase + rel;
      // this lane's segment: the (sub*32 + lane)-th set bit of the key mask
      int want = sub * 32 + lane, seg = -1;
      for (int w = 0; w < MW; ++w) {
        unsigned m = mask[rel * MW + w];
        int pc = __popc(m);
        if (seg < 0 && want >= 0 && want < pc) {
          for (int q = 0; q < want; ++q) m &= m - 1;
          seg = w * 32 + __ffs(m) - 1;
        }
        want -= pc;
      }
      const bool act = seg >= 0;
      const int sg = act ? seg : 0;
      // segment id = warp * 32 + lane of the owner thread = rb * TX + col
      const int col = sg % TX, rb = sg / TX;
      const int f = key / P.Z, z = key - f * P.Z;
      // quadrant bank: field cell and flips (x: mirror columns and exchange
      // L and R; y: mirror rows); radial bank: flips = 0
      const int flips = f / P.FC, cell = f - flips * P.FC;
      const TB* K0 = reinterpret_cast<const TB*>(P.bank) +
                     (((size_t)cell * P.Z + z) * P.NL + lam) * 2 * ks2;
      const TB* KL = (flips & 1) ? K0 + ks2 : K0;
      const TB* KR = (flips & 1) ? K0 : K0 + ks2;
      const bool mx = flips & 1, my = flips & 2;
      // K block b covers v in [b*VB, b*VB + VB): element (u, vv, side) =
      // K_side[ks-1-u][ks-1-(b*VB+vv)] at kb[buf][(u*VB + vv)*2 + side]
      float pre[NR];
      auto fetch = [&](int b) {
#pragma unroll
        for (int r = 0; r < NR; ++r) {
          int e = lane + 32 * r;
          float v = 0.f;
          if (e < kb_elems) {
            int side = e & 1, uv = e >> 1, u = uv / VB, vv = uv - u * VB;
            int v_ = b * VB + vv;
            if (v_ < ks && u < ks)
              v = ldk<TB>((side ? KR : KL) + (my ? u : ks - 1 - u) * ks + (mx ? v_ : ks - 1 - v_));
          }
          pre[r] = v;
        }
      };
      auto commit = [&](float* dst) {
#pragma unroll
        for (int r = 0; r < NR; ++r) {
          int e = lane + 32 * r;
          if (e < kb_elems) dst[e] = pre[r];
        }
      };
      // rows [ulo, uhi] of the fetched block holding a non-zero tap (of
      // either side): blur discs leave many kernel rows empty
      auto extent = [&](int& ulo, int& uhi) {
        unsigned lo_l = 0xffffffffu, hi_l = 0u;
#pragma unroll
        for (int r = 0; r < NR; ++r) {
          int e = lane + 32 * r;
          if (e < kb_elems && pre[r] != 0.f) {
            unsigned u = (unsigned)((e >> 1) / VB);
            lo_l = min(lo_l, u);
            hi_l = max(hi_l, u + 1u);
          }
        }
        ulo = (int)__reduce_min_sync(0xffffffffu, lo_l);
        uhi = (int)__reduce_max_sync(0xffffffffu, hi_l) - 1;
      };
      int ulo_n, uhi_n;
      fetch(0);
      extent(ulo_n, uhi_n);
      commit(kb);
      __syncwarp();
      // (L, R) sums of the SEG pixels: one packed two-lane FMA per tap and
      // pixel (its components round like fmaf)
      float2 a2[SEG];
#pragma unroll
      for (int j = 0; j < SEG; ++j) a2[j] = make_float2(0.f, 0.f);
      const float* base = halo + (rb * SEG) * S + col;
      for (int b = 0; b < nblk; ++b) {
        const float* kcur = kb + (b & 1) * kb_elems;
        const int ulo = ulo_n, uhi = uhi_n;
        if (b + 1 < nblk) fetch(b + 1);  // loads in flight during the compute
        // rows u0 in [u_begin, uhi]: the taps outside are zero (KU = ks
        // rounded up to SEG; the padding taps are zero too)
        const int u_begin = (ulo / SEG) * SEG;
        const int vmax = uhi < 0 ? 0 : min(VB, ks - b * VB);
        for (int vv = 0; vv < vmax; ++vv) {
          // the deepest halo row this column's window reaches
          if (!SD_CHECK((size_t)(rb * SEG + (uhi / SEG) * SEG + 2 * SEG - 1) * S + col + b * VB + vv,
                        SM::halo_words(ks)))
            continue;
          const float* colp = base + b * VB + vv;
          float win[SEG];
#pragma unroll
          for (int j = 0; j < SEG; ++j) win[j] = colp[(u_begin + j) * S];
          const float2* kp = reinterpret_cast<const float2*>(kcur) + vv;
          for (int u0 = u_begin; u0 <= uhi; u0 += SEG) {
#pragma unroll
            for (int q = 0; q < SEG; ++q) {
              const int u = u0 + q;
              float2 w2 = kp[u * VB];
#pragma unroll
              for (int j = 0; j < SEG; ++j) {
                const float iv = win[(q + j) % SEG];
                a2[j] = __ffma2_rn(make_float2(iv, iv), w2, a2[j]);
              }
              win[q] = colp[(u + SEG) * S];
            }
          }
        }
        if (b + 1 < nblk) {
          extent(ulo_n, uhi_n);
          commit(kb + ((b + 1) & 1) * kb_elems);
        }
        __syncwarp();
      }
      if (act) {
#pragma unroll
        for (int j = 0; j < SEG; ++j) {
          int pix = (rb * SEG + j) * TX + col;
          if (!SD_CHECK(pix, SM::NPX)) continue;
          unsigned short r16 = prel[pix];
          if (r16 == 0xffff) continue;
          int k0 = kmin + (int)r16;
          float t = pt[pix];
          float w = (k0 == key) ? (two ? 1.f - t : 1.f) : ((two && k0 + 1 == key) ? t : 0.f);
          if (w != 0.f) {
            atomicAdd(&accL[pix], a2[j].x * w);
            atomicAdd(&accR[pix], a2[j].y * w);
          }
        }
      }
      int nxt = 0;
      if (lane == 0) nxt = atomicAdd(&s_next, 1);
      ch = __shfl_sync(0xffffffffu, nxt, 0);
    }
    __syncthreads();
  }
  // ---- 5. write the L and R planes of channel c ---------------------------------
  TI* outL = reinterpret_cast<TI*>(P.out) + (((size_t)n * 2 * P.C + c) * H) * W;
  TI* outR = reinterpret_cast<TI*>(P.out) + (((size_t)n * 2 * P.C + P.C + c) * H) * W;
  for (int i = tid; i < NPX; i += NT) {
    int yy = ty0 + i / TX, xx = tx0 + i % TX;
    if (yy < H && xx < W) {
      outL[(size_t)yy * W + xx] = from_f32<TI>(accL[i]);
      outR[(size_t)yy * W + xx] = from_f32<TI>(accR[i]);
    }
  }
}

template <class TI, class TB, int TX, int VB, int KSMAX>
sd_status launch_fwd_cfg(RenderParams& P, cudaStream_t s) {
  using SM = RenderSmem<TX, VB>;
  P.halo_w = TX + P.ks - 1;
  P.halo_h = RT_Y + P.ks - 1 + SEG;
  size_t smem = SM::bytes(P.ks);
  auto k = render_fwd_kernel<TI, TB, TX, VB, KSMAX>;
  SD_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  dim3 grid((P.W + TX - 1) / TX, (P.H + RT_Y - 1) / RT_Y, P.N * P.C);
  k<<<grid, SM::NT, smem, s>>>(P);
  return launch_status();
}

// ---------------------------------------------------------------------------
// Renders through a re-laid bank (render_quad_kernel).  A warp renders 2 rows
// x 8 neighbouring pixels with its lanes over the taps: a lane owns an item
// of 2 x 4 taps (both planes), so one read of 3 rows x 12 image values and
// one of 16 tap values feed 128 packed two-lane FMAs, and a warp only visits
// the slices its 16 pixels use (2.8 of them on a 1024 x 1024 Perlin depth map
// and a 32 x 32 bank) with every lane at work.  render_fwd_kernel's lanes are
// pixel segments that share a slice: its chunks of 32 segments were 78 %
// full there, 50 % at 256 x 256 (more slices a tile), and its tiles of 0.5 ms
// filled 5.05 waves.
//   The taps come from a per-call re-layout: for every key and wavelength the
// items with a non-zero tap, compacted in raster order (blur discs smaller
// than the patch and empty corners are never visited), 32 to an iteration:
//   float4 [it][part][lane]: part = 2 row + half: (L, R) of taps 2 half, + 1;
//   uint16 [it][lane]: row pair << 8 | quad.
// Neighbouring warps use the same slices in the same order, so most tap reads
// hit L1.  Bound by the FMA pipe and the shared-memory and L1 reads (52
// wavefronts per 128 FMAs).  Sums in a fixed order: deterministic.
//   Blocks whose tile holds an infinite or NaN value skip the zero taps (the
// same sums where the values are finite), so that a pixel takes such a value
// through its non-zero taps only, whatever the items cover.
//   Against render_fwd_kernel (us, FP32, bank 32 x 32 but where noted; smaller
// kernels: direct_is_faster):
// 64 x 64 gray at ks 31 and an 8 x 4 bank 157 -> 16 (two launches); RGB at
// ks 65: 256 x 256 1930 -> 364, 512 x 512 1630 -> 780, 8 x 512 x 512
// 8590 -> 4990, 1024 x 1024 3077 -> 2040 (re-layout 41 of them); ks 127
// 256 x 256 2266 -> 700.
// ---------------------------------------------------------------------------
constexpr int RQ_W = 8;             // warps per block
constexpr int RQ_R = 2, RQ_X = 8;   // pixels of a warp's group

struct QuadLayout {
  int nq, maxit;      // quads per kernel row, iterations of a full kernel
  bool mark;          // re-lay only the slices that a pixel uses
  size_t tap_bytes, pos_bytes, cnt_bytes, use_bytes, total;
};

inline QuadLayout quad_layout(const RenderParams& P) {
  QuadLayout L;
  L.nq = (P.ks + 3) / 4;
  L.maxit = ((P.ks + 1) / 2 * L.nq + 31) / 32;
  const size_t slices = (size_t)P.FC * P.Z, kl = slices * P.NL;
  L.tap_bytes = kl * L.maxit * 32 * 64;
  L.pos_bytes = (kl * L.maxit * 32 * 2 + 255) & ~(size_t)255;
  L.cnt_bytes = (kl * 4 + 255) & ~(size_t)255;
  // marking costs a pass over the pixels, the re-layout one over the bank:
  // worth it where the image is small beside the bank
  L.mark = (size_t)P.N * P.H * P.W * 64 <= kl * P.ks * P.ks;
  L.use_bytes = L.mark ? (slices + 255) & ~(size_t)255 : 0;
  L.total = L.tap_bytes + L.pos_bytes + L.cnt_bytes + L.use_bytes;
  return L;
}

// Marks the stored slices that a pixel uses.
__global__ void __launch_bounds__(256) mark_slices_kernel(const RenderParams P,
                                                          unsigned char* __restrict__ use) {
  const size_t npx = (size_t)P.N * P.H * P.W;
  const int slices = P.FC * P.Z;
  for (size_t i = (size_t)blockIdx.x * 256 + threadIdx.x; i < npx; i += (size_t)gridDim.x * 256) {
    const int x = (int)(i % P.W), y = (int)(i / P.W % P.H);
    int key;
    float t;
    select_slice(P, y, x, P.depth[i], &key, &t);
    key %= slices;  // flip classes share the stored slice
    if (P.Z == 1 || t < 1.f) use[key] = 1;
    if (P.Z > 1 && t > 0.f) use[key + 1] = 1;
  }
}

// One stored (slice, wavelength) per block: the flipped kernel in shared
// memory, then its non-zero items.
template <class TB>
__global__ void __launch_bounds__(256) quad_taps_kernel(const RenderParams P, QuadLayout QL,
                                                        float4* __restrict__ taps,
                                                        unsigned short* __restrict__ pos,
                                                        int* __restrict__ cnt,
                                                        const unsigned char* __restrict__ use) {
  extern __shared__ __align__(16) float kf[];  // [2][ks][ks]
  __shared__ int s_wc[8];
  if (use && !use[blockIdx.x / P.NL]) return;
  const int ks = P.ks, ks2 = ks * ks, kl = blockIdx.x, tid = threadIdx.x;
  const int lane = tid & 31, warp = tid >> 5;
  const TB* src = reinterpret_cast<const TB*>(P.bank) + (size_t)kl * 2 * ks2;
  for (int i = tid; i < 2 * ks2; i += 256) {  // both axes flipped: each plane reversed
    const int sd = i >= ks2;
    kf[(sd ? 3 : 1) * ks2 - 1 - i] = to_f32<TB>(__ldg(&src[i]));
  }
  __syncthreads();
  const int items = (ks + 1) / 2 * QL.nq;
  float4* dst = taps + (size_t)kl * QL.maxit * 128;
  unsigned short* dpos = pos + (size_t)kl * QL.maxit * 32;
  int n = 0;  // items so far
  for (int e0 = 0; e0 < items; e0 += 256) {
    const int e = e0 + tid, rp = e / QL.nq, q = e - rp * QL.nq;
    float v[16];
    bool nz = false;
#pragma unroll
    for (int i = 0; i < 16; ++i) {  // row, tap, side
      const int u = 2 * rp + (i >> 3), c = 4 * q + ((i >> 1) & 3);
      v[i] = e < items && u < ks && c < ks ? kf[((i & 1) * ks + u) * ks + c] : 0.f;
      nz = nz || v[i] != 0.f;
    }
    const unsigned bal = __ballot_sync(0xffffffffu, nz);
    if (lane == 0) s_wc[warp] = __popc(bal);
    __syncthreads();
    int at = n + __popc(bal & ((1u << lane) - 1u));
    for (int w = 0; w < 8; ++w) {
      at += w < warp ? s_wc[w] : 0;
      n += s_wc[w];
    }
    if (nz && SD_CHECK(at, QL.maxit * 32)) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        dst[((at >> 5) * 4 + i) * 32 + (at & 31)] =
            make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
      dpos[at] = (unsigned short)(rp << 8 | q);
    }
    __syncthreads();
  }
  // the last iteration's idle lanes: zero taps
  const int end = (n + 31) & ~31;
  for (int at = n + tid; at < end; at += 256) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
      dst[((at >> 5) * 4 + i) * 32 + (at & 31)] = make_float4(0.f, 0.f, 0.f, 0.f);
    dpos[at] = 0;
  }
  if (tid == 0) cnt[kl] = end >> 5;
}

// Sum over the warp of 32 values per lane, as a reduce-scatter: lane l
// returns the total of value l.
__device__ __forceinline__ float warp_sum32(float (&v)[32]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int h = 16; h >= 1; h >>= 1) {
    const bool up = lane & h;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const float send = up ? v[i] : v[i + h], keep = up ? v[i + h] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, h);
    }
  }
  return v[0];
}

// A block's tile is RQ_X * NG columns x 2 * RQ_W / SPLIT rows; each warp renders
// NG groups side by side, or (SPLIT > 1, NG = 1) SPLIT warps share a group,
// each taking every SPLIT-th iteration of a slice.
//   A quadrant bank's flip classes (select_slice) share the stored slices: a
// class's pixels are rendered with the tile staged mirrored and the local
// pixel order with it (and L and R exchanged when columns are mirrored), one
// class after the other in the few blocks that hold more than one.
template <class TI, int NG, int SPLIT>
__global__ void __launch_bounds__(RQ_W * 32, 2) render_quad_kernel(
    const RenderParams P, QuadLayout QL, const float4* __restrict__ taps,
    const unsigned short* __restrict__ pos, const int* __restrict__ cnt) {
  static_assert(NG == 1 || SPLIT == 1, "split groups come one to a block column");
  constexpr int TW = RQ_X * NG, TH = RQ_R * RQ_W / SPLIT;
  extern __shared__ __align__(16) float tile[];  // [P.halo_h][S]
  __shared__ float s_part[RQ_W][32];
  const int ks = P.ks, p = (ks - 1) >> 1, H = P.H, W = P.W, S = P.halo_w;
  const int x0 = blockIdx.x * TW, y0 = blockIdx.y * TH;
  const int n = blockIdx.z / P.C, c = blockIdx.z - n * P.C;
  const int lam = (P.NL == P.C) ? c : 0;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int row = RQ_R * (warp / SPLIT), sub = warp % SPLIT;  // local row of the group
  const bool two = P.Z > 1;
  const TI* img = reinterpret_cast<const TI*>(P.aif) + ((size_t)n * P.C + c) * H * W;
  const int n_class = P.fmode == SD_FIELD_QUADRANT ? 4 : 1, slices = P.FC * P.Z;
  for (int cls = 0; cls < n_class; ++cls) {
    const bool mx = cls & 1, my = cls & 2;
    // image row / column of a local one
    auto img_y = [&](int l) { return my ? y0 + TH - 1 - l : y0 + l; };
    auto img_x = [&](int l) { return mx ? x0 + TW - 1 - l : x0 + l; };
    // lane l < 16: pixel (l >> 3, l & 7) of every group
    int key[NG];
    float t[NG];
    bool any = false;
#pragma unroll
    for (int g = 0; g < NG; ++g) {
      const int yy = img_y(row + (lane >> 3)), xx = img_x(g * RQ_X + (lane & 7));
      key[g] = -1;
      t[g] = 0.f;
      if (lane < 16 && yy < H && xx < W) {
        select_slice(P, yy, xx, P.depth[((size_t)n * H + yy) * W + xx], &key[g], &t[g]);
        if (n_class > 1) key[g] = key[g] / slices == cls ? key[g] % slices : -1;
      }
      any = any || key[g] >= 0;
    }
    if (n_class > 1 && !__syncthreads_or(any)) continue;
    float zero = 0.f;  // NaN once an infinite or NaN value is staged
    for (int r = warp; r < P.halo_h; r += RQ_W) {
      const TI* src = img + (size_t)min(max(img_y(r - p), 0), H - 1) * W;
      for (int i = lane; i < S; i += 32) {
        const float v = to_f32<TI>(__ldg(&src[min(max(img_x(i - p), 0), W - 1)]));
        zero = fmaf(v, 0.f, zero);
        tile[r * S + i] = v;
      }
    }
    const bool odd = __syncthreads_or(zero != 0.f);
    auto groups = [&](auto masked) {
      for (int g = 0; g < NG; ++g) {
        int kg = key[0];
        float tg = t[0];
#pragma unroll
        for (int i = 1; i < NG; ++i) {
          kg = g == i ? key[i] : kg;
          tg = g == i ? t[i] : tg;
        }
        const float* base = tile + row * S + g * RQ_X;
        float tot = 0.f;  // lane l: side l & 1 of pixel l >> 1
        int last = -1;
        while (true) {
          // the next slice in use: k0 unless t is 1, k0 + 1 if t is not 0
          int cand = 0x7fffffff;
          if (kg >= 0) {
            if ((!two || tg < 1.f) && kg > last) cand = kg;
            else if (two && tg > 0.f && kg + 1 > last) cand = kg + 1;
          }
          const int k = (int)__reduce_min_sync(0xffffffffu, (unsigned)cand);
          if (k == 0x7fffffff) break;
          last = k;
          const float w_l = kg < 0 ? 0.f : kg == k ? (two ? 1.f - tg : 1.f)
                                       : (two && kg + 1 == k) ? tg : 0.f;
          const size_t kl = (size_t)k * P.NL + lam;
          const int iters = __ldg(&cnt[kl]);
          const float4* kt = taps + (kl * QL.maxit + sub) * 128 + lane;
          const unsigned short* kp = pos + (kl * QL.maxit + sub) * 32 + lane;
          float2 acc[16];
#pragma unroll
          for (int j = 0; j < 16; ++j) acc[j] = make_float2(0.f, 0.f);
          // an iteration's item positions are loaded one ahead: the image reads
          // wait for them (8 x 512 x 512 RGB at ks 65 5.15 -> 5.03 ms; the taps
          // ahead as well 5.16)
          int pk_n = sub < iters ? __ldg(kp) : 0;
          for (int it = sub; it < iters; it += SPLIT, kt += 128 * SPLIT, kp += 32 * SPLIT) {
            const int pk = pk_n;
            float4 kv[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) kv[i] = __ldg(kt + 32 * i);
            if (it + SPLIT < iters) pk_n = __ldg(kp + 32 * SPLIT);
            const int off = (pk >> 8) * (2 * S) + (pk & 255) * 4;
            if (!SD_CHECK(row * S + g * RQ_X + off + 2 * S + 11, P.halo_h * S)) continue;
            const float* wp = base + off;
#pragma unroll
            for (int ir = 0; ir < 3; ++ir) {
              float w[12];
#pragma unroll
              for (int i = 0; i < 3; ++i) {
                const float4 q = *reinterpret_cast<const float4*>(wp + ir * S + 4 * i);
                w[4 * i] = q.x;
                w[4 * i + 1] = q.y;
                w[4 * i + 2] = q.z;
                w[4 * i + 3] = q.w;
              }
#pragma unroll
              for (int pr = 0; pr < 2; ++pr) {
                const int tr = ir - pr;  // tap row of pixel row pr
                if (tr < 0 || tr > 1) continue;
#pragma unroll
                for (int tp = 0; tp < 4; ++tp) {
                  const float4 kq = kv[2 * tr + (tp >> 1)];
                  const float2 k2 = (tp & 1) ? make_float2(kq.z, kq.w) : make_float2(kq.x, kq.y);
#pragma unroll
                  for (int j = 0; j < 8; ++j) {
                    const float2 f =
                        __ffma2_rn(make_float2(w[j + tp], w[j + tp]), k2, acc[pr * 8 + j]);
                    if (!decltype(masked)::value) {
                      acc[pr * 8 + j] = f;
                    } else {
                      if (k2.x != 0.f) acc[pr * 8 + j].x = f.x;
                      if (k2.y != 0.f) acc[pr * 8 + j].y = f.y;
                    }
                  }
                }
              }
            }
          }
          float v[32];
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            v[2 * j] = acc[j].x;
            v[2 * j + 1] = acc[j].y;
          }
          const float sum = warp_sum32(v);
          const float w = __shfl_sync(0xffffffffu, w_l, lane >> 1);
          // a pixel that does not use the slice takes nothing of it (not even
          // 0 * inf)
          if (w != 0.f) tot = fmaf(w, sum, tot);
        }
        if (SPLIT > 1) {  // the warps' parts added in order by the first
          s_part[warp][lane] = tot;
          __syncthreads();
          if (sub == 0)
            for (int w = 1; w < SPLIT; ++w) tot += s_part[warp + w][lane];
        }
        const int j = lane >> 1, side = (lane & 1) ^ (mx ? 1 : 0);
        const int yy = img_y(row + (j >> 3)), xx = img_x(g * RQ_X + (j & 7));
        const bool mine = __shfl_sync(0xffffffffu, kg, j) >= 0;
        if (sub == 0 && mine && yy < H && xx < W) {
          TI* out = reinterpret_cast<TI*>(P.out) + ((size_t)n * 2 + side) * P.C * H * W;
          out[((size_t)c * H + yy) * W + xx] = from_f32<TI>(tot);
        }
      }
    };
    // items, and the idle lanes of a last iteration, reach past the kernel with
    // zero taps: over an infinite value those would add NaN
    if (odd) groups(std::true_type{}); else groups(std::false_type{});
    if (n_class > 1) __syncthreads();  // the next class stages the tile again
  }
}

template <class TI, int NG, int SPLIT>
sd_status launch_quad_cfg(RenderParams& P, const QuadLayout& QL, char* ws, cudaStream_t s) {
  constexpr int TW = RQ_X * NG, TH = RQ_R * RQ_W / SPLIT;
  // rows and columns an item's 3 x 12 image values reach
  P.halo_h = TH + (P.ks + 1) / 2 * 2 - 1;
  P.halo_w = TW + 4 * QL.nq;
  const size_t smem = (size_t)P.halo_w * P.halo_h * sizeof(float);
  auto k = render_quad_kernel<TI, NG, SPLIT>;
  SD_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  dim3 grid((P.W + TW - 1) / TW, (P.H + TH - 1) / TH, P.N * P.C);
  k<<<grid, RQ_W * 32, smem, s>>>(P, QL, reinterpret_cast<const float4*>(ws),
                                  reinterpret_cast<const unsigned short*>(ws + QL.tap_bytes),
                                  reinterpret_cast<const int*>(ws + QL.tap_bytes + QL.pos_bytes));
  return launch_status();
}

// groups of 2 x 8 pixels, each rendered by a warp or several
inline long long quad_groups(const RenderParams& P) {
  return (long long)((P.W + RQ_X - 1) / RQ_X) * ((P.H + RQ_R - 1) / RQ_R) * P.N * P.C;
}

// Whether render_fwd_kernel beats the render from a re-laid bank, for a caller
// with the choice.  A warp of the re-laid form pays for a slice by whole
// iterations of 32 items (256 taps) and a reduction of 31 shuffles, so below
// about 17 x 17 taps its time hardly falls with ks, while the direct form's
// does; the direct form needs images of many 128 x 32 tiles, on which few
// slices meet (pixels a slice), and loses least to a quadrant bank, whose
// flip classes the re-laid form selects one after the other.  The largest ks
// at which the direct form wins was measured over banks of discs (16 x 16
// slices, quadrant 8 x 8 x 8; FP16 the same within 3 %), by groups of 2 x 8
// pixels (RGB but where noted; us, direct / re-laid):
//   radial, 512 x 512 gray  ks 5 50 / 53, 7 55 / 53; 512 x 512 ks 9 114 / 130,
//     13 144 / 133; 1024 x 1024 gray ks 15 152 / 162, 21 192 / 190;
//     2048 x 2048 ks 3 805 / 1613, 21 1683 / 1815, 25 1919 / 1863, 65 6256 /
//     4278;
//   quadrant, 512 x 512 gray ks 9 60 / 80, 15 85 / 81; 1024 x 1024 ks 3 210 /
//     661, 21 432 / 712, 33 636 / 816, 51 1016 / 1035; 2048 x 2048 ks 41
//     2775 / 3423, 65 4940 / 4797.
// Denser slices (1024 x 1024 with 32 x 32 of them: even at ks 15) shift it
// down, one slice for the whole image up (1024 x 1024 gray, ks 21: 1.3 times).
//   Both accumulate in FP32, the re-laid form in shorter chains: 4e-8 of the
// result against FP64 at every ks, the direct form 5e-8 at ks 3, 2e-7 at ks 21
// and 3e-7 at ks 41.
inline bool direct_is_faster(const RenderParams& P) {
  const long long g = quad_groups(P), slices = (long long)P.FC * P.Z;
  int k;
  if (P.fmode == SD_FIELD_QUADRANT)
    k = g < 10240    ? 0
        : g < 14336  ? 7
        : g < 32768  ? 9
        : g < 47104  ? 13
        : g < 61440  ? 21
        : g < 90112  ? 29
        : g < 229376 ? 31
                     : 41;
  else
    k = g < 14336    ? 0
        : g < 32768  ? 5
        : g < 53248  ? 9
        : g < 61440  ? 13
        : g < 131072 ? 15
        : g < 229376 ? 17
                     : 21;
  if ((long long)P.H * P.W <= 256 * slices) k -= P.fmode == SD_FIELD_QUADRANT ? 4 : 2;
  if (slices == 1) k = std::max(k, g >= 45056 ? 21 : g >= 2048 ? 7 : 0);
  return P.ks <= k;
}

// the rows of its blocks fit the grid
inline bool quad_fits(const RenderParams& P) { return P.H <= 65535 * RQ_R * RQ_W; }

template <class TI, class TB>
sd_status launch_quad(RenderParams& P, void* workspace, cudaStream_t s) {
  const QuadLayout QL = quad_layout(P);
  char* ws = reinterpret_cast<char*>(workspace);
  unsigned char* use = nullptr;
  if (QL.mark) {
    use = reinterpret_cast<unsigned char*>(ws + QL.tap_bytes + QL.pos_bytes + QL.cnt_bytes);
    SD_CUDA_TRY(cudaMemsetAsync(use, 0, QL.use_bytes, s));
    const size_t blocks = ((size_t)P.N * P.H * P.W + 255) / 256;
    mark_slices_kernel<<<(unsigned)std::min<size_t>(blocks, 2048), 256, 0, s>>>(P, use);
    const sd_status st = launch_status();
    if (st != SD_OK) return st;
  }
  auto k = quad_taps_kernel<TB>;
  const size_t smem = (size_t)2 * P.ks * P.ks * sizeof(float);
  SD_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  k<<<P.FC * P.Z * P.NL, 256, smem, s>>>(
      P, QL, reinterpret_cast<float4*>(ws), reinterpret_cast<unsigned short*>(ws + QL.tap_bytes),
      reinterpret_cast<int*>(ws + QL.tap_bytes + QL.pos_bytes), use);
  const sd_status st = launch_status();
  if (st != SD_OK) return st;
  // groups of 2 x 8 pixels against the 152 x 16 warps the GPU holds: with
  // less than a warp each (a thumbnail) several warps share a group; with many
  // rounds wider blocks stage fewer halo values per pixel.  Measured (us, RGB,
  // split 8 / 4 / one / two / four groups a warp): 64 x 64 gray at ks 65
  // 54 / 60 / 114 / - / -, 128 x 128 168 / 135 / 149 / 163 / 197, 256 x 256
  // 571 / 431 / 364 / 438 / 450, 512 x 512 - / - / 832 / 780 / 868,
  // 1024 x 1024 - / - / 2482 / 2220 / 2137.
  const long long groups = quad_groups(P);
  if (groups < 1024 && QL.maxit >= 8) return launch_quad_cfg<TI, 1, 8>(P, QL, ws, s);
  if (groups < 4096 && QL.maxit >= 4) return launch_quad_cfg<TI, 1, 4>(P, QL, ws, s);
  if (groups < 24576) return launch_quad_cfg<TI, 1, 1>(P, QL, ws, s);
  if (groups < 131072) return launch_quad_cfg<TI, 2, 1>(P, QL, ws, s);
  return launch_quad_cfg<TI, 4, 1>(P, QL, ws, s);
}

constexpr size_t SMEM_CAP = 227 * 1024;

template <class TI, class TB>
sd_status launch_fwd(RenderParams& P, cudaStream_t s) {
  // the widest tile whose block fits in shared memory.  Up to ks = 65 the
  // kernel columns are fetched one at a time: the row extent of non-zero
  // taps is then taken per column (more empty rows skipped) and the smaller
  // tap buffers leave more shared storage to L1; measured 8 % (FP32 bank)
  // to 15 % (BF16 bank) faster at 1024x1024x3 than four columns at a time.
  if (P.ks <= 65 && RenderSmem<128, 1>::bytes(P.ks) <= SMEM_CAP)
    return launch_fwd_cfg<TI, TB, 128, 1, 65>(P, s);
  if (RenderSmem<64, 4>::bytes(P.ks) <= SMEM_CAP) return launch_fwd_cfg<TI, TB, 64, 4, 127>(P, s);
  return launch_fwd_cfg<TI, TB, 64, 2, 127>(P, s);
}

}  // namespace sd

namespace sd {
namespace {

// Argument checks shared by the render entry points; fills P.
sd_status render_args(const sd_bank_layout* layout, int N, int C, int H, int W, RenderParams& P) {
  if (N < 0 || C < 1 || H < 0 || W < 0) return SD_ERR_ARG;
  std::memset(&P, 0, sizeof P);
  P.N = N;
  P.C = C;
  P.H = H;
  P.W = W;
  if (N == 0 || H == 0 || W == 0) return SD_OK;
  if ((long long)N * C > 65535 || (long long)H * W > (1ll << 31)) return SD_ERR_UNSUPPORTED;
  const sd_status st = check_layout(layout, P);
  if (st != SD_OK) return st;
  if (!(P.NL == C || P.NL == 1)) return SD_ERR_ARG;
  // 16-bit relative keys (quadrant keys carry 4 flip classes)
  if ((long long)P.FC * P.Z * (P.fmode == SD_FIELD_QUADRANT ? 4 : 1) > 65000)
    return SD_ERR_UNSUPPORTED;
  return SD_OK;
}

template <class TI, class TB>
sd_status render_typed(RenderParams& P, void* workspace, cudaStream_t s) {
  return workspace && quad_fits(P) ? launch_quad<TI, TB>(P, workspace, s)
                                   : launch_fwd<TI, TB>(P, s);
}

sd_status render(const void* aif, const float* depth_m, const void* bank,
                 const sd_bank_layout* layout, int N, int C, int H, int W, int image_dtype,
                 void* out, void* workspace, size_t workspace_bytes, void* stream) {
  if (!aif || !depth_m || !bank || !out) return SD_ERR_ARG;
  RenderParams P;
  const sd_status st = render_args(layout, N, C, H, W, P);
  if (st != SD_OK || N == 0 || H == 0 || W == 0) return st;
  if (workspace && quad_fits(P) && (workspace_bytes < quad_layout(P).total ||
                                    (reinterpret_cast<uintptr_t>(workspace) & 255)))
    return SD_ERR_ARG;
  P.aif = aif;
  P.depth = depth_m;
  P.bank = bank;
  P.out = out;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const int bt = layout->dtype;
  if (image_dtype == SD_F32 && bt == SD_F32) return render_typed<float, float>(P, workspace, s);
  if (image_dtype == SD_F32 && bt == SD_BF16)
    return render_typed<float, __nv_bfloat16>(P, workspace, s);
  if (image_dtype == SD_BF16 && bt == SD_BF16)
    return render_typed<__nv_bfloat16, __nv_bfloat16>(P, workspace, s);
  if (image_dtype == SD_F16 && bt == SD_F16) return render_typed<__half, __half>(P, workspace, s);
  if (image_dtype == SD_F32 && bt == SD_F16) return render_typed<float, __half>(P, workspace, s);
  return SD_ERR_UNSUPPORTED;
}

}  // namespace
}  // namespace sd

extern "C" {

sd_status sd_dp_render(const void* aif, const float* depth_m, const void* bank,
                       const sd_bank_layout* layout, int N, int C, int H, int W,
                       int image_dtype, void* out, void* stream) {
  SD_API_RANGE("sd_dp_render");
  return sd::render(aif, depth_m, bank, layout, N, C, H, W, image_dtype, out, nullptr, 0, stream);
}

sd_status sd_dp_render_workspace(const sd_bank_layout* layout, int N, int C, int H, int W,
                                 size_t* bytes) {
  using namespace sd;
  if (!bytes) return SD_ERR_ARG;
  RenderParams P;
  const sd_status st = render_args(layout, N, C, H, W, P);
  if (st != SD_OK) return st;
  *bytes = N == 0 || H == 0 || W == 0 || !quad_fits(P) ? 0 : quad_layout(P).total;
  return SD_OK;
}

sd_status sd_dp_render_advised_workspace(const sd_bank_layout* layout, int N, int C, int H,
                                         int W, size_t* bytes) {
  using namespace sd;
  if (!bytes) return SD_ERR_ARG;
  RenderParams P;
  const sd_status st = render_args(layout, N, C, H, W, P);
  if (st != SD_OK) return st;
  *bytes = N == 0 || H == 0 || W == 0 || !quad_fits(P) || direct_is_faster(P)
               ? 0
               : quad_layout(P).total;
  return SD_OK;
}

sd_status sd_dp_render_ws(const void* aif, const float* depth_m, const void* bank,
                          const sd_bank_layout* layout, int N, int C, int H, int W,
                          int image_dtype, void* out, void* workspace, size_t workspace_bytes,
                          void* stream) {
  SD_API_RANGE("sd_dp_render_ws");
  return sd::render(aif, depth_m, bank, layout, N, C, H, W, image_dtype, out, workspace,
                    workspace_bytes, stream);
}

}  // extern "C"

SD_CHECK_TU(render)

// Learned warm start: a 3D convolutional U-Net that predicts the Newton
// update from the residual, ln k, s_w and the previous update, trained on
// systems the simulator solves.  Not part of the paper's method.
//
// Architecture (4 resolution levels, 32 channels, 3x3x3 kernels):
//   c00,c01 | pool | c10,c11 | pool | c20,c21 | pool | c30,c31
//   up, concat [up, skip] -> d20,d21 | up, concat -> d10,d11 | up, concat -> d00,d01 | head h
// conv: Z[v,o] = b[o] + sum_{d in {-1,0,1}^3} sum_c X[v+d, c] W[t(d), o, c]
// (X = 0 outside the grid, t(d) = (dx+1) + 3(dy+1) + 9(dz+1)), ReLU after
// every conv but the head; pool: average of the existing children (coarse
// size ceil(n/2)); up: nearest parent.  Loss 0.5/n sum (Y - T)^2 over the two
// predicted channels.
//
// Data layout: activations are BF16, voxel-major with the channels
// contiguous ([v][C], v = i + nx (j + ny k), the simulator's cell order).
// The network input has 16 channels (8 used; the rest stay zero so every
// contraction is a whole number of 16-wide MMA steps).  Weights: FP32 master
// copy [27][Co][Ci] (+ Adam moments), and two BF16 copies made with every
// update: [27][Co][Ci] for the forward pass and the tap-flipped transpose
// [26-t][Ci][Co] for the data gradient, which is then the same kernel; both
// stored as the core matrices of the MMAs' descriptors (woffs).
//
// Every contraction runs on the tensor cores, BF16 with FP32 accumulation.
// The forward / data-gradient kernel is an implicit GEMM (M = voxels, N =
// output channels, K = 27 taps x input channels) on tcgen05, fed from one
// halo copy per tile (k_conv_tc); k_conv and k_conv_halo are the same
// contraction with mma.sync m16n8k16, in the same order.  The weight-gradient
// kernel contracts over voxels for all layers in one launch, partials reduced
// in a fixed order so results do not depend on scheduling.
#include "common.cuh"
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <algorithm>
#include <cmath>
#include <utility>
#include <memory>
#include <mutex>

typedef __nv_bfloat16 bf16;

namespace nn {

constexpr int NLAYER = 15;
constexpr int CIN_GPU = 16;     // channels of the input feature tensor on the device
constexpr int CIN_USED = 8;     // the network's input channels
constexpr int COUT_HEAD = 8;    // head outputs (the first two are the prediction)
constexpr int NPRED = 2;

struct layer_def { const char *name; int ci, co, relu; };
// ci is the device-side input width (the input layer is padded from 8 to 16)
static const layer_def LAYERS[NLAYER] = {
    {"c00", 16, 32, 1}, {"c01", 32, 32, 1}, {"c10", 32, 32, 1}, {"c11", 32, 32, 1},
    {"c20", 32, 32, 1}, {"c21", 32, 32, 1}, {"c30", 32, 32, 1}, {"c31", 32, 32, 1},
    {"d20", 64, 32, 1}, {"d21", 32, 32, 1}, {"d10", 64, 32, 1}, {"d11", 32, 32, 1},
    {"d00", 64, 32, 1}, {"d01", 32, 32, 1}, {"h", 32, 8, 0}};
enum { C00, C01, C10, C11, C20, C21, C30, C31, D20, D21, D10, D11, D00, D01, HEAD };

static inline int ci_true(int l) { return l == C00 ? CIN_USED : LAYERS[l].ci; }
static inline int cob(int l) { return std::max(16, LAYERS[l].co); }   // data-gradient input width

// ------------------------------------------------------------ PTX helpers -
__device__ __forceinline__ unsigned smem_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void cp_async16(void *dst, const void *src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(smem_u32(dst)), "l"(src), "r"(bytes));
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N> __device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N)); }
__device__ __forceinline__ void ldsm_x4(unsigned r[4], const void *p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(smem_u32(p)));
}
__device__ __forceinline__ void ldsm_x2(unsigned r[2], const void *p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];\n" : "=r"(r[0]), "=r"(r[1]) : "r"(smem_u32(p)));
}
__device__ __forceinline__ void ldsm_x4_t(unsigned r[4], const void *p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(smem_u32(p)));
}
__device__ __forceinline__ void mma16816(float c[4], const unsigned a[4], const unsigned b[2]) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
               "{%0,%1,%2,%3};\n"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// Weight copies: per tap [CO rows][CI], stored as the 8 x 8 core matrices the
// tcgen05 descriptors address (16-byte chunks of 8 inputs; the two chunks of
// a 16-wide K block 128 bytes apart, 8-row groups 256 apart, K blocks CO / 8
// groups apart), so that one bulk copy brings a layer's weights.  Element
// offset of chunk ch of row o (rows padded to 16):
__host__ __device__ constexpr int wrows(int co) { return co < 16 ? 16 : co; }
__host__ __device__ inline int woffs(int rows, int o, int ch) {
  return ((ch >> 1) * (rows / 8) + (o >> 3)) * 128 + (ch & 1) * 64 + (o & 7) * 8;
}

// --------------------------------------------------- implicit-GEMM conv ---
// out[v, o] for v in this CTA's 128 voxels, o < NT*8.
// MODE 0: BF16 out = act(acc + bias)           (forward)
// MODE 1: FP32 out = acc + bias                (head forward)
// MODE 2: BF16 out = acc * (mask[v, o] > 0)    (data gradient through a ReLU)
// MODE 3: BF16 out = acc                       (data gradient, no ReLU below)
constexpr int CBM = 128;    // voxels per CTA (4 warps x 32)
template <int CI, int NT>
struct conv_smem {
  static constexpr int AST = CI + 8, BST = CI + 8, CO = NT * 8;
  static constexpr int A_EL = CBM * AST, B_EL = CO * BST;
  static constexpr int BYTES = 2 * (A_EL + B_EL) * 2;
};

template <int CI, int NT, int MODE>
__global__ void __launch_bounds__(128) k_conv(int nx, int ny, int nz, const bf16 *__restrict__ X, int ldx, int offx,
                                              const bf16 *__restrict__ Wt, const float *__restrict__ bias, int relu,
                                              void *out, int ldo, int offo, const bf16 *__restrict__ mask, int ldm,
                                              int offm) {
  typedef conv_smem<CI, NT> S;
  constexpr int CO = NT * 8, CH = CI / 8;            // 16-byte chunks per input row
  constexpr int AJ = CBM * CH / 128;                  // A chunks per thread and tap
  constexpr int BJ = (CO * CH + 127) / 128;           // B chunks per thread and tap
  extern __shared__ __align__(16) unsigned char smraw[];
  bf16 *sA = reinterpret_cast<bf16 *>(smraw);
  bf16 *sB = sA + 2 * S::A_EL;
  const int V = nx * ny * nz, nxy = nx * ny;
  const int v0 = blockIdx.x * CBM, t = threadIdx.x, lane = t & 31, warp = t >> 5;
  // the voxels whose input rows this thread copies (same for every tap)
  int vx[AJ], vy[AJ], vz[AJ], vrow[AJ], vch[AJ];
#pragma unroll
  for (int j = 0; j < AJ; j++) {
    int q = j * 128 + t;
    vrow[j] = q / CH; vch[j] = q % CH;
    int v = v0 + vrow[j];
    if (v < V) { vz[j] = v / nxy; int r = v - vz[j] * nxy; vy[j] = r / nx; vx[j] = r - vy[j] * nx; }
    else { vx[j] = -1000000; vy[j] = 0; vz[j] = 0; }
  }
  auto load = [&](int stage, int tap) {
    int dx = tap % 3 - 1, dy = (tap / 3) % 3 - 1, dz = tap / 9 - 1;
    bf16 *a = sA + stage * S::A_EL;
#pragma unroll
    for (int j = 0; j < AJ; j++) {
      int x = vx[j] + dx, y = vy[j] + dy, z = vz[j] + dz;
      bool ok = x >= 0 && x < nx && y >= 0 && y < ny && z >= 0 && z < nz;
      const bf16 *src = ok ? X + ((size_t)(x + nx * (y + ny * z)) * ldx + offx + vch[j] * 8) : X;
      cp_async16(a + vrow[j] * S::AST + vch[j] * 8, src, ok ? 16 : 0);
    }
    bf16 *b = sB + stage * S::B_EL;
    const bf16 *w = Wt + (size_t)tap * wrows(CO) * CI;
#pragma unroll
    for (int j = 0; j < BJ; j++) {
      int q = j * 128 + t;
      if (q < CO * CH) {
        int o = q / CH, ch = q % CH;
        cp_async16(b + o * S::BST + ch * 8, w + woffs(wrows(CO), o, ch), 16);
      }
    }
  };
  float acc[2][NT][4];
#pragma unroll
  for (int mt = 0; mt < 2; mt++)
#pragma unroll
    for (int nt = 0; nt < NT; nt++)
#pragma unroll
      for (int e = 0; e < 4; e++) acc[mt][nt][e] = 0.f;

  load(0, 0);
  cp_commit();
  for (int tap = 0; tap < 27; tap++) {
    if (tap + 1 < 27) { load((tap + 1) & 1, tap + 1); cp_commit(); cp_wait<1>(); }
    else cp_wait<0>();
    __syncthreads();
    const bf16 *a = sA + (tap & 1) * S::A_EL;
    const bf16 *b = sB + (tap & 1) * S::B_EL;
#pragma unroll
    for (int ks = 0; ks < CI / 16; ks++) {
      unsigned af[2][4];
#pragma unroll
      for (int mt = 0; mt < 2; mt++)
        ldsm_x4(af[mt], a + (warp * 32 + mt * 16 + (lane & 15)) * S::AST + ks * 16 + (lane >> 4) * 8);
      unsigned bfr[NT][2];
      if constexpr (NT == 1) {
        ldsm_x2(bfr[0], b + (lane & 7) * S::BST + ks * 16 + ((lane >> 3) & 1) * 8);
      } else {
#pragma unroll
        for (int np = 0; np < NT / 2; np++) {
          unsigned r[4];
          ldsm_x4(r, b + (np * 16 + (lane & 7) + ((lane >> 4) << 3)) * S::BST + ks * 16 + ((lane >> 3) & 1) * 8);
          bfr[2 * np][0] = r[0]; bfr[2 * np][1] = r[1];
          bfr[2 * np + 1][0] = r[2]; bfr[2 * np + 1][1] = r[3];
        }
      }
#pragma unroll
      for (int mt = 0; mt < 2; mt++)
#pragma unroll
        for (int nt = 0; nt < NT; nt++) mma16816(acc[mt][nt], af[mt], bfr[nt]);
    }
    __syncthreads();                                  // the stage is reloaded two taps later
  }
  // epilogue
#pragma unroll
  for (int mt = 0; mt < 2; mt++)
#pragma unroll
    for (int hh = 0; hh < 2; hh++) {
      int v = v0 + warp * 32 + mt * 16 + (lane >> 2) + hh * 8;
      if (v >= V) continue;
#pragma unroll
      for (int nt = 0; nt < NT; nt++) {
        int o = nt * 8 + (lane & 3) * 2;
        float y0 = acc[mt][nt][2 * hh], y1 = acc[mt][nt][2 * hh + 1];
        if (MODE == 0 || MODE == 1) { y0 += bias[o]; y1 += bias[o + 1]; }
        if (MODE == 0 && relu) { y0 = fmaxf(y0, 0.f); y1 = fmaxf(y1, 0.f); }
        if (MODE == 2) {
          __nv_bfloat162 m = *reinterpret_cast<const __nv_bfloat162 *>(mask + (size_t)v * ldm + offm + o);
          if (!(__bfloat162float(m.x) > 0.f)) y0 = 0.f;
          if (!(__bfloat162float(m.y) > 0.f)) y1 = 0.f;
        }
        if (MODE == 1) {
          float *op = reinterpret_cast<float *>(out) + (size_t)v * ldo + offo + o;
          op[0] = y0; op[1] = y1;
        } else {
          *reinterpret_cast<__nv_bfloat162 *>(reinterpret_cast<bf16 *>(out) + (size_t)v * ldo + offo + o) =
              __floats2bfloat162_rn(y0, y1);
        }
      }
    }
}

// ------------------------------------------- halo-tiled forward conv ------
// The forward contraction (MODE 0 / 1 of k_conv) with the input read once per
// tile: a CTA owns an 8 x 4 x 4 box of output voxels (row r = x + 8 y + 32 z,
// warp w = z-slice w), stages the 10 x 6 x 6 input halo in shared memory
// (cp.async, zero-filled outside the grid) and, for each of the 27 taps,
// reads its A fragments straight from the halo with per-lane ldmatrix row
// addresses (the shifted voxel of each output row), so only the tap's
// weights stream per tap (two stages).  k_conv gathers 128 shifted rows per
// tap instead, 27 reads of the input per tile.  MMAs are issued in the same
// tap / K order as k_conv.
constexpr int HX = 8, HY = 4, HZ = 4;                         // output box
constexpr int HHX = HX + 2, HHY = HY + 2, HHZ = HZ + 2, HNV = HHX * HHY * HHZ;
template <int CI, int NT>
struct halo_smem {
  static constexpr int AST = CI + 8, BST = CI + 8, CO = NT * 8;
  static constexpr int A_EL = HNV * AST, B_EL = CO * BST;
  static constexpr int BYTES = (A_EL + 2 * B_EL) * 2;
};
template <int CI, int NT, int MODE>
__global__ void __launch_bounds__(128) k_conv_halo(int nx, int ny, int nz, const bf16 *__restrict__ X, int ldx,
                                                   int offx, const bf16 *__restrict__ Wt,
                                                   const float *__restrict__ bias, int relu, void *out, int ldo,
                                                   int offo) {
  typedef halo_smem<CI, NT> S;
  constexpr int CO = NT * 8, CH = CI / 8;
  constexpr int BJ = (CO * CH + 127) / 128;
  extern __shared__ __align__(16) unsigned char smraw[];
  bf16 *sA = reinterpret_cast<bf16 *>(smraw);
  bf16 *sB = sA + S::A_EL;
  const int tx = (nx + HX - 1) / HX, ty = (ny + HY - 1) / HY;
  const int bx = blockIdx.x % tx, by = (blockIdx.x / tx) % ty, bz = blockIdx.x / (tx * ty);
  const int X0 = bx * HX, Y0 = by * HY, Z0 = bz * HZ;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  // the halo: HNV voxels x CH chunks of 16 bytes
  for (int q = t; q < HNV * CH; q += 128) {
    int h = q / CH, ch = q % CH;
    int hx = h % HHX, hy = (h / HHX) % HHY, hz = h / (HHX * HHY);
    int x = X0 + hx - 1, y = Y0 + hy - 1, z = Z0 + hz - 1;
    bool ok = x >= 0 && x < nx && y >= 0 && y < ny && z >= 0 && z < nz;
    const bf16 *src = ok ? X + ((size_t)(x + nx * (y + ny * z)) * ldx + offx + ch * 8) : X;
    cp_async16(sA + h * S::AST + ch * 8, src, ok ? 16 : 0);
  }
  auto loadw = [&](int stage, int tap) {
    bf16 *b = sB + stage * S::B_EL;
    const bf16 *w = Wt + (size_t)tap * wrows(CO) * CI;
#pragma unroll
    for (int j = 0; j < BJ; j++) {
      int q = j * 128 + t;
      if (q < CO * CH) {
        int o = q / CH, ch = q % CH;
        cp_async16(b + o * S::BST + ch * 8, w + woffs(wrows(CO), o, ch), 16);
      }
    }
  };
  loadw(0, 0);
  cp_commit();
  // halo row of output row (warp, mt, lane & 15) at the centre tap
  int hbase[2];
#pragma unroll
  for (int mt = 0; mt < 2; mt++) {
    int r = warp * 32 + mt * 16 + (lane & 15);
    int x = r % HX, y = (r / HX) % HY, z = r / (HX * HY);
    hbase[mt] = (x + 1) + HHX * ((y + 1) + HHY * (z + 1));
  }
  float acc[2][NT][4];
#pragma unroll
  for (int mt = 0; mt < 2; mt++)
#pragma unroll
    for (int nt = 0; nt < NT; nt++)
#pragma unroll
      for (int e = 0; e < 4; e++) acc[mt][nt][e] = 0.f;
  for (int tap = 0; tap < 27; tap++) {
    if (tap + 1 < 27) { loadw((tap + 1) & 1, tap + 1); cp_commit(); cp_wait<1>(); }
    else cp_wait<0>();
    __syncthreads();
    const int dx = tap % 3 - 1, dy = (tap / 3) % 3 - 1, dz = tap / 9 - 1;
    const int shift = dx + HHX * (dy + HHY * dz);
    const bf16 *b = sB + (tap & 1) * S::B_EL;
#pragma unroll
    for (int ks = 0; ks < CI / 16; ks++) {
      unsigned af[2][4];
#pragma unroll
      for (int mt = 0; mt < 2; mt++)
        ldsm_x4(af[mt], sA + (hbase[mt] + shift) * S::AST + ks * 16 + (lane >> 4) * 8);
      unsigned bfr[NT][2];
      if constexpr (NT == 1) {
        ldsm_x2(bfr[0], b + (lane & 7) * S::BST + ks * 16 + ((lane >> 3) & 1) * 8);
      } else {
#pragma unroll
        for (int np = 0; np < NT / 2; np++) {
          unsigned r[4];
          ldsm_x4(r, b + (np * 16 + (lane & 7) + ((lane >> 4) << 3)) * S::BST + ks * 16 + ((lane >> 3) & 1) * 8);
          bfr[2 * np][0] = r[0]; bfr[2 * np][1] = r[1];
          bfr[2 * np + 1][0] = r[2]; bfr[2 * np + 1][1] = r[3];
        }
      }
#pragma unroll
      for (int mt = 0; mt < 2; mt++)
#pragma unroll
        for (int nt = 0; nt < NT; nt++) mma16816(acc[mt][nt], af[mt], bfr[nt]);
    }
    __syncthreads();                                  // the weight stage is reloaded two taps later
  }
#pragma unroll
  for (int mt = 0; mt < 2; mt++)
#pragma unroll
    for (int hh = 0; hh < 2; hh++) {
      int r = warp * 32 + mt * 16 + (lane >> 2) + hh * 8;
      int x = X0 + r % HX, y = Y0 + (r / HX) % HY, z = Z0 + r / (HX * HY);
      if (x >= nx || y >= ny || z >= nz) continue;
      size_t v = (size_t)x + (size_t)nx * (y + (size_t)ny * z);
#pragma unroll
      for (int nt = 0; nt < NT; nt++) {
        int o = nt * 8 + (lane & 3) * 2;
        float y0 = acc[mt][nt][2 * hh] + bias[o], y1 = acc[mt][nt][2 * hh + 1] + bias[o + 1];
        if (MODE == 0 && relu) { y0 = fmaxf(y0, 0.f); y1 = fmaxf(y1, 0.f); }
        if (MODE == 1) {
          float *op = reinterpret_cast<float *>(out) + v * ldo + offo + o;
          op[0] = y0; op[1] = y1;
        } else {
          *reinterpret_cast<__nv_bfloat162 *>(reinterpret_cast<bf16 *>(out) + v * ldo + offo + o) =
              __floats2bfloat162_rn(y0, y1);
        }
      }
    }
}

// ------------------------------------------ implicit-GEMM conv, tcgen05 ---
// The same contraction on the 5th-generation tensor cores, the operands of
// all 27 taps taken from one copy of the input halo in shared memory.  Bound
// by the MMAs' shared-memory reads (M = 128, N = 32, K = 16: 5 KB, 40 cycles
// measured) and, on small grids, by the chain copy -> MMAs -> store.  Under
// ncu with cold caches, 32 -> 32 channels: 65,536 voxels 11.3 us (28 with
// k_conv_halo), 128 voxels 5.9; 64 -> 32 at 136,091 voxels 39 us.
//
// A CTA owns an 8 x 16 x NZ box of output voxels; each z slice is one M = 128
// accumulator of CO columns in TMEM (row r = x + 8 y).  The halo lies in
// planes of 8 channels, [chunk][z][y][x] with 16 bytes per voxel: 8 voxels
// consecutive in x are one core matrix (8 rows x 16 bytes, contiguous) from
// any start, the next 8 rows (y + 1) lie 160 bytes on, the other half of a K
// block one plane on.  So the A operand of a tap is the same memory from a
// shifted start address, and nothing is gathered per tap; a plane's pad
// keeps the copies' writes free of bank conflicts.  The weights of all taps
// come by one bulk copy (they are stored as core matrices), issued before
// the wait for the kernel that makes X.  The ninth warp
// issues a slice's 27 x CI / 16 MMAs, K ascending within each tap as in
// k_conv, once its three halo slices are there; the results are the same bits
// as with mma.sync.  Epilogue, while the next slice is contracted: tcgen05.ld,
// thread = voxel row, bias / ReLU or the data-gradient mask.  Every wait is
// bounded; on a timeout the kernel records an error and writes nothing.
__device__ __forceinline__ uint64_t tc_desc(unsigned saddr, unsigned lbo, unsigned sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);
  d |= (uint64_t)(lbo >> 4) << 16;             // K-major: K halves of a block; MN-major: next 8 of K
  d |= (uint64_t)(sbo >> 4) << 32;             // next 8 rows (K-major) or 8 of M / N (MN-major)
  d |= (uint64_t)1 << 46;                      // descriptor version; no swizzle, base offset 0
  return d;
}
// BF16 x BF16 -> FP32, M = 128, N = n; MN-major operands when mn
__device__ __forceinline__ uint32_t tc_idesc(int n, bool mn) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (mn ? 3u << 15 : 0u) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}
// MMAs are issued by a whole warp with one elected lane's predicate on the
// instruction only: the descriptors then stay in uniform registers, while in
// a branch of one thread each MMA cost 80 to 170 cycles to issue.
__device__ __forceinline__ uint32_t elect_one() {
  uint32_t e;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(e));
  return e;
}
__device__ __forceinline__ void tc_mma(uint32_t e, uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile("{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n"
               " @q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
               ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(acc), "r"(e) : "memory");
}
__device__ __forceinline__ void tc_commit(uint32_t e, uint64_t *bar) {
  asm volatile("{\n .reg .pred q;\n setp.ne.b32 q, %1, 0;\n"
               " @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n"
               ::"r"(smem_u32(bar)), "r"(e) : "memory");
}
__device__ __forceinline__ void bar_init(uint64_t *bar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void bar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// whole warp: allocate ncol TMEM columns (a power of two, at least 32)
__device__ __forceinline__ void tc_alloc(uint32_t *slot, int ncol) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(ncol) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tc_free(uint32_t taddr, int ncol) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncol) : "memory");
}
__device__ __forceinline__ void tc_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ bool tc_wait(uint64_t *bar, unsigned parity) {
  for (int it = 0; it < (1 << 24); it++) {
    unsigned ok;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    if (ok) return true;
  }
  return false;
}
__device__ __forceinline__ void tc_ld32(uint32_t taddr, float *v) {
  uint32_t r[32];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
               "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                 "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
                 "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
                 "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
               : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int c = 0; c < 32; c++) v[c] = __uint_as_float(r[c]);
}

__device__ __forceinline__ void tc_ld8(uint32_t taddr, float *v) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int c = 0; c < 8; c++) v[c] = __uint_as_float(r[c]);
}
__device__ __forceinline__ void tc_ld16(uint32_t taddr, float *v) {
  uint32_t r[16];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                 "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
               : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int c = 0; c < 16; c++) v[c] = __uint_as_float(r[c]);
}

constexpr int TBX = 8, TBY = 16, THX = TBX + 2, THY = TBY + 2, TSL = THX * THY;   // box, halo, halo voxels per slice
__host__ __device__ constexpr int tc_plane(int ci, int nz) {                      // bytes of an 8-channel plane
  return (TSL * (nz + 2) * 16 + 127) / 128 * 128 + 1024 / ci;
}
__host__ __device__ constexpr int tc_bytes(int ci, int co, int nz) { return 27 * ci * co * 2 + ci / 8 * tc_plane(ci, nz); }
__host__ __device__ constexpr int tc_cols(int co, int nz) {                       // TMEM columns to allocate
  int n = 32;
  while (n < co * nz) n *= 2;
  return n;
}

// MODE as for k_conv: 0 forward (bias, ReLU flag), 1 head forward (FP32, 8 of
// the 16 columns), 2 data gradient with mask, 3 data gradient.
constexpr int TC_T = 288;                              // 8 warps copy and store, the ninth issues the MMAs
template <int CI, int CO, int MODE>
__global__ void __launch_bounds__(TC_T) k_conv_tc(int nx, int ny, int nz, int NZ, const bf16 *X, int ldx, int offx,
                                                 const bf16 *Wt, const float *bias, int relu, void *out, int ldo,
                                                 int offo, const bf16 *mask, int ldm, int offm, int *err) {
  constexpr int CH = CI / 8, W_BYTES = 27 * CI * CO * 2;
  extern __shared__ __align__(128) unsigned char smtc[];
  __shared__ uint64_t wbar, full[4], done[4];           // weights; halo of slice z complete; its MMAs complete
  __shared__ uint32_t tslot;
  __shared__ float sbias[32];
  unsigned char *sA = smtc + W_BYTES;
  const int plane = tc_plane(CI, NZ), ncol = tc_cols(CO, NZ);
  const int tx = (nx + TBX - 1) / TBX, ty = (ny + TBY - 1) / TBY;
  const int X0 = (int)(blockIdx.x % tx) * TBX, Y0 = (int)(blockIdx.x / tx % ty) * TBY, Z0 = (int)(blockIdx.x / (tx * ty)) * NZ;
  const int t = threadIdx.x, warp = __shfl_sync(0xffffffffu, t >> 5, 0);
  if (MODE <= 1 && t < (MODE == 1 ? 8 : 32)) sbias[t] = bias[t];
  if (t == 0) {
    bar_init(&wbar, 1);
    for (int z = 0; z < 4; z++) { bar_init(&full[z], 256); bar_init(&done[z], 1); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) tc_alloc(&tslot, ncol);
  tc_before();
  __syncthreads();
  tc_after();
  const uint32_t taddr = tslot;
  // the next kernel may start only now: every CTA of this one has its TMEM,
  // so CTAs of the next that hold theirs cannot keep this one from finishing
  pdl_trigger();
  if (t == 0) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(&wbar)), "n"(W_BYTES) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(smtc)), "l"(Wt), "n"(W_BYTES), "r"(smem_u32(&wbar)) : "memory");
  }
  const int nzv = min(NZ, nz - Z0);
  bool ok = true;
  if (warp == 8) {
    ok = tc_wait(&wbar, 0);
    const uint32_t idesc = tc_idesc(CO, false), e = elect_one();
    const uint64_t da0 = tc_desc(smem_u32(sA), plane, THX * 16), db0 = tc_desc(smem_u32(smtc), 128, 256);
    const int kstep = plane >> 3;                      // two planes, in 16-byte units
    for (int z = 0; z < nzv && ok; z++) {
      ok = tc_wait(&full[z], 0);
      if (!ok) break;
      tc_after();
      uint64_t da = da0 + z * TSL, db = db0;
      uint32_t acc = 0;
#pragma unroll 1
      for (int ryz = 0; ryz < 9; ryz++) {              // (dy, dz)
#pragma unroll
        for (int dx = 0; dx < 3; dx++)
#pragma unroll
          for (int kb = 0; kb < CI / 16; kb++) {
            tc_mma(e, taddr + z * CO, da + dx + kb * kstep, db, idesc, acc);
            acc = 1;
            db += CO * 2;                              // CO / 8 groups of 256 bytes
          }
        da += ryz % 3 == 2 ? TSL - 2 * THX : THX;
      }
      tc_commit(e, &done[z]);
    }
  } else {
    pdl_wait();
    // thread: chunk ch of voxels h, h + DH, ... of the halo, coordinates
    // carried along; slice z's MMAs can start when z + 3 halo slices are there
    constexpr int DH = 256 / CH, DX = DH % THX, DY = DH / THX;
    const int ch = t % CH;
    int h = t / CH, hx = h % THX, hy = h / THX, hz = 0;
    const bf16 *Xc = X + offx + ch * 8;
    unsigned char *dst = sA + ch * plane;
    for (int g = 0; g < nzv; g++) {
      for (; h < TSL * (3 + g); h += DH) {
        const int x = X0 + hx - 1, y = Y0 + hy - 1, z = Z0 + hz - 1;
        const bool in = x >= 0 && x < nx && y >= 0 && y < ny && z >= 0 && z < nz;
        cp_async16(dst + h * 16, in ? Xc + ((size_t)x + (size_t)nx * (y + (size_t)ny * z)) * ldx : X, in ? 16 : 0);
        hx += DX; hy += DY;
        if (hx >= THX) { hx -= THX; hy++; }
        if (hy >= THY) { hy -= THY; hz++; }
      }
      cp_commit();
    }
    const int r = (warp & 3) * 32 + (t & 31), x = X0 + r % TBX, y = Y0 + r / TBX;
    const bool live = x < nx && y < ny;
    [[maybe_unused]] uint4 mk[CO / 8];                 // the mask of this thread's next voxel, ahead of the MMAs
    auto load_mask = [&](int z) {
      if (MODE == 2 && live && z < nzv) {
        const uint4 *p = reinterpret_cast<const uint4 *>(mask + ((size_t)x + (size_t)nx * (y + (size_t)ny * (Z0 + z))) * ldm + offm);
#pragma unroll
        for (int u = 0; u < CO / 8; u++) mk[u] = p[u];
      }
    };
    load_mask(warp >> 2);
    for (int g = 0; g < nzv; g++) {
      const int pending = nzv - 1 - g;
      if (pending == 3) cp_wait<3>();
      else if (pending == 2) cp_wait<2>();
      else if (pending == 1) cp_wait<1>();
      else cp_wait<0>();
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      bar_arrive(&full[g]);
    }
    for (int z = warp >> 2; z < nzv; z += 2) {
      ok = tc_wait(&done[z], 0);
      if (!ok) break;
      tc_after();
      const size_t v = (size_t)x + (size_t)nx * (y + (size_t)ny * (Z0 + z));
      const uint32_t ta = taddr + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(z * CO);
      if constexpr (MODE == 1) {
        float acc[8];
        tc_ld8(ta, acc);
        if (live) {
          float *op = reinterpret_cast<float *>(out) + v * ldo + offo;
#pragma unroll
          for (int c = 0; c < 8; c++) acc[c] += sbias[c];
          reinterpret_cast<float4 *>(op)[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
          reinterpret_cast<float4 *>(op)[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
        }
      } else {
#pragma unroll
        for (int c0 = 0; c0 < CO; c0 += 32) {
          float acc[32];
          tc_ld32(ta + (uint32_t)c0, acc);
          if (live) {
            if (MODE == 0) {
#pragma unroll
              for (int c = 0; c < 32; c++) { acc[c] += sbias[c0 + c]; if (relu) acc[c] = fmaxf(acc[c], 0.f); }
            } else if (MODE == 2) {
#pragma unroll
              for (int u = 0; u < 4; u++) {
                const bf16 *m = reinterpret_cast<const bf16 *>(&mk[c0 / 8 + u]);
#pragma unroll
                for (int c = 0; c < 8; c++) if (!(__bfloat162float(m[c]) > 0.f)) acc[8 * u + c] = 0.f;
              }
            }
            uint4 pk[4];
            __nv_bfloat162 *h2 = reinterpret_cast<__nv_bfloat162 *>(pk);
#pragma unroll
            for (int c = 0; c < 16; c++) h2[c] = __floats2bfloat162_rn(acc[2 * c], acc[2 * c + 1]);
            uint4 *dst = reinterpret_cast<uint4 *>(reinterpret_cast<bf16 *>(out) + v * ldo + offo + c0);
#pragma unroll
            for (int u = 0; u < 4; u++) dst[u] = pk[u];
          }
        }
        load_mask(z + 2);
      }
    }
  }
  if (!ok) *(volatile int *)err = 1;
  tc_before();
  __syncthreads();
  if (warp == 0) tc_free(taddr, ncol);
}

// ------------------------------------------------------ weight gradient ---
// part[tap][chunk][o][c] = sum over the chunk's voxels u of dZ[u - d(tap), o] X[u, c],
// and bpart[chunk][o] = sum_u dZ[u, o], of all layers in one launch.
//
// On tcgen05 with the voxels as K: M = 128 rows are four x shifts of 32 input
// channels (three used), N three z shifts of the output channels, one
// accumulator per dy; so an MMA reads 7 KB of shared memory (which bounds it:
// 56 cycles) for three taps in z, where one per dz would read 15.  A CTA owns
// a range of X slices (8 x 16 voxels of one z, z fastest) and 32 of the input
// channels.  Both operands are MN-major core matrices (8 channels of 16
// bytes, 8 voxels consecutive in y).  X lies as [x][chunk][y] with a halo of
// one, so that the channel groups of x - 1, x, x + 1 follow each other at one
// stride and dy is a shift of the start by 16 bytes.  dZ lies as
// [x][slot][chunk][y] in a ring of six z slices, the first two slots held
// twice, so that three consecutive slices are always adjacent.  One MMA
// contracts the 16 voxels of an x column.
//
// Step i brings dZ slice z and X slice z - 1 and then contracts the latter
// with dZ slices z - 2, z - 1, z (zero outside the grid); two steps at the
// start of a column only load.  Eight warps copy two steps ahead, the ninth
// issues the MMAs; after WFL slices (64 MMAs on an accumulator) all twelve
// move the sums to FP32 registers, one z shift per four warps, so that the
// tensor cores' accumulation chains stay short.  One CTA per SM (TMEM and
// registers).  All 15 layers of a 64x64x16 grid: 59 us, where a launch per
// layer with mma.sync and its reduction took 507.
constexpr int WYP = THY + 1, WYB = TBY + 1;                      // y pitches, odd: copies free of bank conflicts
constexpr int WR = 6, WSLOT = WR + 2;                            // dZ ring: slots, with the two copies
constexpr int WA_BYTES = 11 * 4 * WYP * 16 + 64, WNS = 4, WLA = 2, WFL = 8;
constexpr int WB_OFF = WNS * WA_BYTES, WG_BYTES = WB_OFF + TBX * (WSLOT * 4 * WYB + 4) * 16;
struct wg_layer {
  const bf16 *X, *dZ;
  float *part, *bpart;
  int ldx, offx, ldz, nx, ny, nz, co, ci, nchunk, block0;
};
struct wg_table { wg_layer l[NLAYER]; };
// the steps of X slices s, s + 1, ... (col nz + z): zz runs from za - 1 to zb in each column
struct wg_steps {
  int col, za, zb, zz, left;
  __device__ void start(long long s, int n, int nz) {
    col = (int)(s / nz); za = (int)(s % nz); zb = min(nz, za + n); zz = za - 1; left = n - (zb - za);
  }
  __device__ void next(int nz) {
    if (++zz > zb && left > 0) { col++; za = 0; zb = min(nz, left); left -= zb; zz = -1; }
  }
};

constexpr int WG_T = 384;
__global__ void __launch_bounds__(WG_T, 1) k_conv_wgrad(const __grid_constant__ wg_table tab, int *err) {
  extern __shared__ __align__(128) unsigned char smtc[];
  __shared__ uint64_t bar[WNS];
  __shared__ uint32_t tslot;
  const int t = threadIdx.x, warp = __shfl_sync(0xffffffffu, t >> 5, 0);
  int li = 0;
  while (li + 1 < NLAYER && (int)blockIdx.x >= tab.l[li + 1].block0) li++;
  const wg_layer &L = tab.l[li];
  const int nx = L.nx, ny = L.ny, nz = L.nz, co = L.co, ci = L.ci, nchunk = L.nchunk, lb = (int)blockIdx.x - L.block0;
  const int chunk = lb % nchunk, half = lb / nchunk;
  const int lch = ci == 16 ? 1 : 2, chn = 1 << lch;              // 16-byte chunks of input channels
  const int lno = co <= 16 ? 1 : 2, no = 8 << lno;               // output channels (padded) and their chunks
  const int xsb = (WSLOT << lno) * WYB + 4;                      // x stride of dZ (16-byte units)
  if (t == 0) {
    for (int k = 0; k < WNS; k++) bar_init(&bar[k], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tc_alloc(&tslot, 512);
  tc_before();
  __syncthreads();
  tc_after();
  pdl_trigger();
  pdl_wait();
  const uint32_t taddr = tslot, idesc = tc_idesc(3 * no, true);
  const int tx = (nx + TBX - 1) / TBX, ty = (ny + TBY - 1) / TBY;
  const long long S = (long long)tx * ty * nz, s0 = S * chunk / nchunk, s1 = S * (chunk + 1) / nchunk;
  const int n = (int)(s1 - s0);                                  // at least 1: nchunk <= S
  const int nstep = n + 2 * (int)((s1 - 1) / nz - s0 / nz + 1);
  const bf16 *X = L.X + L.offx + half * 32, *dZ = L.dZ;
  const int ldx = L.ldx, ldz = L.ldz;
  bool ok = true;
  // the chunks this thread copies of every slice: voxel in the box and offset
  // in shared memory (X: up to three, dZ: up to two)
  int xh[3], yh[3], xo[3], xz[2], yz[2], zo[2];
#pragma unroll
  for (int k = 0; k < 3; k++) {
    const int q = t + 256 * k, ch = q & (chn - 1), h = q >> lch;
    xh[k] = h % THX - 1; yh[k] = h / THX - 1;
    xo[k] = t < 256 && h < TSL ? ((((xh[k] + 1) << lch) + ch) * WYP + yh[k] + 1) * 16 : -1;
  }
  const int xch = (t & (chn - 1)) * 8, zch = (t & ((1 << lno) - 1)) * 8;
#pragma unroll
  for (int k = 0; k < 2; k++) {
    const int q = t + 256 * k, ch = q & ((1 << lno) - 1), h = q >> lno;
    xz[k] = h % TBX; yz[k] = h / TBX;
    zo[k] = t < 256 && h < TBX * TBY ? WB_OFF + (xz[k] * xsb + ch * WYB + yz[k]) * 16 : -1;
  }
  wg_steps ls, ms;                                               // the copies' and the MMAs' steps
  ls.start(s0, n, nz);
  ms = ls;
  int lx = ls.col % tx * TBX, ly = ls.col / tx * TBY;
  auto load = [&](int u) {
    // the slot and the stage were last read by the MMAs of step u - 4
    if (u >= WNS) ok = ok && tc_wait(&bar[u % WNS], (unsigned)((u / WNS - 1) & 1));
    const int slot = u % WR;
    const bool zin = ls.zz >= 0 && ls.zz < nz;
    const size_t zz = (size_t)ny * ls.zz, zx = (size_t)ny * (ls.zz - 1);
#pragma unroll
    for (int k = 0; k < 2; k++)
      if (zo[k] >= 0) {
        const int x = lx + xz[k], y = ly + yz[k];
        const bool in = zin && x < nx && y < ny;
        const bf16 *src = in ? dZ + (x + nx * (y + zz)) * ldz + zch : dZ;
        unsigned char *d = smtc + zo[k] + (slot << lno) * WYB * 16;
        cp_async16(d, src, in ? 16 : 0);
        if (slot < 2) cp_async16(d + (WR << lno) * WYB * 16, src, in ? 16 : 0);
      }
    if (ls.zz - 1 >= ls.za) {
      unsigned char *a = smtc + u % WNS * WA_BYTES;
#pragma unroll
      for (int k = 0; k < 3; k++)
        if (xo[k] >= 0) {
          const int x = lx + xh[k], y = ly + yh[k];
          const bool in = x >= 0 && x < nx && y >= 0 && y < ny;
          cp_async16(a + xo[k], in ? X + (x + nx * (y + zx)) * ldx + xch : X, in ? 16 : 0);
        }
    }
    const int col = ls.col;
    ls.next(nz);
    if (ls.col != col) { lx += TBX; if (lx >= nx) { lx = 0; ly += TBY; } }
  };
  float sum[3][32], bsum[8];                                     // dy, output channel; z shift warp / 4
#pragma unroll
  for (int d = 0; d < 3; d++)
#pragma unroll
    for (int j = 0; j < 32; j++) sum[d][j] = 0.f;
#pragma unroll
  for (int j = 0; j < 8; j++) bsum[j] = 0.f;
  const uint32_t e = elect_one();
  int done = 0;                                                  // X slices contracted
#pragma unroll 1
  for (int u = 0; u < WLA; u++) { if (warp < 8) load(u); cp_commit(); }   // (nstep >= 3)
#pragma unroll 1
  for (int i = 0; i < nstep; i++) {
    if (warp < 8 && i + WLA < nstep) load(i + WLA);
    cp_commit();
    cp_wait<WLA>();
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    ok = __syncthreads_and(ok);
    if (!ok) break;
    const bool work = ms.zz - 1 >= ms.za;
    ms.next(nz);
    if (warp == 8) {
      if (work) {
        tc_after();
        const uint64_t da = tc_desc(smem_u32(smtc + i % WNS * WA_BYTES), 128, WYP * 16),
                       db = tc_desc(smem_u32(smtc + WB_OFF + ((i - 2) % WR << lno) * WYB * 16), 128, WYB * 16);
        const int ax = WYP << lch;
#pragma unroll
        for (int x = 0; x < TBX; x++)
#pragma unroll
          for (int dy = 0; dy < 3; dy++)
            tc_mma(e, taddr + dy * 96, da + x * ax + dy, db + x * xsb, idesc, x > 0 || done % WFL > 0);
      }
      tc_commit(e, &bar[i % WNS]);
    } else if (warp < 8 && work && half == 0) {                  // bias: the middle one of the three slices
      const unsigned char *b = smtc + WB_OFF + ((i - 1) % WR << lno) * WYB * 16;
#pragma unroll
      for (int k = 0; k < 2; k++) {
        const int u = t + 256 * k, g = u >> 4;
        if (g < TBX << lno) {
          const uint4 v = *reinterpret_cast<const uint4 *>(b + ((g >> lno) * xsb + (g & ((1 << lno) - 1)) * WYB + (u & 15)) * 16);
          const bf16 *p = reinterpret_cast<const bf16 *>(&v);
#pragma unroll
          for (int j = 0; j < 8; j++) bsum[j] += __bfloat162float(p[j]);
        }
      }
    }
    if (!work) continue;
    done++;
    if (done % WFL == 0 || done == n) {
      ok = __syncthreads_and(tc_wait(&bar[i % WNS], (unsigned)((i / WNS) & 1)));
      if (!ok) break;
      tc_after();
#pragma unroll
      for (int d = 0; d < 3; d++)
#pragma unroll
        for (int k = 0; k < 2; k++)
          if (k < lno) {
            float v[16];
            tc_ld16(taddr + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(d * 96 + (warp >> 2) * no + 16 * k), v);
#pragma unroll
            for (int j = 0; j < 16; j++) sum[d][16 * k + j] += v[j];
          }
      tc_before();
      __syncthreads();
    }
  }
  if (ok) {
    const int m = (warp & 3) * 32 + (t & 31), dx = m >> (lch + 3), c = half * 32 + (m & (8 * chn - 1));
    if (dx < 3)
#pragma unroll
      for (int d = 0; d < 3; d++) {
        const int dz = 2 - (warp >> 2);                // of dZ slice z - 1 + warp / 4
        float *dst = L.part + ((size_t)(dx + 3 * d + 9 * dz) * nchunk + chunk) * co * ci + c;
#pragma unroll
        for (int o = 0; o < 32; o++)
          if (o < co) dst[(size_t)o * ci] = sum[d][o];
      }
    if (half == 0) {                                   // (the last MMAs are done: the stages are free)
      float *bred = reinterpret_cast<float *>(smtc);
      __syncthreads();
      if (warp < 8)
#pragma unroll
        for (int j = 0; j < 8; j++) bred[t * 8 + j] = bsum[j];
      __syncthreads();
      if (t < co) {
        float s = 0.f;
        for (int k = 0; k < 256; k++)
          if (((k >> 4) & ((1 << lno) - 1)) == t >> 3) s += bred[k * 8 + (t & 7)];
        L.bpart[(size_t)chunk * co + t] = s;
      }
    }
  } else if (t == 0) {
    *(volatile int *)err = 1;
  }
  tc_before();
  __syncthreads();
  if (warp == 0) tc_free(taddr, 512);
}

// G += sums over the chunks (in order) of all layers' partials, G in the flat
// parameter order (a layer's weights, then its biases); the last block adds
// the loss (see k_sum_parts)
__device__ __forceinline__ void sum_parts(int n, const float *part, double scale, double *out, int accumulate) {
  double t = 0.0;
  for (int k = threadIdx.x; k < n; k += 32) t += (double)part[k];
  for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
  if (threadIdx.x == 0) out[0] = (accumulate ? out[0] : 0.0) + scale * t;
}
__global__ void __launch_bounds__(256) k_wgrad_reduce(const __grid_constant__ wg_table tab, int np, float *G, int nl,
                                                      const float *lpart, double lscale, double *lsum) {
  pdl_trigger();
  pdl_wait();
  if (blockIdx.x == gridDim.x - 1) {
    if (threadIdx.x < 32) sum_parts(nl, lpart, lscale, lsum, 1);
    return;
  }
  const int q = blockIdx.x * 256 + threadIdx.x;
  if (q >= np) return;
  int r = q, l = 0;
  for (; l < NLAYER - 1; l++) {
    const int sz = 27 * tab.l[l].co * tab.l[l].ci + tab.l[l].co;
    if (r < sz) break;
    r -= sz;
  }
  const wg_layer &L = tab.l[l];
  const int per = L.co * L.ci, nc = L.nchunk;
  const float *p;
  size_t st;
  if (r < 27 * per) { p = L.part + (size_t)(r / per) * nc * per + r % per; st = per; }
  else { p = L.bpart + (r - 27 * per); st = L.co; }
  float s = 0.f;
  for (int c0 = 0; c0 < nc; c0 += 8) {
    float v[8];
#pragma unroll
    for (int u = 0; u < 8; u++) v[u] = c0 + u < nc ? p[(c0 + u) * st] : 0.f;
#pragma unroll
    for (int u = 0; u < 8; u++) if (c0 + u < nc) s += v[u];
  }
  G[q] += s;
}

// ------------------------------------------------------- pool and up ------
struct dims { int nx, ny, nz; __host__ __device__ int V() const { return nx * ny * nz; } };
__host__ __device__ inline dims coarse(dims d) { return {(d.nx + 1) / 2, (d.ny + 1) / 2, (d.nz + 1) / 2}; }

// P[V, c] = mean of the existing children, 32 channels, 8 per thread
__global__ void k_pool(dims f, dims c, const bf16 *X, int ldx, int offx, bf16 *P) {
  pdl_trigger();
  pdl_wait();
  int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= c.V() * 4) return;
  int V = q >> 2, g = (q & 3) * 8;
  int Z = V / (c.nx * c.ny), r = V - Z * c.nx * c.ny, Y = r / c.nx, Xc = r - Y * c.nx;
  float s[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  int cnt = 0;
  uint4 u[8];                                          // the children's loads together, then the sums in order
  bool in[8];
#pragma unroll
  for (int k = 0; k < 8; k++) {
    int x = 2 * Xc + (k & 1), y = 2 * Y + (k >> 1 & 1), z = 2 * Z + (k >> 2);
    in[k] = x < f.nx && y < f.ny && z < f.nz;
    if (in[k]) u[k] = *reinterpret_cast<const uint4 *>(X + (size_t)(x + f.nx * (y + f.ny * z)) * ldx + offx + g);
  }
#pragma unroll
  for (int k = 0; k < 8; k++)
    if (in[k]) {
      const bf16 *e = reinterpret_cast<const bf16 *>(&u[k]);
#pragma unroll
      for (int a = 0; a < 8; a++) s[a] += __bfloat162float(e[a]);
      cnt++;
    }
  uint4 o;
  bf16 *e = reinterpret_cast<bf16 *>(&o);
#pragma unroll
  for (int a = 0; a < 8; a++) e[a] = __float2bfloat16_rn(s[a] / (float)cnt);
  *reinterpret_cast<uint4 *>(P + (size_t)V * 32 + g) = o;
}

// out[v, off + c] = C[parent(v), c], 32 channels
__global__ void k_up(dims f, dims c, const bf16 *C, bf16 *out, int ldo, int offo) {
  pdl_trigger();
  pdl_wait();
  int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= f.V() * 4) return;
  int v = q >> 2, g = (q & 3) * 8;
  int z = v / (f.nx * f.ny), r = v - z * f.nx * f.ny, y = r / f.nx, x = r - y * f.nx;
  int P = (x >> 1) + c.nx * ((y >> 1) + c.ny * (z >> 1));
  *reinterpret_cast<uint4 *>(out + (size_t)v * ldo + offo + g) = *reinterpret_cast<const uint4 *>(C + (size_t)P * 32 + g);
}

// dC[V, c] = sum over children of G[v, offg + c]  (32 channels)
__global__ void k_up_back(dims f, dims c, const bf16 *G, int ldg, int offg, bf16 *dC) {
  pdl_trigger();
  pdl_wait();
  int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= c.V() * 4) return;
  int V = q >> 2, g = (q & 3) * 8;
  int Z = V / (c.nx * c.ny), r = V - Z * c.nx * c.ny, Y = r / c.nx, Xc = r - Y * c.nx;
  float s[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  uint4 u[8];
  bool in[8];
#pragma unroll
  for (int k = 0; k < 8; k++) {
    int x = 2 * Xc + (k & 1), y = 2 * Y + (k >> 1 & 1), z = 2 * Z + (k >> 2);
    in[k] = x < f.nx && y < f.ny && z < f.nz;
    if (in[k]) u[k] = *reinterpret_cast<const uint4 *>(G + (size_t)(x + f.nx * (y + f.ny * z)) * ldg + offg + g);
  }
#pragma unroll
  for (int k = 0; k < 8; k++)
    if (in[k]) {
      const bf16 *e = reinterpret_cast<const bf16 *>(&u[k]);
#pragma unroll
      for (int a = 0; a < 8; a++) s[a] += __bfloat162float(e[a]);
    }
  uint4 o;
  bf16 *e = reinterpret_cast<bf16 *>(&o);
#pragma unroll
  for (int a = 0; a < 8; a++) e[a] = __float2bfloat16_rn(s[a]);
  *reinterpret_cast<uint4 *>(dC + (size_t)V * 32 + g) = o;
}

// dE[v, c] = (S[v, offs + c] + dP[parent, c] / children(parent)) * (E[v, offe + c] > 0)
// (the skip gradient, already masked, plus the pooled path's gradient)
__global__ void k_pool_back(dims f, dims c, const bf16 *dP, const bf16 *S, int lds, int offs, const bf16 *E, int lde,
                            int offe, bf16 *dE) {
  pdl_trigger();
  pdl_wait();
  int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= f.V() * 4) return;
  int v = q >> 2, g = (q & 3) * 8;
  int z = v / (f.nx * f.ny), r = v - z * f.nx * f.ny, y = r / f.nx, x = r - y * f.nx;
  int X = x >> 1, Y = y >> 1, Z = z >> 1;
  int cnt = (min(f.nx, 2 * X + 2) - 2 * X) * (min(f.ny, 2 * Y + 2) - 2 * Y) * (min(f.nz, 2 * Z + 2) - 2 * Z);
  uint4 up = *reinterpret_cast<const uint4 *>(dP + (size_t)(X + c.nx * (Y + c.ny * Z)) * 32 + g);
  uint4 us = *reinterpret_cast<const uint4 *>(S + (size_t)v * lds + offs + g);
  uint4 ue = *reinterpret_cast<const uint4 *>(E + (size_t)v * lde + offe + g);
  const bf16 *ep = reinterpret_cast<const bf16 *>(&up), *es = reinterpret_cast<const bf16 *>(&us),
             *ee = reinterpret_cast<const bf16 *>(&ue);
  uint4 o;
  bf16 *eo = reinterpret_cast<bf16 *>(&o);
#pragma unroll
  for (int a = 0; a < 8; a++) {
    float val = __bfloat162float(es[a]) + __bfloat162float(ep[a]) / (float)cnt;
    eo[a] = __float2bfloat16_rn(__bfloat162float(ee[a]) > 0.f ? val : 0.f);
  }
  *reinterpret_cast<uint4 *>(dE + (size_t)v * 32 + g) = o;
}

// ---------------------------------------------------------- loss, Adam ----
// dY[v, c] = (Y[v, c] - T[v, c]) / V for c < 2, 0 for the other 14 channels;
// part[block] = sum of the block's squared errors
__global__ void k_loss(int V, const float *Y, const float *T, bf16 *dY, float *part) {
  pdl_trigger();
  pdl_wait();
  __shared__ float sh[256];
  int v = blockIdx.x * blockDim.x + threadIdx.x;
  float s = 0.f;
  if (v < V) {
    float e0 = Y[(size_t)v * COUT_HEAD] - T[2 * (size_t)v], e1 = Y[(size_t)v * COUT_HEAD + 1] - T[2 * (size_t)v + 1];
    s = e0 * e0 + e1 * e1;
    float inv = 1.0f / (float)V;
    uint4 z0 = make_uint4(0, 0, 0, 0);
    uint4 *d = reinterpret_cast<uint4 *>(dY + (size_t)v * 16);
    __nv_bfloat162 g = __floats2bfloat162_rn(e0 * inv, e1 * inv);
    uint4 first = z0;
    first.x = *reinterpret_cast<unsigned *>(&g);
    d[0] = first;
    d[1] = z0;
  }
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

// out[0] (+)= scale * sum of the n partials (one warp, fixed order)
__global__ void k_sum_parts(int n, const float *part, double scale, double *out, int accumulate) {
  sum_parts(n, part, scale, out, accumulate);
}

// Adam (Kingma and Ba, Algorithm 1) on the flat parameter array (the gradient
// is divided by `gdiv`, the number of samples accumulated, and cleared), and
// the BF16 copies of all layers, core matrices as woffs describes:
// Wf[t][o][c] = W[t][o][c] and Wb[26-t][c][o] = W[t][o][c].  Rows and columns
// beyond co (the head's 8 outputs) stay zero.  One launch for both: one per
// layer took 45 us of 1.2 ms per training step.
struct pack_table { int w0[NLAYER], wf[NLAYER], wb[NLAYER], co[NLAYER], ci[NLAYER]; };
template <bool ADAM>
__global__ void k_adam_pack(int n, const __grid_constant__ pack_table T, float *p, float *m, float *v, float *g, float lr,
                            float b1, float b2, float c1, float c2, float eps, float gdiv, bf16 *Wf, bf16 *Wb) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float pi = p[i];
  if (ADAM) {
    float gi = g[i] / gdiv;
    float mi = b1 * m[i] + (1.f - b1) * gi;
    float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi; v[i] = vi;
    pi -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    p[i] = pi;
    g[i] = 0.f;
  }
  int l = 0;
  while (l + 1 < NLAYER && i >= T.w0[l + 1]) l++;
  const int co = T.co[l], ci = T.ci[l], q = i - T.w0[l];
  if (q >= 27 * co * ci) return;                       // a bias
  const int t = q / (co * ci), r = q - t * co * ci, o = r / ci, c = r - o * ci, cr = wrows(co);
  const bf16 w = __float2bfloat16_rn(pi);
  Wf[(size_t)T.wf[l] + (size_t)t * cr * ci + woffs(cr, o, c >> 3) + (c & 7)] = w;
  Wb[(size_t)T.wb[l] + (size_t)(26 - t) * ci * cr + woffs(ci, c, o >> 3) + (o & 7)] = w;
}

// the exported layout (input layer's 8 used channels only) of the parameters,
// or of the mean gradients
__global__ void k_export(int n, const float *p, float div, float *out) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  constexpr int n0 = 27 * 32 * CIN_USED, d0 = 27 * 32 * (CIN_GPU - CIN_USED);
  out[i] = p[i < n0 ? i / CIN_USED * CIN_GPU + i % CIN_USED : i + d0] / div;
}

// network input from FP32 features [V][8] -> BF16 [V][16]
__global__ void k_feat_in(int V, const float *F, bf16 *X) {
  int v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= V) return;
  const float4 *f = reinterpret_cast<const float4 *>(F + (size_t)v * CIN_USED);
  const float4 a = f[0], b = f[1];
  uint4 o;
  __nv_bfloat162 *h = reinterpret_cast<__nv_bfloat162 *>(&o);
  h[0] = __floats2bfloat162_rn(a.x, a.y); h[1] = __floats2bfloat162_rn(a.z, a.w);
  h[2] = __floats2bfloat162_rn(b.x, b.y); h[3] = __floats2bfloat162_rn(b.z, b.w);
  uint4 *d = reinterpret_cast<uint4 *>(X + (size_t)v * CIN_GPU);
  d[0] = o;
  d[1] = make_uint4(0, 0, 0, 0);
}

// ------------------------------------------------------------ the net -----
struct level_bufs {
  dims d;
  dbuf<bf16> a, da, b, cat, p;          // encoder / decoder first-conv outputs, second decoder conv,
                                        // concat [up, skip] [V][64], pooled input
  dbuf<bf16> ga, gda, gb, gcat, ge, gp; // gradients
};

}  // namespace nn
using namespace nn;

struct sim_ws_s {
  cudaStream_t st = nullptr;
  size_t np = 0;                          // number of parameters (device layout)
  size_t woff[NLAYER], boff[NLAYER];      // offsets into the flat arrays
  size_t wfoff[NLAYER], wboff[NLAYER];    // offsets into the BF16 copies
  dbuf<float> P, M, Vm, G;                // master parameters, Adam moments, gradients
  dbuf<bf16> Wf, Wb;
  long long tstep = 0;                    // Adam steps taken
  int accum = 0;                          // samples accumulated in G
  // activations for the current grid
  dims cur = {0, 0, 0};
  level_bufs L[4];
  dbuf<bf16> X0, dY;
  dbuf<float> Y, part, lpart, T32, F32, E;
  dbuf<double> lsum;
  // dataset of (features, target) pairs taken from simulator solves
  struct sample { dims d; dbuf<bf16> X; dbuf<float> T; };
  std::vector<std::unique_ptr<sample>> data;
  size_t max_samples = 1u << 30;
  unsigned long long seed = 0;
  std::mutex use;                         // one caller at a time (activations are shared): see ws_turn
  cudaEvent_t last = nullptr;             // the last simulator's reads of the output, on its own stream
  bool recorded = false;                  // last has been recorded (never for a network that no simulator uses)
  bool tc = true;                         // tcgen05 convolutions (else mma.sync)
  int *err = nullptr, *err_dev = nullptr; // host-mapped: set by a kernel whose bounded wait gave up
  int *err_turn = nullptr;                // where the kernels of the present turn set it: err_dev, or a simulator's own word
  pack_table tab;
  ~sim_ws_s() {
    if (st) cudaStreamDestroy(st);
    if (last) cudaEventDestroy(last);
    if (err) cudaFreeHost(err);
  }
};

// A caller's turn on the handle: the host lock, and stream s (the stream of
// its first access to the activations) behind the last simulator's reads of
// them.  ws_predict returns with its GPU work queued on two streams, so the
// lock alone would let the next caller write what that work still reads.
// The kernels report to err: the handle's own word, or a simulator's, which
// reads it after its own synchronisation, when the next turn may have begun.
struct ws_turn {
  std::lock_guard<std::mutex> guard;
  ws_turn(sim_ws_s *w, cudaStream_t s, int *err = nullptr) : guard(w->use) {
    if (w->recorded) RS_CUDA(cudaStreamWaitEvent(s, w->last, 0));
    w->err_turn = err ? err : w->err_dev;
  }
};

namespace nn {

static void ws_layout(sim_ws_s *w) {
  size_t o = 0, fo = 0, bo = 0;
  for (int l = 0; l < NLAYER; l++) {
    w->woff[l] = o; o += (size_t)27 * LAYERS[l].co * LAYERS[l].ci;
    w->boff[l] = o; o += LAYERS[l].co;
    w->wfoff[l] = fo; fo += (size_t)27 * cob(l) * LAYERS[l].ci;
    w->wboff[l] = bo; bo += (size_t)27 * LAYERS[l].ci * cob(l);
    w->tab.w0[l] = (int)w->woff[l]; w->tab.wf[l] = (int)w->wfoff[l]; w->tab.wb[l] = (int)w->wboff[l];
    w->tab.co[l] = LAYERS[l].co; w->tab.ci[l] = LAYERS[l].ci;
  }
  w->np = o;
  w->P.alloc(o); w->M.alloc(o); w->Vm.alloc(o); w->G.alloc(o);
  w->Wf.alloc(fo); w->Wb.alloc(bo);
  RS_CUDA(cudaMemsetAsync(w->Wf.p, 0, fo * sizeof(bf16), w->st));
  RS_CUDA(cudaMemsetAsync(w->Wb.p, 0, bo * sizeof(bf16), w->st));
}

static void ws_pack(sim_ws_s *w) {
  k_adam_pack<false><<<grid_for(w->np, 256), 256, 0, w->st>>>((int)w->np, w->tab, w->P.p, nullptr, nullptr, nullptr, 0.f,
                                                             0.f, 0.f, 0.f, 0.f, 0.f, 0.f, w->Wf.p, w->Wb.p);
  RS_LAUNCHED(1);
  RS_CHECK_LAUNCH();
}

template <int CI, int NT, int MODE>
static void conv_launch(sim_ws_s *w, dims d, const bf16 *X, int ldx, int offx, const bf16 *Wt, const float *bias,
                        int relu, void *out, int ldo, int offo, const bf16 *mask, int ldm, int offm) {
  static bool attr = false;
  int bytes = conv_smem<CI, NT>::BYTES;
  if (!attr) {
    RS_CUDA(cudaFuncSetAttribute(k_conv<CI, NT, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    attr = true;
  }
  k_conv<CI, NT, MODE><<<grid_for(d.V(), CBM), 128, bytes, w->st>>>(d.nx, d.ny, d.nz, X, ldx, offx, Wt, bias, relu, out,
                                                                     ldo, offo, mask, ldm, offm);
  RS_LAUNCHED(1);
}

template <int CI, int NT, int MODE>
static void conv_halo_launch(sim_ws_s *w, dims d, const bf16 *X, int ldx, int offx, const bf16 *Wt, const float *bias,
                             int relu, void *out, int ldo, int offo) {
  static bool attr = false;
  int bytes = halo_smem<CI, NT>::BYTES;
  if (!attr) {
    RS_CUDA(cudaFuncSetAttribute(k_conv_halo<CI, NT, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    attr = true;
  }
  unsigned tiles = (unsigned)(((d.nx + HX - 1) / HX) * ((d.ny + HY - 1) / HY) * ((d.nz + HZ - 1) / HZ));
  k_conv_halo<CI, NT, MODE><<<tiles, 128, bytes, w->st>>>(d.nx, d.ny, d.nz, X, ldx, offx, Wt, bias, relu, out, ldo,
                                                           offo);
  RS_LAUNCHED(1);
}

// Slices per CTA: more of them share a halo and the weights' copy, fewer fill
// the chip on small grids.  Taken by a model of the time in units of one
// slice's MMAs at 32 input channels (1 us): rounds of resident CTAs, each a
// start (TMEM, copies, epilogue: 2) and its resident slices one after the other.
template <int CI, int CO, int MODE>
static void conv_tc_launch(sim_ws_s *w, dims d, const bf16 *X, int ldx, int offx, const bf16 *Wt, const float *bias,
                           int relu, void *out, int ldo, int offo, const bf16 *mask, int ldm, int offm) {
  static int per_sm[5] = {0, 0, 0, 0, 0};     // resident CTAs per SM by slices (0: does not fit)
  static int sms = 0;
  static std::once_flag once;
  std::call_once(once, [&] {
    int dev = 0, cap = 0;
    RS_CUDA(cudaGetDevice(&dev));
    RS_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    RS_CUDA(cudaDeviceGetAttribute(&cap, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    int top = 0;
    for (int z = 1; z <= 4; z++) if (tc_bytes(CI, CO, z) + 128 <= cap) top = z;
    RS_CUDA(cudaFuncSetAttribute(k_conv_tc<CI, CO, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, tc_bytes(CI, CO, top)));
    for (int z = 1; z <= top; z++) {
      RS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm[z], k_conv_tc<CI, CO, MODE>, TC_T, tc_bytes(CI, CO, z)));
      per_sm[z] = std::max(1, std::min(per_sm[z], 512 / tc_cols(CO, z)));
    }
  });
  const long long txy = (long long)((d.nx + TBX - 1) / TBX) * ((d.ny + TBY - 1) / TBY);
  int NZ = 1;
  double best = 1e300;
  for (int z = 1; z <= 4 && per_sm[z]; z++) {
    const long long tiles = txy * ((d.nz + z - 1) / z), r = std::min<long long>(per_sm[z], (tiles + sms - 1) / sms),
                    rounds = (tiles + sms * r - 1) / (sms * r);
    const double c = rounds * (2.0 + r * z * (CI / 32.0));
    if (c < best) { best = c; NZ = z; }
  }
  const unsigned tiles = (unsigned)(txy * ((d.nz + NZ - 1) / NZ));
  launch_pdl(k_conv_tc<CI, CO, MODE>, tiles, TC_T, (size_t)tc_bytes(CI, CO, NZ), w->st, d.nx, d.ny, d.nz, NZ, X, ldx, offx,
             Wt, bias, relu, out, ldo, offo, mask, ldm, offm, w->err_turn);
  RS_LAUNCHED(1);
}

// forward conv of layer l: in (ld, off) -> out (ldo, offo)
static void fwd(sim_ws_s *w, int l, dims d, const bf16 *X, int ldx, int offx, void *out, int ldo, int offo) {
  const bf16 *Wt = w->Wf.p + w->wfoff[l];
  const float *b = w->P.p + w->boff[l];
  int ci = LAYERS[l].ci;
  if (w->tc) {
    if (l == HEAD) conv_tc_launch<32, 16, 1>(w, d, X, ldx, offx, Wt, b, 0, out, ldo, offo, nullptr, 0, 0);
    else if (ci == 16) conv_tc_launch<16, 32, 0>(w, d, X, ldx, offx, Wt, b, 1, out, ldo, offo, nullptr, 0, 0);
    else if (ci == 32) conv_tc_launch<32, 32, 0>(w, d, X, ldx, offx, Wt, b, 1, out, ldo, offo, nullptr, 0, 0);
    else conv_tc_launch<64, 32, 0>(w, d, X, ldx, offx, Wt, b, 1, out, ldo, offo, nullptr, 0, 0);
  }
  else if (l == HEAD) conv_halo_launch<32, 1, 1>(w, d, X, ldx, offx, Wt, b, 0, out, ldo, offo);
  else if (ci == 16) conv_halo_launch<16, 4, 0>(w, d, X, ldx, offx, Wt, b, 1, out, ldo, offo);
  else if (ci == 32) conv_halo_launch<32, 4, 0>(w, d, X, ldx, offx, Wt, b, 1, out, ldo, offo);
  else conv_halo_launch<64, 4, 0>(w, d, X, ldx, offx, Wt, b, 1, out, ldo, offo);
}

// data gradient of layer l: dZ (ldz, offz) -> dX (ldo, offo), masked by the
// layer's input (mask != nullptr) when that input came out of a ReLU
static void bwd_data(sim_ws_s *w, int l, dims d, const bf16 *dZ, int ldz, int offz, bf16 *out, int ldo, int offo,
                     const bf16 *mask, int ldm, int offm) {
  const bf16 *Wt = w->Wb.p + w->wboff[l];
  int ci = LAYERS[l].ci;
  if (w->tc && l != C00) {
    if (l == HEAD) {
      if (mask) conv_tc_launch<16, 32, 2>(w, d, dZ, ldz, offz, Wt, nullptr, 0, out, ldo, offo, mask, ldm, offm);
      else conv_tc_launch<16, 32, 3>(w, d, dZ, ldz, offz, Wt, nullptr, 0, out, ldo, offo, mask, ldm, offm);
    } else if (ci == 64) {
      if (mask) conv_tc_launch<32, 64, 2>(w, d, dZ, ldz, offz, Wt, nullptr, 0, out, ldo, offo, mask, ldm, offm);
      else conv_tc_launch<32, 64, 3>(w, d, dZ, ldz, offz, Wt, nullptr, 0, out, ldo, offo, mask, ldm, offm);
    } else {
      if (mask) conv_tc_launch<32, 32, 2>(w, d, dZ, ldz, offz, Wt, nullptr, 0, out, ldo, offo, mask, ldm, offm);
      else conv_tc_launch<32, 32, 3>(w, d, dZ, ldz, offz, Wt, nullptr, 0, out, ldo, offo, mask, ldm, offm);
    }
    return;
  }
  if (l == HEAD) {     // input: dY with 16 channels; output 32
    if (mask) conv_launch<16, 4, 2>(w, d, dZ, ldz, offz, Wt, nullptr, 0, out, ldo, offo, mask, ldm, offm);
    else conv_launch<16, 4, 3>(w, d, dZ, ldz, offz, Wt, nullptr, 0, out, ldo, offo, mask, ldm, offm);
  } else if (ci == 64) {
    if (mask) conv_launch<32, 8, 2>(w, d, dZ, ldz, offz, Wt, nullptr, 0, out, ldo, offo, mask, ldm, offm);
    else conv_launch<32, 8, 3>(w, d, dZ, ldz, offz, Wt, nullptr, 0, out, ldo, offo, mask, ldm, offm);
  } else if (ci == 32) {
    if (mask) conv_launch<32, 4, 2>(w, d, dZ, ldz, offz, Wt, nullptr, 0, out, ldo, offo, mask, ldm, offm);
    else conv_launch<32, 4, 3>(w, d, dZ, ldz, offz, Wt, nullptr, 0, out, ldo, offo, mask, ldm, offm);
  } else {
    RS_FAIL(SIM_ERR_ARG, "no data gradient for the input layer");
  }
}

// Weight gradients of all layers, from the activations and the gradients that
// the data-gradient passes left (each in a buffer of its own): one launch of
// at most a CTA per SM, shared out by the layers' slices, and one that adds
// the chunks and the loss.
struct wg_in { const bf16 *X; int ldx, offx; const bf16 *dZ; int ldz; dims d; };
static void wgrad(sim_ws_s *w, const wg_in in[NLAYER], int nl, double lscale) {
  wg_table tab;
  static int sms = 0;
  static std::once_flag once;
  std::call_once(once, [&] {
    int dev = 0;
    RS_CUDA(cudaGetDevice(&dev));
    RS_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    RS_CUDA(cudaFuncSetAttribute(k_conv_wgrad, cudaFuncAttributeMaxDynamicSharedMemorySize, WG_BYTES));
  });
  auto slices = [&](int l) { return (long long)((in[l].d.nx + TBX - 1) / TBX) * ((in[l].d.ny + TBY - 1) / TBY) * in[l].d.nz; };
  auto halves = [](int l) { return (LAYERS[l].ci + 31) / 32; };
  // the fewest slices per CTA that need no second round
  long long units = 0, per = 1;
  for (int l = 0; l < NLAYER; l++) units += slices(l) * halves(l);
  for (per = std::max(1LL, units / sms);; per += 1 + per / 64) {
    long long ctas = 0;
    for (int l = 0; l < NLAYER; l++) ctas += halves(l) * ((slices(l) + per - 1) / per);
    if (ctas <= sms || per >= units) break;
  }
  int block = 0;
  size_t need = 0;
  for (int l = 0; l < NLAYER; l++) {
    wg_layer &L = tab.l[l];
    const int co = LAYERS[l].co, ci = LAYERS[l].ci;
    L.X = in[l].X; L.ldx = in[l].ldx; L.offx = in[l].offx; L.dZ = in[l].dZ; L.ldz = in[l].ldz;
    L.nx = in[l].d.nx; L.ny = in[l].d.ny; L.nz = in[l].d.nz; L.co = co; L.ci = ci;
    L.nchunk = (int)((slices(l) + per - 1) / per);
    L.block0 = block;
    block += L.nchunk * halves(l);
    need += (size_t)L.nchunk * (27 * co * ci + co);
  }
  w->part.ensure(need);
  float *p = w->part.p;
  for (int l = 0; l < NLAYER; l++) {
    wg_layer &L = tab.l[l];
    L.part = p; p += (size_t)L.nchunk * 27 * L.co * L.ci;
    L.bpart = p; p += (size_t)L.nchunk * L.co;
  }
  launch_pdl(k_conv_wgrad, (unsigned)block, WG_T, (size_t)WG_BYTES, w->st, tab, w->err_turn);
  launch_pdl(k_wgrad_reduce, grid_for(w->np, 256) + 1, 256, 0, w->st, tab, (int)w->np, w->G.p, nl, w->lpart.p, lscale,
             w->lsum.p);
  RS_LAUNCHED(2);
}

static void ensure_dims(sim_ws_s *w, dims d) {
  if (d.nx == w->cur.nx && d.ny == w->cur.ny && d.nz == w->cur.nz) return;
  dims c = d;
  for (int k = 0; k < 4; k++) {
    level_bufs &B = w->L[k];
    B.d = c;
    size_t V = c.V();
    B.a.alloc(V * 32); B.da.alloc(V * 32); B.b.alloc(V * 32); B.cat.alloc(V * 64); B.p.alloc(V * 32);
    B.ga.alloc(V * 32); B.gda.alloc(V * 32); B.gb.alloc(V * 32); B.gcat.alloc(V * 64); B.ge.alloc(V * 32);
    B.gp.alloc(V * 32);
    c = coarse(c);
  }
  size_t V = d.V();
  w->X0.alloc(V * CIN_GPU); w->dY.alloc(V * 16); w->Y.alloc(V * COUT_HEAD);
  w->lpart.alloc(grid_for(V, 256));
  w->cur = d;
}

// Forward pass on w->X0 (BF16 [V][16]) -> w->Y (FP32 [V][8]).
// Level k buffers: a = first encoder conv, cat = [up, skip] (skip = second
// encoder conv), p = pooled input (levels 1..3), da = first decoder conv,
// b = second decoder conv (the bottom's second conv at level 3).
static void forward(sim_ws_s *w) {
  level_bufs *L = w->L;
  fwd(w, C00, L[0].d, w->X0.p, CIN_GPU, 0, L[0].a.p, 32, 0);
  fwd(w, C01, L[0].d, L[0].a.p, 32, 0, L[0].cat.p, 64, 32);
  for (int k = 1; k <= 3; k++) {
    launch_pdl(k_pool, grid_for((size_t)L[k].d.V() * 4, 256), 256, 0, w->st, L[k - 1].d, L[k].d, L[k - 1].cat.p, 64, 32, L[k].p.p);
    RS_LAUNCHED(1);
    int c0 = k == 1 ? C10 : k == 2 ? C20 : C30;
    fwd(w, c0, L[k].d, L[k].p.p, 32, 0, L[k].a.p, 32, 0);
    if (k < 3) fwd(w, c0 + 1, L[k].d, L[k].a.p, 32, 0, L[k].cat.p, 64, 32);
    else fwd(w, c0 + 1, L[k].d, L[k].a.p, 32, 0, L[k].b.p, 32, 0);
  }
  for (int k = 2; k >= 0; k--) {
    launch_pdl(k_up, grid_for((size_t)L[k].d.V() * 4, 256), 256, 0, w->st, L[k].d, L[k + 1].d, L[k + 1].b.p, L[k].cat.p, 64, 0);
    RS_LAUNCHED(1);
    int d0 = k == 2 ? D20 : k == 1 ? D10 : D00;
    fwd(w, d0, L[k].d, L[k].cat.p, 64, 0, L[k].da.p, 32, 0);
    fwd(w, d0 + 1, L[k].d, L[k].da.p, 32, 0, L[k].b.p, 32, 0);
  }
  fwd(w, HEAD, L[0].d, L[0].b.p, 32, 0, w->Y.p, COUT_HEAD, 0);
  RS_CHECK_LAUNCH();
}

// loss against T32 ([V][2]) accumulated into lsum (scaled 0.5/V); gradients
// accumulated into G.  Uses the activations of the last forward().
static void backward(sim_ws_s *w, const float *T) {
  level_bufs *L = w->L;
  int V = L[0].d.V();
  wg_in in[NLAYER];
  auto wgrad = [&](int l, dims d, const bf16 *X, int ldx, int offx, const bf16 *dZ, int ldz) { in[l] = {X, ldx, offx, dZ, ldz, d}; };
  launch_pdl(k_loss, grid_for(V, 256), 256, 0, w->st, V, w->Y.p, T, w->dY.p, w->lpart.p);
  RS_LAUNCHED(1);
  // head: input b0, output dY
  wgrad(HEAD, L[0].d, L[0].b.p, 32, 0, w->dY.p, 16);
  bwd_data(w, HEAD, L[0].d, w->dY.p, 16, 0, L[0].gb.p, 32, 0, L[0].b.p, 32, 0);
  // decoder, finest level first
  for (int k = 0; k <= 2; k++) {
    int d0 = k == 2 ? D20 : k == 1 ? D10 : D00;
    // second decoder conv: input da, output gradient gb
    wgrad(d0 + 1, L[k].d, L[k].da.p, 32, 0, L[k].gb.p, 32);
    bwd_data(w, d0 + 1, L[k].d, L[k].gb.p, 32, 0, L[k].gda.p, 32, 0, L[k].da.p, 32, 0);
    // first decoder conv: input cat, output gradient gda
    wgrad(d0, L[k].d, L[k].cat.p, 64, 0, L[k].gda.p, 32);
    bwd_data(w, d0, L[k].d, L[k].gda.p, 32, 0, L[k].gcat.p, 64, 0, L[k].cat.p, 64, 0);
    // up-sampled half -> gradient of the coarser level's output (gb there)
    launch_pdl(k_up_back, grid_for((size_t)L[k + 1].d.V() * 4, 256), 256, 0, w->st, L[k].d, L[k + 1].d, L[k].gcat.p, 64, 0, L[k + 1].gb.p);
    RS_LAUNCHED(1);
  }
  // bottom: c31 (input a3, output b3), c30 (input p3)
  wgrad(C31, L[3].d, L[3].a.p, 32, 0, L[3].gb.p, 32);
  bwd_data(w, C31, L[3].d, L[3].gb.p, 32, 0, L[3].ga.p, 32, 0, L[3].a.p, 32, 0);
  wgrad(C30, L[3].d, L[3].p.p, 32, 0, L[3].ga.p, 32);
  bwd_data(w, C30, L[3].d, L[3].ga.p, 32, 0, L[3].gp.p, 32, 0, nullptr, 0, 0);
  // encoder, coarse to fine: ge(k) = mask * (skip part of gcat(k) + pool-back of gp(k+1))
  for (int k = 2; k >= 0; k--) {
    launch_pdl(k_pool_back, grid_for((size_t)L[k].d.V() * 4, 256), 256, 0, w->st, L[k].d, L[k + 1].d, L[k + 1].gp.p, L[k].gcat.p, 64, 32, L[k].cat.p, 64, 32, L[k].ge.p);
    RS_LAUNCHED(1);
    int c0 = k == 2 ? C20 : k == 1 ? C10 : C00;
    wgrad(c0 + 1, L[k].d, L[k].a.p, 32, 0, L[k].ge.p, 32);
    bwd_data(w, c0 + 1, L[k].d, L[k].ge.p, 32, 0, L[k].ga.p, 32, 0, L[k].a.p, 32, 0);
    if (k > 0) {
      wgrad(c0, L[k].d, L[k].p.p, 32, 0, L[k].ga.p, 32);
      bwd_data(w, c0, L[k].d, L[k].ga.p, 32, 0, L[k].gp.p, 32, 0, nullptr, 0, 0);
    } else {
      wgrad(C00, L[0].d, w->X0.p, CIN_GPU, 0, L[0].ga.p, 32);
    }
  }
  nn::wgrad(w, in, (int)grid_for(V, 256), 0.5 / V);
  RS_CHECK_LAUNCH();
  w->accum++;
}

static void zero_grad(sim_ws_s *w) {
  RS_CUDA(cudaMemsetAsync(w->G.p, 0, w->np * sizeof(float), w->st));
  w->accum = 0;
}

static void adam(sim_ws_s *w, double lr) {
  if (w->accum == 0) return;
  w->tstep++;
  const double b1 = 0.9, b2 = 0.999;
  float c1 = (float)(1.0 - std::pow(b1, (double)w->tstep)), c2 = (float)(1.0 - std::pow(b2, (double)w->tstep));
  k_adam_pack<true><<<grid_for(w->np, 256), 256, 0, w->st>>>((int)w->np, w->tab, w->P.p, w->M.p, w->Vm.p, w->G.p, (float)lr,
                                                            (float)b1, (float)b2, c1, c2, 1e-8f, (float)w->accum, w->Wf.p,
                                                            w->Wb.p);
  RS_LAUNCHED(1);
  RS_CHECK_LAUNCH();
  w->accum = 0;
}

// splitmix64 (Steele, Lea and Flood 2014) and a Box-Muller normal draw for
// the He initialisation
static inline uint64_t smix(uint64_t &s) {
  uint64_t z = (s += 0x9E3779B97F4A7C15ull);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
static inline double unif(uint64_t &s) { return ((smix(s) >> 11) + 0.5) * (1.0 / 9007199254740992.0); }

}  // namespace nn

// ---------------------------------------------------------------- ABI -----
#define ABI_BEGIN try {
#define ABI_END                                                       \
  }                                                                   \
  catch (const rs_error &e) { return e.code; }                        \
  catch (const std::bad_alloc &) { rs_set_error("host allocation failed"); return SIM_ERR_OOM; } \
  catch (...) { rs_set_error("unexpected exception"); return SIM_ERR_CUDA; }                       \
  return SIM_OK;

// parameter count in the exported layout: per layer W[27][Co][Ci] (Ci = 8 for
// the input layer) then b[Co]
static size_t export_count() {
  size_t n = 0;
  for (int l = 0; l < NLAYER; l++) n += (size_t)27 * LAYERS[l].co * ci_true(l) + LAYERS[l].co;
  return n;
}

// a tensor-core kernel whose bounded wait gave up leaves a flag in the
// turn's error word; report it (the caller has synchronised with the kernels)
void ws_check(volatile int *e) {
  if (*e) {
    *e = 0;
    RS_FAIL(SIM_ERR_TIMEOUT, "warm-start network: a tensor-core pipeline wait gave up");
  }
}
static void check_err(sim_ws_s *w) { ws_check(w->err); }

extern "C" sim_status sim_ws_create(sim_ws_t *out, unsigned long long seed) {
  ABI_BEGIN
  if (!out) RS_FAIL(SIM_ERR_ARG, "sim_ws_create: NULL argument");
  *out = nullptr;
  std::unique_ptr<sim_ws_s> w(new sim_ws_s());
  RS_CUDA(cudaStreamCreateWithFlags(&w->st, cudaStreamNonBlocking));
  RS_CUDA(cudaEventCreateWithFlags(&w->last, cudaEventDisableTiming));
  ws_layout(w.get());
  w->seed = seed;
  // He-normal weights (std sqrt(2 / (27 ci))), zero biases; padding channels
  // zero; the head starts at zero, so an untrained network predicts no
  // correction
  std::vector<float> h(w->np, 0.f);
  uint64_t s = seed;
  for (int l = 0; l < HEAD; l++) {
    int co = LAYERS[l].co, ci = LAYERS[l].ci, ct = ci_true(l);
    double sd = std::sqrt(2.0 / (27.0 * ct));
    for (int t = 0; t < 27; t++)
      for (int o = 0; o < co; o++)
        for (int c = 0; c < ct; c++) {
          double u1 = unif(s), u2 = unif(s);
          h[w->woff[l] + ((size_t)t * co + o) * ci + c] = (float)(sd * std::sqrt(-2.0 * std::log(u1)) * std::cos(6.283185307179586 * u2));
        }
  }
  RS_CUDA(cudaMemcpyAsync(w->P.p, h.data(), w->np * sizeof(float), cudaMemcpyHostToDevice, w->st));
  RS_CUDA(cudaMemsetAsync(w->M.p, 0, w->np * sizeof(float), w->st));
  RS_CUDA(cudaMemsetAsync(w->Vm.p, 0, w->np * sizeof(float), w->st));
  w->lsum.alloc(2);
  RS_CUDA(cudaHostAlloc((void **)&w->err, sizeof(int), cudaHostAllocMapped));
  *w->err = 0;
  RS_CUDA(cudaHostGetDevicePointer((void **)&w->err_dev, w->err, 0));
  zero_grad(w.get());
  ws_pack(w.get());
  RS_CUDA(cudaStreamSynchronize(w->st));
  *out = w.release();
  ABI_END
}

extern "C" void sim_ws_destroy(sim_ws_t w) { delete w; }

extern "C" sim_status sim_ws_use_tcgen05(sim_ws_t w, int on) {
  ABI_BEGIN
  if (!w) RS_FAIL(SIM_ERR_ARG, "NULL handle");
  std::lock_guard<std::mutex> guard(w->use);
  w->tc = on != 0;
  ABI_END
}

// which = 0: master parameters, 1: accumulated gradients (divided by the
// number of samples accumulated, i.e. the mean over the batch)
extern "C" sim_status sim_ws_params(sim_ws_t w, int which, float *dst, size_t n, size_t *needed) {
  ABI_BEGIN
  if (!w || (which != 0 && which != 1)) RS_FAIL(SIM_ERR_ARG, "sim_ws_params: bad argument");
  size_t ne = export_count();
  if (needed) *needed = ne;
  if (!dst) return SIM_OK;
  if (n < ne) RS_FAIL(SIM_ERR_ARG, "sim_ws_params: buffer holds %zu of %zu values", n, ne);
  ws_turn turn(w, w->st);
  w->E.ensure(ne);
  k_export<<<grid_for(ne, 256), 256, 0, w->st>>>((int)ne, which == 0 ? w->P.p : w->G.p,
                                                which == 1 && w->accum > 0 ? (float)w->accum : 1.f, w->E.p);
  RS_LAUNCHED(1);
  RS_CUDA(cudaMemcpyAsync(dst, w->E.p, ne * sizeof(float), cudaMemcpyDefault, w->st));
  RS_CUDA(cudaStreamSynchronize(w->st));
  ABI_END
}

extern "C" sim_status sim_ws_set_params(sim_ws_t w, const float *src, size_t n) {
  ABI_BEGIN
  if (!w || !src) RS_FAIL(SIM_ERR_ARG, "sim_ws_set_params: NULL argument");
  size_t ne = export_count();
  if (n != ne) RS_FAIL(SIM_ERR_ARG, "sim_ws_set_params: expected %zu values, got %zu", ne, n);
  std::vector<float> h(w->np, 0.f);
  size_t q = 0;
  for (int l = 0; l < NLAYER; l++) {
    int co = LAYERS[l].co, ci = LAYERS[l].ci, ct = ci_true(l);
    for (int t = 0; t < 27; t++)
      for (int o = 0; o < co; o++)
        for (int c = 0; c < ct; c++) h[w->woff[l] + ((size_t)t * co + o) * ci + c] = src[q++];
    for (int o = 0; o < co; o++) h[w->boff[l] + o] = src[q++];
  }
  ws_turn turn(w, w->st);
  RS_CUDA(cudaMemcpyAsync(w->P.p, h.data(), w->np * sizeof(float), cudaMemcpyHostToDevice, w->st));
  RS_CUDA(cudaMemsetAsync(w->M.p, 0, w->np * sizeof(float), w->st));
  RS_CUDA(cudaMemsetAsync(w->Vm.p, 0, w->np * sizeof(float), w->st));
  w->tstep = 0;
  zero_grad(w);
  ws_pack(w);
  RS_CUDA(cudaStreamSynchronize(w->st));
  ABI_END
}

static void load_features(sim_ws_s *w, dims d, const float *feat) {
  ensure_dims(w, d);
  size_t V = d.V();
  w->F32.ensure(V * CIN_USED);
  RS_CUDA(cudaMemcpyAsync(w->F32.p, feat, V * CIN_USED * sizeof(float), cudaMemcpyDefault, w->st));
  k_feat_in<<<grid_for(V, 256), 256, 0, w->st>>>((int)V, w->F32.p, w->X0.p);
  RS_LAUNCHED(1);
}

extern "C" sim_status sim_ws_forward(sim_ws_t w, int nx, int ny, int nz, const float *feat, float *y) {
  ABI_BEGIN
  if (!w || !feat || !y || nx < 1 || ny < 1 || nz < 1) RS_FAIL(SIM_ERR_ARG, "sim_ws_forward: bad argument");
  ws_turn turn(w, w->st);
  dims d = {nx, ny, nz};
  load_features(w, d, feat);
  forward(w);
  RS_CUDA(cudaMemcpyAsync(y, w->Y.p, (size_t)d.V() * COUT_HEAD * sizeof(float), cudaMemcpyDefault, w->st));
  RS_CUDA(cudaStreamSynchronize(w->st));
  check_err(w);
  ABI_END
}

// Forward, loss and backward for one sample; gradients are added to the
// accumulated ones (sim_ws_zero_grad clears them) and *loss receives this
// sample's loss.
extern "C" sim_status sim_ws_backward(sim_ws_t w, int nx, int ny, int nz, const float *feat, const float *target,
                                      double *loss) {
  ABI_BEGIN
  if (!w || !feat || !target || nx < 1 || ny < 1 || nz < 1) RS_FAIL(SIM_ERR_ARG, "sim_ws_backward: bad argument");
  ws_turn turn(w, w->st);
  dims d = {nx, ny, nz};
  load_features(w, d, feat);
  size_t V = d.V();
  w->T32.ensure(V * NPRED);
  RS_CUDA(cudaMemcpyAsync(w->T32.p, target, V * NPRED * sizeof(float), cudaMemcpyDefault, w->st));
  forward(w);
  RS_CUDA(cudaMemsetAsync(w->lsum.p, 0, sizeof(double), w->st));
  backward(w, w->T32.p);
  double l = 0.0;
  RS_CUDA(cudaMemcpyAsync(&l, w->lsum.p, sizeof(double), cudaMemcpyDeviceToHost, w->st));
  RS_CUDA(cudaStreamSynchronize(w->st));
  check_err(w);
  if (loss) *loss = l;
  ABI_END
}

extern "C" sim_status sim_ws_zero_grad(sim_ws_t w) {
  ABI_BEGIN
  if (!w) RS_FAIL(SIM_ERR_ARG, "NULL handle");
  ws_turn turn(w, w->st);
  zero_grad(w);
  RS_CUDA(cudaStreamSynchronize(w->st));
  ABI_END
}

extern "C" sim_status sim_ws_adam(sim_ws_t w, double lr) {
  ABI_BEGIN
  if (!w || !(lr > 0)) RS_FAIL(SIM_ERR_ARG, "sim_ws_adam: bad argument");
  ws_turn turn(w, w->st);
  adam(w, lr);
  RS_CUDA(cudaStreamSynchronize(w->st));
  ABI_END
}

extern "C" sim_status sim_ws_dataset(sim_ws_t w, int *n_samples) {
  ABI_BEGIN
  if (!w || !n_samples) RS_FAIL(SIM_ERR_ARG, "NULL argument");
  std::lock_guard<std::mutex> guard(w->use);
  *n_samples = (int)w->data.size();
  ABI_END
}

// Epochs over the recorded samples in a seeded random order, Adam step every
// `batch` samples; *mean_loss = mean sample loss of the last epoch.
extern "C" sim_status sim_ws_train(sim_ws_t w, int epochs, int batch, double lr, unsigned long long seed,
                                   double *mean_loss) {
  ABI_BEGIN
  if (!w || epochs < 0 || batch < 1 || !(lr > 0)) RS_FAIL(SIM_ERR_ARG, "sim_ws_train: bad argument");
  ws_turn turn(w, w->st);
  int n = (int)w->data.size();
  if (n == 0) RS_FAIL(SIM_ERR_STATE, "sim_ws_train: no recorded samples");
  std::vector<int> order(n);
  uint64_t s = seed;
  double last = 0.0;
  zero_grad(w);
  for (int e = 0; e < epochs; e++) {
    for (int k = 0; k < n; k++) order[k] = k;
    for (int k = n - 1; k > 0; k--) std::swap(order[k], order[(int)(smix(s) % (uint64_t)(k + 1))]);   // Fisher-Yates
    RS_CUDA(cudaMemsetAsync(w->lsum.p, 0, sizeof(double), w->st));
    for (int k = 0; k < n; k++) {
      auto &S = *w->data[order[k]];
      ensure_dims(w, S.d);
      RS_CUDA(cudaMemcpyAsync(w->X0.p, S.X.p, (size_t)S.d.V() * CIN_GPU * sizeof(bf16), cudaMemcpyDeviceToDevice, w->st));
      forward(w);
      backward(w, S.T.p);
      if (w->accum == batch || k == n - 1) adam(w, lr);
    }
    double l = 0.0;
    RS_CUDA(cudaMemcpyAsync(&l, w->lsum.p, sizeof(double), cudaMemcpyDeviceToHost, w->st));
    RS_CUDA(cudaStreamSynchronize(w->st));
    check_err(w);
    last = l / n;
  }
  if (mean_loss) *mean_loss = last;
  ABI_END
}

// mean loss over the recorded samples with the current weights (no update)
extern "C" sim_status sim_ws_eval(sim_ws_t w, double *mean_loss) {
  ABI_BEGIN
  if (!w || !mean_loss) RS_FAIL(SIM_ERR_ARG, "NULL argument");
  ws_turn turn(w, w->st);
  int n = (int)w->data.size();
  if (n == 0) RS_FAIL(SIM_ERR_STATE, "sim_ws_eval: no recorded samples");
  RS_CUDA(cudaMemsetAsync(w->lsum.p, 0, sizeof(double), w->st));
  for (int k = 0; k < n; k++) {
    auto &S = *w->data[k];
    ensure_dims(w, S.d);
    RS_CUDA(cudaMemcpyAsync(w->X0.p, S.X.p, (size_t)S.d.V() * CIN_GPU * sizeof(bf16), cudaMemcpyDeviceToDevice, w->st));
    forward(w);
    int V = S.d.V();
    k_loss<<<grid_for(V, 256), 256, 0, w->st>>>(V, w->Y.p, S.T.p, w->dY.p, w->lpart.p);
    k_sum_parts<<<1, 32, 0, w->st>>>((int)grid_for(V, 256), w->lpart.p, 0.5 / V, w->lsum.p, 1);
    RS_LAUNCHED(2);
  }
  double l = 0.0;
  RS_CUDA(cudaMemcpyAsync(&l, w->lsum.p, sizeof(double), cudaMemcpyDeviceToHost, w->st));
  RS_CUDA(cudaStreamSynchronize(w->st));
  check_err(w);
  *mean_loss = l / n;
  ABI_END
}

// ------------------------------------------------ simulator integration ---
// Features of the current system, on the simulator's stream: X [n][16] BF16,
// from the decoupled right-hand side b (the Newton residual), ln k, s_w and
// the previous solve's update yp (cell rows; each vector component over its
// rms over the cells; channels 6-7 are zero):
//   sc[0], sc[1] = rms of b (pressure / saturation rows),
//   sc[2], sc[3] = rms of the solved update (recording only: the target's scales),
//   sc[4], sc[5] = rms of yp (0 when there is no previous update).
__global__ void k_ws_features(int n, const double *b, const double *kx, const double *sw, const double *yp,
                              const double *sc, bf16 *X) {
  int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= n) return;
  auto q = [](double a, double s) { return s > 0.0 ? (float)(a / s) : 0.f; };
  float f[8];
  f[0] = q(b[2 * (size_t)c], sc[0]);
  f[1] = q(b[2 * (size_t)c + 1], sc[1]);
  f[2] = (float)((log(kx[c]) - 4.0) * 0.5);
  f[3] = (float)((sw[c] - 0.5) * 4.0);
  f[4] = q(yp[2 * (size_t)c], sc[4]);
  f[5] = q(yp[2 * (size_t)c + 1], sc[5]);
  f[6] = 0.f;
  f[7] = 0.f;
  bf16 *o = X + (size_t)c * CIN_GPU;
#pragma unroll
  for (int a = 0; a < 8; a++) o[a] = __float2bfloat16_rn(f[a]);
#pragma unroll
  for (int a = 8; a < CIN_GPU; a++) o[a] = __float2bfloat16_rn(0.f);
}

// The network predicts the update's shape, each component with unit rms:
// two candidate vectors, its pressure part dp = (Y[c][0], 0) and its
// saturation part ds = (0, Y[c][1]) for cells, 0 for well rows (the least-
// squares fit of the initial guess sets both scales)
__global__ void k_ws_predict(int n, int nb, const float *Y, double *dp, double *ds) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 2 * nb) return;
  int c = i >> 1, a = i & 1;
  double v = c < n ? (double)Y[(size_t)c * COUT_HEAD + a] : 0.0;
  dp[i] = a == 0 ? v : 0.0;
  ds[i] = a == 1 ? v : 0.0;
}

// T[c][a] = y[2c + a] / rms(y_a) (the training target of this system)
__global__ void k_ws_target(int n, const double *y, const double *sc, float *T) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 2 * n) return;
  double s = sc[2 + (i & 1)];
  T[i] = s > 0.0 ? (float)(y[i] / s) : 0.f;
}

// rms over the n cells of the two interleaved components of v -> out[0], out[1].
// One cluster of eight CTAs, whose partial sums the first adds through
// distributed shared memory: no workspace and a fixed order.  With a single
// CTA its SM's FP64 pipe and latency bounded the sum.  Another CTA's shared
// memory may be written only once that CTA runs: every thread arrives on the
// cluster's barrier at the start and waits for it before the store, so that
// the summation hides the barrier; the second barrier ends the stores.
constexpr int RMS_C = 8, RMS_U = 4;
__global__ void __cluster_dims__(RMS_C, 1, 1) __launch_bounds__(1024) k_rms2(int n, const double *v, double *out) {
  __shared__ double sh[2][32];
  __shared__ double all[2][RMS_C];
  cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
  const int t = threadIdx.x, rank = (int)cl.block_rank(), step = RMS_C * 1024;
  auto running = cl.barrier_arrive();
  double s0 = 0.0, s1 = 0.0;
  for (int c0 = rank * 1024 + t; c0 < n; c0 += RMS_U * step) {
    double2 a[RMS_U];
#pragma unroll
    for (int u = 0; u < RMS_U; u++)
      a[u] = c0 + (long long)u * step < n ? reinterpret_cast<const double2 *>(v)[c0 + u * step] : make_double2(0.0, 0.0);
#pragma unroll
    for (int u = 0; u < RMS_U; u++) { s0 += a[u].x * a[u].x; s1 += a[u].y * a[u].y; }
  }
  auto warp_sum = [](double x) {
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    return x;
  };
  s0 = warp_sum(s0); s1 = warp_sum(s1);
  if ((t & 31) == 0) { sh[0][t >> 5] = s0; sh[1][t >> 5] = s1; }
  __syncthreads();
  cl.barrier_wait(std::move(running));                 // all eight CTAs run
  if (t < 64) {
    const double x = warp_sum(sh[t >> 5][t & 31]);
    if ((t & 31) == 0) *cl.map_shared_rank(&all[t >> 5][rank], 0) = x;
  }
  cl.sync();
  if (rank == 0 && t < 2) {
    double x = 0.0;
    for (int k = 0; k < RMS_C; k++) x += all[t][k];
    out[t] = sqrt(x / n);
  }
}

void ws_rms2(int n, const double *v, double *out, cudaStream_t s) {
  k_rms2<<<RMS_C, 1024, 0, s>>>(n, v, out);
  RS_LAUNCHED(1);
}

// predicted update as two candidates in y (2 x 2 nb, FP64, device: pressure
// part, then saturation part) for the system whose decoupled right-hand side
// is b; yp, sc as above (device).  err (device address of a host-mapped word):
// set by a kernel that gave up, for ws_check after a synchronisation with s
void ws_predict(sim_ws_s *w, int nx, int ny, int nz, int nb, const double *b, const double *kx, const double *sw,
                const double *yp, const double *sc, double *y, int *err, cudaStream_t s) {
  ws_turn turn(w, s, err);
  dims d = {nx, ny, nz};
  ensure_dims(w, d);
  int n = d.V();
  // the network runs on its own stream, ordered after the simulator's work
  cudaEvent_t ev;
  RS_CUDA(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
  k_ws_features<<<grid_for(n, 256), 256, 0, s>>>(n, b, kx, sw, yp, sc, w->X0.p);
  RS_LAUNCHED(1);
  RS_CUDA(cudaEventRecord(ev, s));
  RS_CUDA(cudaStreamWaitEvent(w->st, ev, 0));
  forward(w);
  RS_CUDA(cudaEventRecord(ev, w->st));
  RS_CUDA(cudaStreamWaitEvent(s, ev, 0));
  RS_CUDA(cudaEventDestroy(ev));
  k_ws_predict<<<grid_for(2 * nb, 256), 256, 0, s>>>(n, nb, w->Y.p, y, y + 2 * (size_t)nb);
  RS_LAUNCHED(1);
  RS_CUDA(cudaEventRecord(w->last, s));
  w->recorded = true;
}

// append (features, target) of a solved system to the dataset
void ws_record(sim_ws_s *w, int nx, int ny, int nz, const double *b, const double *kx, const double *sw,
               const double *yp, const double *sc, const double *y, cudaStream_t s) {
  std::lock_guard<std::mutex> guard(w->use);
  if (w->data.size() >= w->max_samples) return;
  dims d = {nx, ny, nz};
  int n = d.V();
  std::unique_ptr<sim_ws_s::sample> S(new sim_ws_s::sample());
  S->d = d;
  S->X.alloc((size_t)n * CIN_GPU);
  S->T.alloc((size_t)n * NPRED);
  k_ws_features<<<grid_for(n, 256), 256, 0, s>>>(n, b, kx, sw, yp, sc, S->X.p);
  k_ws_target<<<grid_for(2 * n, 256), 256, 0, s>>>(n, y, sc, S->T.p);
  RS_LAUNCHED(2);
  RS_CUDA(cudaStreamSynchronize(s));       // the sample is complete before another stream reads it
  w->data.push_back(std::move(S));
}

cudaStream_t ws_stream(sim_ws_s *w) { return w->st; }

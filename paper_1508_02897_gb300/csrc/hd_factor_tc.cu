// Block-Schur factorisation of every local PML problem (Eq. (pmlij)) on the tensor
// cores, for complex FP32 factors and boxes up to 192 cells wide.
//
// As in hd_factor.cu, each box is block tridiagonal along its grid rows and the
// solve needs S_j^{-1} for S_0 = D_0, S_j = D_j - L_j S_{j-1}^{-1} L_j (L_j diagonal,
// D_j tridiagonal, A complex symmetric).  Here each S_j (m x m) is inverted in place
// by blocked Gauss-Jordan elimination WITHOUT pivoting, in panels of 16 columns.
// On the Schur blocks of these PML problems the diagonal entry is the largest
// remaining one of its column at every step, so the diagonal pivots are the ones
// partial pivoting would pick; every pivot is still checked (below).
//
// The working matrix lives in tensor memory for the whole box (one CTA per SM):
// lane l holds row l, columns [0, NP) the real parts and [NP, 2 NP) the imaginary
// parts of rows 0..127 (NP = m rounded up to 16), and for m > 128 the lanes 0..mb-1
// of columns [2 NP, 2 NP + NB) and [2 NP + NB, 2 NP + 2 NB) hold the bottom-right
// block (rows and columns 128..m-1, mb = m - 128, NB = mb rounded up to 16).  The
// bottom-left block is not stored: Gauss-Jordan on a symmetric matrix keeps the
// eliminated block and the Schur complement symmetric and the two off-diagonal
// blocks negative transposes of each other, so W[r][c] for r >= 128 > c is +-W[c][r]
// (+ while both indices are still unprocessed, which is the only case read).
//
// Eliminating panel K (columns k0 .. k0+w-1) with C = W[:, K], P = C_K^{-1} (the
// w x w diagonal block inverted by the SIMT threads), X = C - E_K and
// Y^T = Z P (Z = C with already eliminated rows negated and rows K replaced by the
// identity; by the symmetry above this is P times the row panel) is one update
//     W <- W with columns K set to E_K,  then  W <- W - X Y,
// which gives all four parts of the in-place Gauss-Jordan step at once (pivot
// block P, row panel P W_KJ, column panel -W_IK P, trailing W_IJ - W_IK P W_KJ).
// W - X Y is a rank-16 complex update accumulated straight into the resident
// matrix by tcgen05.mma kind::f16: every real operand is split into three BF16
// pieces (x = h + m + l exactly to 2^-25 |x|, rounded to nearest), and the six
// products h h, h m, m h, h l, m m, l h of each real product give FP32-grade
// products (the neglected terms are below 2^-25); with FP32 accumulation in tensor
// memory the update matches FP32 arithmetic.  The complex product takes the four
// real products Xr Yr, Xi Yi, Xr Yi, Xi Yr, each accumulated into its real or
// imaginary plane with the sign stored in the operands (A = -Xr, -Xi; B = Yr, Yi,
// -Yi).  One panel is 24 MMAs for rows 0..127 (N = NP) and 24 for the bottom-right
// block (M = 128 rows starting at operand row 128, N = NB); for boxes wider than 128 the
// columns from the next panel on are updated first, and the others under that panel's copy,
// pivot block and A operand (a second A operand; every entry still receives the same
// products in the same order).
//
// What bounds it: the chain of the panels, one CTA per SM (tensor and shared memory are both
// full).  Cycles per panel of 16 columns at m = 176: copy 0.7K, pivot block 5.2K (sixteen
// dependent elimination steps, two per barrier; the A operand and the next row's band entries
// are formed beside it), B operand 3.6K, rows K 0.6K, waits for the first MMAs 2.5K; per grid
// row 15K to write S_j^{-1} out and rebuild.  64 boxes of 174: 21.6 ms with eight warps and
// the phases one after another, 16.5 ms with sixteen, 15.8 ms with the split update; 4096^2
// (1024 boxes of 176): 154 -> 118 -> 113 ms.
//
// Pivot check: within each diagonal block every pivot is compared with the other
// unprocessed entries of its column (and, for the first column of the panel, with
// all unprocessed rows below the panel); a pivot smaller than pivot_ratio times the
// largest of them, or a non-finite one, marks the box, and hd_factor_subdomains
// refactors marked boxes with the partially pivoted SIMT kernel right after this one.
//
// After the last panel, S_j^{-1} is read out of tensor memory once: written to the
// factor storage (full column-major, upper 16 x 16 tiles or TF32 planes; complex
// FP32 or FP16) and turned in place into S_{j+1} = D_{j+1} - L S_j^{-1} L, so the
// recursion runs on the FP32 values and storage rounding never feeds back.
#include <cuda_bf16.h>

#include "hd_internal.cuh"
#include "hd_tc.cuh"

namespace hd {

namespace {

constexpr int FX_THREADS = 512;   // 16 warps, four per lane quarter of tensor memory
constexpr int FX_MAXM = 192;     // 2 NP + 2 NB <= 512 tensor-memory columns
constexpr int FX_KP = 16;        // panel width = K of one kind::f16 MMA
constexpr int FX_ROWS = 192;     // rows of the B operand tiles and of the panel copy
constexpr int FX_AROWS = 256;    // rows of the A operand tiles (the bottom MMA reads rows 128..255)
constexpr uint32_t FX_ATILE = FX_AROWS * 32;   // bytes of one A tile: 16 BF16 per row
constexpr uint32_t FX_BTILE = FX_ROWS * 32;
constexpr int FX_NA = 6, FX_NBT = 9;           // A: -Xr, -Xi; B: Yr, Yi, -Yi; three pieces each
constexpr uint32_t FX_TMEM_COLS = 512;
constexpr int CLD = 17;          // row stride (entries) of the panel copy: conflict-free rows and columns

constexpr size_t kOffA = 0;
constexpr size_t kOffB = kOffA + 2 * (size_t)FX_NA * FX_ATILE;   // two A operands: the next panel's is formed under this one's MMAs
constexpr size_t kOffC = kOffB + (size_t)FX_NBT * FX_BTILE;
constexpr size_t kOffY = kOffC + sizeof(float2) * FX_ROWS * CLD;
constexpr size_t kOffG = kOffY + sizeof(float2) * FX_ROWS * CLD;
constexpr size_t kOffL = kOffG + sizeof(float2) * 2 * FX_KP * FX_KP;
constexpr size_t kOffD = kOffL + sizeof(float2) * FX_ROWS;
constexpr size_t kOffM = kOffD + sizeof(float2) * 3 * FX_ROWS;
constexpr size_t kSmem = kOffM + 48;

// (x0, x1) = h + m + l piecewise, BF16 pieces rounded to nearest (each remainder is
// exact in FP32), two values per conversion instruction; the pieces come packed as
// BF16 pairs (x0 in the low half).
__device__ __forceinline__ void split3x2(float x0, float x1, uint32_t &h, uint32_t &m, uint32_t &l) {
  const __nv_bfloat162 bh = __floats2bfloat162_rn(x0, x1);
  const float2 fh = __bfloat1622float2(bh);
  const float r0 = __fsub_rn(x0, fh.x), r1 = __fsub_rn(x1, fh.y);
  const __nv_bfloat162 bm = __floats2bfloat162_rn(r0, r1);
  const float2 fm = __bfloat1622float2(bm);
  const __nv_bfloat162 bl = __floats2bfloat162_rn(__fsub_rn(r0, fm.x), __fsub_rn(r1, fm.y));
  h = *reinterpret_cast<const uint32_t *>(&bh);
  m = *reinterpret_cast<const uint32_t *>(&bm);
  l = *reinterpret_cast<const uint32_t *>(&bl);
}

// Row r of an operand tile (16 BF16 values as 8 pairs) in the no-swizzle K-major layout:
// 8-row groups 256 bytes apart (SBO), the two 8-column core matrices 128 bytes apart (LBO).
__device__ __forceinline__ void put_row(unsigned char *tile, int r, const uint32_t *v) {
  unsigned char *p = tile + (r >> 3) * 256 + (r & 7) * 16;
  *reinterpret_cast<uint4 *>(p) = make_uint4(v[0], v[1], v[2], v[3]);
  *reinterpret_cast<uint4 *>(p + 128) = make_uint4(v[4], v[5], v[6], v[7]);
}

// Half a row (8 values: one 8-column core matrix, h = 0 or 1) split into three pieces, row r
// of tiles t, t+1, t+2.
__device__ __forceinline__ void put_split8(unsigned char *tiles, uint32_t tile_bytes, int t, int r, int half, const float *v) {
  uint32_t h[4], m[4], l[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) split3x2(v[2 * i], v[2 * i + 1], h[i], m[i], l[i]);
  unsigned char *p = tiles + (size_t)t * tile_bytes + (r >> 3) * 256 + (r & 7) * 16 + half * 128;
  *reinterpret_cast<uint4 *>(p) = make_uint4(h[0], h[1], h[2], h[3]);
  *reinterpret_cast<uint4 *>(p + tile_bytes) = make_uint4(m[0], m[1], m[2], m[3]);
  *reinterpret_cast<uint4 *>(p + 2 * (size_t)tile_bytes) = make_uint4(l[0], l[1], l[2], l[3]);
}

// Splits 16 values and writes the three pieces as row r of tiles t, t+1, t+2.
__device__ __forceinline__ void put_split(unsigned char *tiles, uint32_t tile_bytes, int t, int r, const float *v) {
  uint32_t h[8], m[8], l[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) split3x2(v[2 * i], v[2 * i + 1], h[i], m[i], l[i]);
  put_row(tiles + (size_t)t * tile_bytes, r, h);
  put_row(tiles + (size_t)(t + 1) * tile_bytes, r, m);
  put_row(tiles + (size_t)(t + 2) * tile_bytes, r, l);
}

__device__ __forceinline__ float cabs2f(float2 a) { return a.x * a.x + a.y * a.y; }

// 1 / x for the pivots: the hardware approximation refined by one Newton step
// (r (2 - x r)), within about one ulp for normal x; a zero or non-finite x is caught by
// the pivot check before the result matters.
__device__ __forceinline__ float recip(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r * fmaf(-x, r, 2.f);
}

// Stored entry (r, c) of S_j^{-1} in the full or tensor-core layouts (zero outside m x m).
template <typename S, int LAY>
__device__ __forceinline__ void emit(S *slot, int r, int c, float2 v, int m, int ldm, int mp8) {
  if (LAY == LAY_FULL) {
    if (r < m && c < m) slot[(int64_t)c * ldm + r] = store_c<S>(v);
  } else {   // LAY_TC: chunk c/8, real then imaginary plane [mp8/8][2][8][4], TF32;
             // LAY_TC3: then the real and imaginary remainders, TF32
    if (r >= mp8 || c >= mp8) return;
    if (r >= m || c >= m) v = make_float2(0.f, 0.f);
    float *F = reinterpret_cast<float *>(slot);
    const int per = 8 * mp8;
    constexpr int NPL = LAY == LAY_TC3 ? 4 : 2;
    const int64_t o = (int64_t)(c >> 3) * NPL * per + (r >> 3) * 64 + ((c >> 2) & 1) * 32 + (r & 7) * 4 + (c & 3);
    const float hr = tf32_round(v.x), hi = tf32_round(v.y);
    F[o] = hr;
    F[o + per] = hi;
    if (LAY == LAY_TC3) {
      F[o + 2 * per] = tf32_round(v.x - hr);
      F[o + 3 * per] = tf32_round(v.y - hi);
    }
  }
}

}  // namespace

size_t factor_tc_smem_bytes() { return kSmem; }

template <typename S, int LAY>
__global__ void __launch_bounds__(FX_THREADS, 1)
k_factor_tc(const SubDev *__restrict__ subs, int nsub, const double2 *__restrict__ pool, const double *__restrict__ k2,
            int NX, double h2, S *__restrict__ factor, float tau2, int32_t *__restrict__ flags, int32_t *status) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char *At = smem_raw + kOffA;
  unsigned char *Bt = smem_raw + kOffB;
  float2 *Cs = reinterpret_cast<float2 *>(smem_raw + kOffC);   // [FX_ROWS][CLD] panel columns
  float2 *Ys = reinterpret_cast<float2 *>(smem_raw + kOffY);   // [FX_ROWS][CLD] Y^T of the panel
  float2 *G = reinterpret_cast<float2 *>(smem_raw + kOffG);    // [2][16][16] pivot block
  float2 *dS = reinterpret_cast<float2 *>(smem_raw + kOffD);   // [3][FX_ROWS] band entries of the next row's D
  float2 *lS = reinterpret_cast<float2 *>(smem_raw + kOffL);   // [FX_ROWS] coupling of the next row
  uint64_t *mbar = reinterpret_cast<uint64_t *>(smem_raw + kOffM);
  uint64_t *fin = mbar + 2;   // the release of tensor memory after a timeout
  uint32_t *tholder = reinterpret_cast<uint32_t *>(fin + 1);
  volatile int *sflag = reinterpret_cast<volatile int *>(tholder + 1);
  volatile int *abort_flag = sflag + 1;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  if (tid == 0) {
    tc::bar_init(mbar, 1);
    tc::bar_init(mbar + 1, 1);
    tc::bar_init(fin, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc::su32(tholder)),
                 "r"(FX_TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tmem = *tholder;
  // this warp's lane quarter in tensor memory, which it shares with three others
  const int q4 = warp & 3, part = warp >> 2;
  const uint32_t tq = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
  const bool issuer = warp == FX_THREADS / 32 - 1 && lane == 0;   // of the MMAs (its warp has no other work while they are issued)
  uint32_t nphase = 0, nrest = 0;   // completed phases of mbar[0] and mbar[1]
  int abuf = 0;
  bool alive = true, rest = false;   // rest: MMAs of mbar[1] are in flight

  for (int box = blockIdx.x; box < nsub && alive; box += gridDim.x) {
    const SubDev s = subs[box];
    const int m = s.ex, rows = s.ey;
    const int NP = (m + 15) & ~15;
    const int mb = m > 128 ? m - 128 : 0;
    const int NB = (mb + 15) & ~15;
    const int mt = NP / 16, mp8 = (m + 7) & ~7;
    const double2 *a1c = pool + s.aoff;
    const double2 *ia1f = a1c + m;
    const double2 *a2c = ia1f + m + 1;
    const double2 *ia2f = a2c + rows;
    S *Fs = factor + s.foff;
    const int64_t slot_elems = LAY == LAY_SYM ? (int64_t)mt * (mt + 1) / 2 * 256
                                              : (LAY == LAY_TC    ? (int64_t)mp8 * mp8
                                                 : LAY == LAY_TC3 ? 2 * (int64_t)mp8 * mp8
                                                                  : (int64_t)m * s.ldm);

    // operand tiles and the panel copy start at zero: rows >= m are never written
    for (int i = tid; i < (int)(kOffG / 16); i += FX_THREADS)
      reinterpret_cast<uint4 *>(smem_raw)[i] = make_uint4(0u, 0u, 0u, 0u);
    if (tid == 0) *sflag = 0;

    // ---- S_0 = D_0 into tensor memory (the three band entries of a row once per row in shared
    //      memory; the four warps of a lane quarter take every fourth chunk of 16 columns)
    auto band_row = [&](int r, int jr) {   // entries (r, r - 1), (r, r), (r, r + 1) of D_jr
      const double *k2row = k2 + (int64_t)(s.ey0 + jr) * NX + s.ex0;
#pragma unroll
      for (int t = 0; t < 3; ++t) {
        const int c = r - 1 + t;
        dS[t * FX_ROWS + r] = r < m && c >= 0 && c < m ? d_entry<float2, float>(r, c, jr, a1c, ia1f, a2c, ia2f, k2row, h2)
                                                       : make_float2(0.f, 0.f);
      }
    };
    __syncthreads();   // (the previous box's write-out has finished reading dS)
    if (tid < FX_ROWS) band_row(tid, 0);
    __syncthreads();
    for (int reg = 0; reg < 2; ++reg) {
      const bool top = reg == 0;
      if (!top && (mb == 0 || q4 >= 2)) break;
      const int r = (top ? 0 : 128) + 32 * q4 + lane;
      const int ncol = top ? NP : NB, cbase = top ? 0 : 128;
      const uint32_t tre = top ? tq : tq + 2 * NP, tim = top ? tq + NP : tq + 2 * NP + NB;
      const float2 d0 = dS[r], d1 = dS[FX_ROWS + r], d2 = dS[2 * FX_ROWS + r];
      for (int cc = 16 * part; cc < ncol; cc += 64) {
        float re[16], im[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const int t = cbase + cc + i - r + 1;   // band position 0, 1, 2, or outside
          const float2 v = t == 0 ? d0 : (t == 1 ? d1 : (t == 2 ? d2 : make_float2(0.f, 0.f)));
          re[i] = v.x;
          im[i] = v.y;
        }
        tc::tmem_st16(tre + cc, re);
        tc::tmem_st16(tim + cc, im);
      }
    }
    tc::tmem_wait_st();

    for (int j = 0; j < rows && alive; ++j) {
      const bool more = j + 1 < rows;
      __syncthreads();   // the previous row's write-out has finished reading lS
      // coupling of the next grid row (used after the last panel)
      if (more)
        for (int r = tid; r < FX_ROWS; r += FX_THREADS) {
          float2 l = make_float2(0.f, 0.f);
          if (r < m) {
            const double2 ld = cmul(a1c[r], ia2f[j + 1]);
            l = make_float2((float)ld.x, (float)ld.y);
          }
          lS[r] = l;
        }

      for (int k0 = 0; k0 < m; k0 += FX_KP) {
        const int w = min(FX_KP, m - k0);
        // ---- A. copy the panel columns C = W[:, K] into shared memory.  Behind a panel whose
        //      remaining MMAs still run, their issuer's warp leaves A and B to the others (its
        //      instructions block while the tensor cores are busy) and joins them before C.
        const bool follow = rest, ahead = !(follow && warp == FX_THREADS / 32 - 1);
        if (!follow) {
          tc::fence_before();
          __syncthreads();
          tc::fence_after();
        }
        if (ahead) {
          if (part == 0) {
            float re[16], im[16];
            tc::tmem_ld16_nw(tq + k0, re);
            tc::tmem_ld16_nw(tq + NP + k0, im);
            tc::tmem_wait_ld();
  #pragma unroll
            for (int i = 0; i < 16; ++i) Cs[tid * CLD + i] = make_float2(re[i], im[i]);
          } else if (mb > 0) {
            if (k0 >= 128) {
              if (part == 1 && q4 < 2) {   // bottom rows from the bottom-right block
                const int rb = 32 * q4 + lane;
                float re[16], im[16];
                tc::tmem_ld16_nw(tq + 2 * NP + (k0 - 128), re);
                tc::tmem_ld16_nw(tq + 2 * NP + NB + (k0 - 128), im);
                tc::tmem_wait_ld();
  #pragma unroll
                for (int i = 0; i < 16; ++i) Cs[(128 + rb) * CLD + i] = make_float2(re[i], im[i]);
              }
            } else if (q4 == (k0 >> 5)) {
              // bottom rows of panel columns k < 128: W[128 + c'][k] = W[k][128 + c'], held by lane k
              const int row = 32 * q4 + lane;
              const bool mine = row >= k0 && row < k0 + FX_KP;
              for (int cc = 16 * (part - 1); cc < NB && part < 3; cc += 32) {
                float re[16], im[16];
                tc::tmem_ld16_nw(tq + 128 + cc, re);
                tc::tmem_ld16_nw(tq + NP + 128 + cc, im);
                tc::tmem_wait_ld();
                if (mine)
  #pragma unroll
                  for (int i = 0; i < 16; ++i) {
                    const int cp = cc + i;
                    Cs[(128 + cp) * CLD + (row - k0)] = cp < mb ? make_float2(re[i], im[i]) : make_float2(0.f, 0.f);
                  }
              }
            }
          }
          if (follow) asm volatile("bar.sync 3, %0;" ::"n"(FX_THREADS - 32) : "memory");
          else __syncthreads();

          // ---- B. side by side: warps 8..13 the A operand, warps 0..7 the pivot block
          if (warp >= 8) {
            // A = -X, X = C outside rows K and zero on rows K (their new values are stored
            // directly), one row per thread; and the first pivot of the panel against every
            // unprocessed row below the panel
            unsigned char *Aw = At + (size_t)abuf * FX_NA * FX_ATILE;
            const int r = tid - 256, kr = r - k0;
            if (r < m) {
              const bool inK = kr >= 0 && kr < w;
              float vr[16], vi[16];
  #pragma unroll
              for (int i = 0; i < 16; ++i) {
                const float2 c = Cs[r * CLD + i];
                vr[i] = inK ? 0.f : -c.x;
                vi[i] = inK ? 0.f : -c.y;
              }
              put_split(Aw, FX_ATILE, 0, r, vr);
              put_split(Aw, FX_ATILE, 3, r, vi);
              if (r >= k0 + w && !(cabs2f(Cs[k0 * CLD]) >= tau2 * cabs2f(Cs[r * CLD]))) *sflag = 1;
            }
            // the band of the next row's D, on the FP64 pipe while the pivot block is inverted
            if (k0 == 0 && more && r < FX_ROWS) band_row(r, j + 1);
          } else {
            // P = C_K^{-1} (w x w) by Gauss-Jordan without pivoting, one entry per thread
            // (i, jj) = (tid / 16, tid % 16), two alternating shared copies.  Two elimination
            // steps k, k+1 per barrier: every thread loads the nine entries it needs and
            // applies both in-place steps to its own entry (the same arithmetic as two
            // separate steps).  In-place value of entry (x, y) after a step with pivot index k:
            // the inverse pivot on (k, k), a_ky / pivot on row k, -a_xk / pivot on column k, else
            // a_xy - a_xk (a_ky / pivot); formed without branches, every case selected from the
            // few products the entries share.  Each pivot is checked by the threads of the
            // unprocessed entries below it.  (Two entries per thread on four warps: 6.8K cycles per
            // panel instead of 5.3K: the instructions of a thread, not the shared work, set the time.)
            const int i = tid >> 4, jj = tid & 15;
            float2 *B0 = G, *B1 = G + 256;
            auto sync8 = []() { asm volatile("bar.sync 2, 256;" ::: "memory"); };
            auto neg = [](float2 v) { return make_float2(-v.x, -v.y); };
            auto sel = [](bool c, float2 x, float2 y) { return make_float2(c ? x.x : y.x, c ? x.y : y.y); };
            B0[tid] = (i < w && jj < w) ? Cs[(k0 + i) * CLD + jj] : make_float2(i == jj ? 1.f : 0.f, 0.f);
            sync8();
            int par = 0;
  #pragma unroll 1
            for (int k = 0; k < w; k += 2, par ^= 1) {
              const float2 *src = par ? B1 : B0;
              float2 *dst = par ? B0 : B1;
              const int k1 = min(k + 1, 15);
              const float2 piv = src[k * 16 + k], aik = src[i * 16 + k], akj = src[k * 16 + jj], aij = src[tid];
              const float2 a_i1 = src[i * 16 + k1], a_k1 = src[k * 16 + k1];
              const float2 a_1j = src[k1 * 16 + jj], a_1k = src[k1 * 16 + k], a_11 = src[k1 * 16 + k1];
              const float p2 = cabs2f(piv);
              const float rd = recip(p2);   // 1 / pivot = conj(pivot) / |pivot|^2
              const float2 ip = make_float2(piv.x * rd, -piv.y * rd);
              const float2 tj = cmul(akj, ip), t1 = cmul(a_k1, ip);
              float2 v = sel(i == k, sel(jj == k, ip, tj), sel(jj == k, neg(cmul(aik, ip)), cfms(aik, tj, aij)));
              bool bad = (jj == k && i > k && i < w && !(p2 >= tau2 * cabs2f(aik))) || (tid == 0 && (!(p2 > 0.f) || !isfinite(p2)));
              if (k + 1 < w) {
                // the second step on the values after the first
                const float2 vi1 = sel(i == k, t1, cfms(aik, t1, a_i1));                    // entry (i, k+1)
                const float2 v1j = sel(jj == k, neg(cmul(a_1k, ip)), cfms(a_1k, tj, a_1j));   // entry (k+1, jj)
                const float2 piv1 = cfms(a_1k, t1, a_11);                                   // next pivot
                const float q2 = cabs2f(piv1);
                const float rd1 = recip(q2);
                const float2 ip1 = make_float2(piv1.x * rd1, -piv1.y * rd1);
                const float2 t2 = cmul(v1j, ip1);
                bad = bad || (jj == k1 && i > k1 && i < w && !(q2 >= tau2 * cabs2f(vi1))) ||
                      (tid == 0 && (!(q2 > 0.f) || !isfinite(q2)));
                v = sel(i == k1, sel(jj == k1, ip1, t2), sel(jj == k1, neg(cmul(vi1, ip1)), cfms(vi1, t2, v)));
              }
              if (bad) *sflag = 1;
              dst[tid] = v;
              sync8();
            }
            // P into the first copy, zero outside w x w (each thread moves its own entry)
            const float2 *res = par ? B1 : B0;
            const float2 pv = (i < w && jj < w) ? res[tid] : make_float2(0.f, 0.f);
            B0[tid] = pv;
          }
        }
        // the previous panel's remaining MMAs read the B operand and write W: done from here on
        if (rest && !tc::bar_spin(mbar + 1, nrest & 1u, abort_flag)) *abort_flag = 1;
        if (rest) ++nrest;
        rest = false;
        tc::fence_after();
        __syncthreads();
        if (*abort_flag) {   // (set before the barrier: every thread leaves here)
          if (tid == 0) atomicOr(status, ST_TIMEOUT);
          alive = false;
          break;
        }
        const float2 *Pm = G;   // P[i][kk] at Pm[i * 16 + kk], zero outside w x w

        // ---- C. the B operand Y^T = Z P (three BF16 pieces), half a row per thread: columns
        //      8 h .. 8 h + 7 of row r; Y^T also goes to Ys for the rows K
        {
          // (warps 0..5 and 10..15: three on each scheduler)
          const int h = warp >= 10, r = h ? tid - 320 : tid, kr = r - k0;
          if ((h || warp < 6) && r < m) {
            const bool inK = kr >= 0 && kr < w;
            float2 y[8];
            if (inK) {
#pragma unroll
              for (int kk = 0; kk < 8; ++kk) y[kk] = Pm[kr * 16 + 8 * h + kk];
            } else {
              // y = zs C[r] P: q outer, 8 independent accumulator chains
#pragma unroll
              for (int kk = 0; kk < 8; ++kk) y[kk] = make_float2(0.f, 0.f);
#pragma unroll 4
              for (int q = 0; q < 16; ++q) {
                const float4 *prow = reinterpret_cast<const float4 *>(Pm + q * 16 + 8 * h);
                const float2 cq = Cs[r * CLD + q];
#pragma unroll
                for (int k2 = 0; k2 < 4; ++k2) {
                  const float4 pp = prow[k2];
                  y[2 * k2] = cfma(cq, make_float2(pp.x, pp.y), y[2 * k2]);
                  y[2 * k2 + 1] = cfma(cq, make_float2(pp.z, pp.w), y[2 * k2 + 1]);
                }
              }
              if (r < k0)
#pragma unroll
                for (int kk = 0; kk < 8; ++kk) y[kk] = make_float2(-y[kk].x, -y[kk].y);
            }
            float vr[8], vi[8];
#pragma unroll
            for (int kk = 0; kk < 8; ++kk) {
              vr[kk] = y[kk].x;
              vi[kk] = y[kk].y;
              Ys[r * CLD + 8 * h + kk] = y[kk];
            }
            put_split8(Bt, FX_BTILE, 0, r, h, vr);
            put_split8(Bt, FX_BTILE, 3, r, h, vi);
#pragma unroll
            for (int kk = 0; kk < 8; ++kk) vi[kk] = -vi[kk];
            put_split8(Bt, FX_BTILE, 6, r, h, vi);
          }
        }
        __syncthreads();
        // rows K take their new values directly, W[k][:] = Y[k - k0][:] (P on the diagonal
        // block, P W_KJ elsewhere: no cancellation), and every other row gets zero in the
        // columns K, which the update below fills with -C P.  Tensor-memory stores are
        // warp-collective, so the warp holding rows K rewrites whole rows: its other lanes
        // store back what they hold (zero in the columns K).
        {
          const int q = q4;
          const bool top_rmw = k0 < 128 && q == (k0 >> 5);
          const bool bot_rmw = k0 >= 128 && q == ((k0 - 128) >> 5);
          // columns K of rows outside K: zero (top rows: warps 0-3; bottom rows: warps 4, 5)
          if (warp < 4 && !top_rmw) {
            const float z[16] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            tc::tmem_st16(tq + k0, z);
            tc::tmem_st16(tq + NP + k0, z);
          } else if (part == 1 && q < 2 && k0 >= 128 && !bot_rmw) {
            const float z[16] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            tc::tmem_st16(tq + 2 * NP + (k0 - 128), z);
            tc::tmem_st16(tq + 2 * NP + NB + (k0 - 128), z);
          }
          if (top_rmw || bot_rmw) {
            // the four warps of this lane quarter rewrite the rows of K, a quarter of the columns each
            const int rrow = top_rmw ? 32 * q + lane : 128 + 32 * q + lane;
            const int kr = rrow - k0;
            const bool inK = kr >= 0 && kr < w;
            const int ncol = top_rmw ? NP : NB, cb = top_rmw ? 0 : 128, kc = k0 - cb;
            const int nch = ncol / 16;
            const int ch0 = nch * part / 4, ch1 = nch * (part + 1) / 4;
            const uint32_t tre = top_rmw ? tq : tq + 2 * NP, tim = top_rmw ? tq + NP : tq + 2 * NP + NB;
            for (int ch = ch0; ch < ch1; ++ch) {
              float re[16], im[16];
              const int cc = 16 * ch;
              tc::tmem_ld16_nw(tre + cc, re);
              tc::tmem_ld16_nw(tim + cc, im);
              tc::tmem_wait_ld();
              {
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                  if (inK) {
                    const float2 v = Ys[(cb + cc + i) * CLD + kr];
                    re[i] = v.x;
                    im[i] = v.y;
                  } else if (cc == kc) {
                    re[i] = 0.f;
                    im[i] = 0.f;
                  }
                }
                tc::tmem_st16(tre + cc, re);
                tc::tmem_st16(tim + cc, im);
              }
            }
          }
        }
        tc::tmem_wait_st();
        tc::fence_async_smem();
        tc::fence_before();
        __syncthreads();

        // ---- D. W -= X Y on the tensor cores (one thread issues).  The columns that the next
        //      panel copies come first, with a commit of their own; the others run while that
        //      panel's copy, pivot block and A operand are formed.  Every entry still receives its
        //      24 products in the same order.
        const int kn = k0 + FX_KP;   // next panel
        const bool last = kn >= m, whole = last || mb == 0;   // (up to 128 wide the split costs more than it hides)
        if (issuer) {
          tc::fence_after();
          const uint32_t a0 = tc::su32(At) + (uint32_t)abuf * FX_NA * FX_ATILE, b0 = tc::su32(Bt);
          // columns c0 .. c0 + n - 1 of rows 0..127 (part 0) or of the bottom-right block (part 1)
          auto update = [&](int bottom, int c0, int n) {
            if (n <= 0) return;
            const uint32_t dr = tmem + (bottom ? 2 * NP : 0) + c0, di = dr + (bottom ? NB : NP);
            const uint32_t ro = bottom ? 16 * 256 : 0;   // operand row 128: 16 groups of 8 rows
            const uint32_t co = ro + (uint32_t)(c0 >> 3) * 256;
            const uint32_t id = tc::idesc_bf16(128, (uint32_t)n);
#pragma unroll
            for (int pq = 0; pq < 6; ++pq) {
              // piece pairs (p, q) with p + q <= 2: (0,0) (0,1) (1,0) (0,2) (1,1) (2,0)
              const int p = pq == 2 ? 1 : (pq == 4 ? 1 : (pq == 5 ? 2 : 0));
              const int q = pq == 1 ? 1 : (pq == 3 ? 2 : (pq == 4 ? 1 : 0));
              const uint64_t axr = tc::mdesc(a0 + (uint32_t)p * FX_ATILE + ro, 128, 256);
              const uint64_t axi = tc::mdesc(a0 + (uint32_t)(3 + p) * FX_ATILE + ro, 128, 256);
              const uint64_t byr = tc::mdesc(b0 + (uint32_t)q * FX_BTILE + co, 128, 256);
              const uint64_t byi = tc::mdesc(b0 + (uint32_t)(3 + q) * FX_BTILE + co, 128, 256);
              const uint64_t byn = tc::mdesc(b0 + (uint32_t)(6 + q) * FX_BTILE + co, 128, 256);
              tc::mma_bf16(dr, axr, byr, id, 1u);   // -Xr Yr
              tc::mma_bf16(dr, axi, byn, id, 1u);   // +Xi Yi
              tc::mma_bf16(di, axr, byi, id, 1u);   // -Xr Yi
              tc::mma_bf16(di, axi, byr, id, 1u);   // -Xi Yr
            }
          };
          if (whole) {
            update(0, 0, NP);
            if (mb > 0) update(1, 0, NB);
            tc::mma_commit(mbar);
          } else {
            // (one range: an instruction takes about as long for 16 columns as for 128; the rows
            // 128.. of a panel left of column 128 come from the columns 128.. by symmetry)
            update(0, kn, NP - kn);
            if (kn >= 128) update(1, kn - 128, NB - (kn - 128));
            tc::mma_commit(mbar);
            update(0, 0, kn);
            if (mb > 0) update(1, 0, kn >= 128 ? kn - 128 : NB);
            tc::mma_commit(mbar + 1);
          }
        }
        rest = !whole;
        abuf ^= 1;
        if (!tc::bar_spin(mbar, nphase & 1u, abort_flag)) *abort_flag = 1;
        ++nphase;
        tc::fence_after();
        if (whole) {   // (behind a split update the next panel starts from each thread's own wait: no barrier between)
          __syncthreads();
          if (*abort_flag) {
            if (tid == 0) atomicOr(status, ST_TIMEOUT);
            alive = false;
            break;
          }
        }
      }
      if (!alive) break;

      // ---- write S_j^{-1} out and turn it into S_{j+1} = D_{j+1} - L S_j^{-1} L in place
      S *slot = Fs + (int64_t)j * slot_elems;
      const int ldm = s.ldm;
      // the four warps of a lane quarter split the 16-column chunks of their rows: rows 0..127,
      // and for the quarters 0 and 1 also the bottom-right block (rows 128..m-1)
      {
        const int q = q4;
        const int nchT = NP / 16, nchB = q < 2 ? NB / 16 : 0, nch = nchT + nchB;
        const int t0 = nch * part / 4, t1 = nch * (part + 1) / 4;
        for (int reg = 0; reg < 2; ++reg) {
          const bool top = reg == 0;
          const int ch0 = top ? min(t0, nchT) : max(t0 - nchT, 0), ch1 = top ? min(t1, nchT) : max(t1 - nchT, 0);
          if (ch0 >= ch1) continue;
          const int r = top ? 32 * q + lane : 128 + 32 * q + lane;
          const int cbase = top ? 0 : 128;
          const uint32_t tre = top ? tq : tq + 2 * NP, tim = top ? tq + NP : tq + 2 * NP + NB;
          const int I = r >> 4, rr = r & 15;
          const float2 lr = lS[r];
          const float2 d0 = dS[r], d1 = dS[FX_ROWS + r], d2 = dS[2 * FX_ROWS + r];   // D_{j+1} in row r
#pragma unroll 1
          for (int ch = ch0; ch < ch1; ++ch) {
            float re[16], im[16];
            const int cc = 16 * ch;
            tc::tmem_ld16_nw(tre + cc, re);
            tc::tmem_ld16_nw(tim + cc, im);
            tc::tmem_wait_ld();
            {
              const int c0 = cbase + cc;
              if (LAY == LAY_SYM) {
                const int J = c0 >> 4;
                if (J >= I && r < 16 * mt) {
                  S *tile = slot + (int64_t)(J * (J + 1) / 2 + I) * 256;
#pragma unroll
                  for (int i = 0; i < 16; ++i) {
                    const int c = c0 + i;
                    const float2 v = (r < m && c < m) ? make_float2(re[i], im[i]) : make_float2(0.f, 0.f);
                    if (J > I || i >= rr) tile[sym_pos<S>(rr, i)] = store_c<S>(v);
                    if (J == I && i > rr) tile[sym_pos<S>(i, rr)] = store_c<S>(v);
                  }
                }
              } else {
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                  const int c = c0 + i;
                  const float2 v = make_float2(re[i], im[i]);
                  emit<S, LAY>(slot, r, c, v, m, ldm, mp8);
                  if (top && c >= 128) emit<S, LAY>(slot, c, r, v, m, ldm, mp8);   // bottom-left block
                }
              }
              if (more) {
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                  const int c = c0 + i;
                  float2 v = make_float2(0.f, 0.f);
                  if (r < m && c < m) {
                    const int t = c - r + 1;   // band position 0, 1, 2, or outside
                    const float2 d = t == 0 ? d0 : (t == 1 ? d1 : (t == 2 ? d2 : make_float2(0.f, 0.f)));
                    v = cfms(cmul(lr, make_float2(re[i], im[i])), lS[c], d);
                  }
                  re[i] = v.x;
                  im[i] = v.y;
                }
                tc::tmem_st16(tre + cc, re);
                tc::tmem_st16(tim + cc, im);
              }
            }
          }
        }
        tc::tmem_wait_st();
      }
    }
    __syncthreads();
    if (tid == 0) flags[box] = *sflag;
  }

  // ---- release tensor memory once no MMA is in flight
  tc::fence_before();
  __syncthreads();
  if (!alive && issuer) {
    // (on a barrier of its own: a panel's barrier that timed out is still in the phase the count has
    // left behind, and the parity of the next one would pass at once)
    tc::mma_commit(fin);   // arrives when every MMA issued so far has completed
    tc::bar_drain(fin, 0);
  }
  __syncthreads();
  tc::fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(FX_TMEM_COLS) : "memory");
}

template <typename S, int LAY>
static cudaError_t launch_tc(hd_ctx *ctx, void *factor, float tau2, cudaStream_t st) {
  cudaError_t e = allow_smem(k_factor_tc<S, LAY>, kSmem);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 152;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int grid = std::min(ctx->nsub, sms);   // one CTA per SM (tensor memory and shared memory both full)
  k_factor_tc<S, LAY><<<grid, FX_THREADS, kSmem, st>>>(ctx->d_subs, ctx->nsub, ctx->d_lpool, ctx->d_k2, ctx->NX,
                                                       ctx->h * ctx->h, reinterpret_cast<S *>(factor), tau2,
                                                       ctx->d_fflag, ctx->d_status);
  return cudaGetLastError();
}

bool factor_tc_supported(const hd_ctx *ctx) { return ctx->prec != HD_C128 && ctx->max_m <= FX_MAXM; }

cudaError_t launch_factor_tc(hd_ctx *ctx, void *factor, cudaStream_t st) {
  const float tau2 = (float)(ctx->fpivot * ctx->fpivot);
  if (ctx->tc3) return launch_tc<float2, LAY_TC3>(ctx, factor, tau2, st);
  if (ctx->tc) return launch_tc<float2, LAY_TC>(ctx, factor, tau2, st);
  if (ctx->prec == HD_C64)
    return ctx->sym ? launch_tc<float2, LAY_SYM>(ctx, factor, tau2, st) : launch_tc<float2, LAY_FULL>(ctx, factor, tau2, st);
  if (ctx->prec == HD_C64_B)
    return ctx->sym ? launch_tc<__nv_bfloat162, LAY_SYM>(ctx, factor, tau2, st)
                    : launch_tc<__nv_bfloat162, LAY_FULL>(ctx, factor, tau2, st);
  return ctx->sym ? launch_tc<__half2, LAY_SYM>(ctx, factor, tau2, st) : launch_tc<__half2, LAY_FULL>(ctx, factor, tau2, st);
}

}  // namespace hd

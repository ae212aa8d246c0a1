// Preconditioner application, Eq. (ddm0) + Eq. (pc):
//   z = sum_ij E_ij^T A_ij^{-1} X_ij r.
//
// k_subst (one CTA per box) fuses the restriction X_ij r (a gather of the
// owned part of each grid row of the box straight from the global residual)
// with the forward block substitution
//     w_0 = S_0^{-1} rho_0,   w_j = S_j^{-1} (rho_j - L_j w_{j-1}),
// and the back substitution
//     x_last = w_last,        x_j = w_j - S_j^{-1} (U_j x_{j+1}),
// leaving the local solution over the whole box (PML area included) in the
// staging buffer.  Each step is one m x m complex GEMV against a stored
// S_j^{-1}, so the kernel streams 2 rows - 1 dense m x m blocks per box: it is
// HBM-bound.  The stream of factor blocks does not depend on the vectors, so a
// producer warp copies them ahead with bulk asynchronous copies
// (cp.async.bulk, completion counted on an mbarrier) into a ring of NS shared
// memory stages of CH columns each, across step boundaries; the consumer
// warps accumulate y[a] = sum_b S[a][b] v[b] from shared memory (thread t owns
// outputs a = t + CT*e) and release each stage on its "empty" mbarrier.
// Every wait is bounded: on timeout the kernel flags ST_TIMEOUT, stops issuing
// copies, lets every warp run to the end, and the producer waits for its own
// copies still in flight before the CTA exits.
//
// k_gather then forms z cell by cell as a fixed-order sum over the (at most
// 3 x 3, in practice 2 x 2) boxes whose extent covers the cell: deterministic,
// no atomics.
#include "hd_internal.cuh"
#include "hd_tc.cuh"

namespace hd {

constexpr uint32_t kWaitLimit = 1u << 24;   // try_wait rounds before a wait gives up

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait; false on timeout or when another warp already gave up.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, volatile int *abort_flag) {
  for (uint32_t it = 0; it < kWaitLimit; ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((it & 255u) == 255u && *abort_flag) return false;
  }
  return false;
}
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void consumer_sync(int nthreads) {
  asm volatile("bar.sync 1, %0;" ::"r"(nthreads) : "memory");
}

// Columns of a stored factor block per ring stage (about 11 KB at m = 176).
template <typename S> __host__ __device__ constexpr int chunk_cols() {
  return sizeof(S) == 16 ? 4 : (sizeof(S) == 8 ? 8 : 16);
}

// Output a handled by consumer thread t, slot e: with two outputs per thread they
// are adjacent (one 2-entry vector load per stored column), else one per thread.
template <int CT, int NA> __device__ __forceinline__ int out_index(int t, int e) {
  return NA == 2 ? 2 * t + e : t + CT * e;
}

// Two adjacent stored entries p[0], p[1] (16-byte aligned for float2 / 8 for half2 and bfloat162).
template <typename T, typename S> __device__ __forceinline__ void load_pair(const S *p, T &v0, T &v1) {
  v0 = load_c<T>(p[0]);
  v1 = load_c<T>(p[1]);
}
template <> __device__ __forceinline__ void load_pair<float2, float2>(const float2 *p, float2 &v0, float2 &v1) {
  const float4 q = *reinterpret_cast<const float4 *>(p);
  v0 = make_float2(q.x, q.y);
  v1 = make_float2(q.z, q.w);
}
template <> __device__ __forceinline__ void load_pair<float2, __half2>(const __half2 *p, float2 &v0, float2 &v1) {
  const uint2 q = *reinterpret_cast<const uint2 *>(p);
  v0 = __half22float2(*reinterpret_cast<const __half2 *>(&q.x));
  v1 = __half22float2(*reinterpret_cast<const __half2 *>(&q.y));
}
template <>
__device__ __forceinline__ void load_pair<float2, __nv_bfloat162>(const __nv_bfloat162 *p, float2 &v0, float2 &v1) {
  const uint2 q = *reinterpret_cast<const uint2 *>(p);
  v0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&q.x));
  v1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&q.y));
}

// Shared memory layout: ring [NS][CH*ldmax] (stored type S) | vs [NR][ldmax] (compute type T) |
// full[NS] | empty[NS] | abort
template <typename T, typename S>
__host__ __device__ inline size_t subst_smem(int ns, int ldmax, int nr) {
  size_t stage = (size_t)chunk_cols<S>() * ldmax * sizeof(S);
  size_t o = (size_t)ns * stage + (size_t)nr * ldmax * sizeof(T);
  o = (o + 15) & ~(size_t)15;
  return o + 2 * (size_t)ns * sizeof(uint64_t) + 16;
}

// One CTA per (box, group of NR right-hand sides): every factor block is read
// once per group and applied to NR vectors.
template <typename R, typename S, int CT, int NA, int NR>
__global__ void __launch_bounds__(CT + 32)
k_subst(const SubDev *__restrict__ subs, const double2 *__restrict__ pool, const S *__restrict__ factor,
        const double2 *__restrict__ rg, int NX, int64_t vec_stride, C<R> *__restrict__ staging, int64_t stg_stride,
        int nrhs, int NS, int ldmax, int32_t *status) {
  using T = C<R>;
  constexpr int CH = chunk_cols<S>();
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const SubDev s = subs[blockIdx.y];
  const int m = s.ex, rows = s.ey, ldm = s.ldm;
  const int r0 = blockIdx.x * NR;
  const size_t stage_elems = (size_t)CH * ldmax;
  S *ring = reinterpret_cast<S *>(smem_raw);
  T *vs = reinterpret_cast<T *>(ring + (size_t)NS * stage_elems);     // [NR][ldmax]
  size_t off = (size_t)NS * stage_elems * sizeof(S) + (size_t)NR * ldmax * sizeof(T);
  off = (off + 15) & ~(size_t)15;
  uint64_t *full = reinterpret_cast<uint64_t *>(smem_raw + off);
  uint64_t *empty = full + NS;
  volatile int *abort_flag = reinterpret_cast<volatile int *>(empty + NS);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) {
    for (int q = 0; q < NS; ++q) {
      mbar_init(&full[q], 1);
      mbar_init(&empty[q], CT / 32);
    }
    *abort_flag = 0;
    mbar_fence_init();
  }
  __syncthreads();

  const int nck = (m + CH - 1) / CH;             // chunks per factor block
  const int nsteps = 2 * rows - 1;
  const int64_t slot_elems = (int64_t)m * ldm;
  const S *Fs = factor + s.foff;

  if (warp == CT / 32) {
    // ---------------- producer warp: stream the factor blocks in use order.  Stage and lap
    // are counted (here and in the consumers): a 64-bit division and remainder per chunk
    // would lengthen the chain from a freed stage to its next copy (complex FP32, per application:
    // 1024^2 in 64 boxes 5.58 -> 4.19 ms, 2048^2 5.84 -> 4.40, 4096^2, at HBM's rate, 12.97 -> 12.76).
    if (lane == 0) {
      int64_t issued = 0;
      bool ok = true;
      int slot = 0;
      uint32_t ph = 0;
      for (int st = 0; st < nsteps && ok; ++st) {
        const S *src = Fs + (st < rows ? st : 2 * rows - 2 - st) * slot_elems;
        for (int c = 0; c < nck; ++c, ++issued) {
          if (!mbar_wait(&empty[slot], ph ^ 1u, abort_flag)) { ok = false; break; }
          const int cols = min(CH, m - c * CH);
          const uint32_t bytes = (uint32_t)(cols * ldm * sizeof(S));
          mbar_arrive_expect_tx(&full[slot], bytes);
          bulk_g2s(ring + (size_t)slot * stage_elems, src, bytes, &full[slot]);
          src += (int64_t)CH * ldm;
          if (++slot == NS) { slot = 0; ph ^= 1u; }
        }
      }
      if (!ok) {
        *abort_flag = 1;
        atomicOr(status, ST_TIMEOUT);
      }
      // no copy may still be landing in shared memory when the CTA exits
      tc::ring_drain(full, issued, NS);
    }
    return;
  }

  // ---------------- consumer warps
  const double2 *a1c = pool + s.aoff;
  const double2 *a2c = a1c + 2 * m + 1;
  const double2 *ia2f = a2c + rows;
  T a1[NA], w[NA][NR];
  bool ownx[NA];
#pragma unroll
  for (int e = 0; e < NA; ++e) {
    const int a = out_index<CT, NA>(tid, e);
    const int gx = s.ex0 + a;
    ownx[e] = a < m && gx >= s.ox0 && gx < s.ox1;
    const double2 t = a < m ? a1c[a] : make_double2(0, 0);
    a1[e] = mk<T>((R)t.x, (R)t.y);
#pragma unroll
    for (int q = 0; q < NR; ++q) w[e][q] = mk<T>(0, 0);
  }
  int slot = 0;
  uint32_t ph = 0;
  bool ok = true;
  for (int st = 0; st < 2 * rows - 1; ++st) {
    const bool fwd = st < rows;
    const int j = fwd ? st : 2 * rows - 2 - st;
    consumer_sync(CT);   // the previous step's reads of vs are done
    if (fwd) {
      const int gy = s.ey0 + j;
      const bool owny = gy >= s.oy0 && gy < s.oy1;
      const double2 isd = ia2f[j];
      const T is = mk<T>((R)isd.x, (R)isd.y);
#pragma unroll
      for (int e = 0; e < NA; ++e) {
        const int a = out_index<CT, NA>(tid, e);
        if (a < m) {
          const T la = cmul(a1[e], is);
#pragma unroll
          for (int q = 0; q < NR; ++q) {
            T rho = mk<T>(0, 0);
            if (owny && ownx[e] && r0 + q < nrhs) {
              const double2 rv = rg[(int64_t)(r0 + q) * vec_stride + (int64_t)gy * NX + s.ex0 + a];
              rho = mk<T>((R)rv.x, (R)rv.y);
            }
            vs[q * ldmax + a] = j > 0 ? cfms(la, w[e][q], rho) : rho;   // rho_j - L_j w_{j-1}
          }
        }
      }
    } else {
      const double2 ind = ia2f[j + 1];
      const T in = mk<T>((R)ind.x, (R)ind.y);
#pragma unroll
      for (int e = 0; e < NA; ++e) {
        const int a = out_index<CT, NA>(tid, e);
        if (a < m) {
          const T ua = cmul(a1[e], in);
#pragma unroll
          for (int q = 0; q < NR; ++q) vs[q * ldmax + a] = cmul(ua, w[e][q]);   // U_j x_{j+1}
        }
      }
    }
    consumer_sync(CT);
    T acc[NA][NR];
#pragma unroll
    for (int e = 0; e < NA; ++e)
#pragma unroll
      for (int q = 0; q < NR; ++q) acc[e][q] = mk<T>(0, 0);
    for (int c = 0; c < nck; ++c) {
      if (ok && !mbar_wait(&full[slot], ph, abort_flag)) {
        ok = false;
        *abort_flag = 1;
        atomicOr(status, ST_TIMEOUT);
      }
      const S *blk = ring + (size_t)slot * stage_elems;
      const int b0 = c * CH;
      const int cols = min(CH, m - b0);
#pragma unroll
      for (int b = 0; b < CH; ++b) {
        if (b < cols) {
          T sv[NA];
          if (NA == 2) {
            // entries 2t, 2t+1 of the column: one vector load (padding up to ldm is readable)
            if (2 * tid < m) load_pair<T, S>(blk + b * ldm + 2 * tid, sv[0], sv[NA - 1]);
            else { sv[0] = mk<T>(0, 0); sv[NA - 1] = mk<T>(0, 0); }
          } else {
#pragma unroll
            for (int e = 0; e < NA; ++e) {
              const int a = out_index<CT, NA>(tid, e);
              sv[e] = a < m ? load_c<T>(blk[b * ldm + a]) : mk<T>(0, 0);
            }
          }
#pragma unroll
          for (int q = 0; q < NR; ++q) {
            const T vb = vs[q * ldmax + b0 + b];
#pragma unroll
            for (int e = 0; e < NA; ++e) acc[e][q] = cfma(sv[e], vb, acc[e][q]);
          }
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty[slot]);
      if (++slot == NS) { slot = 0; ph ^= 1u; }
    }
#pragma unroll
    for (int q = 0; q < NR; ++q) {
      if (r0 + q >= nrhs) continue;
      T *stg = staging + (int64_t)(r0 + q) * stg_stride + s.soff;
#pragma unroll
      for (int e = 0; e < NA; ++e) {
        const int a = out_index<CT, NA>(tid, e);
        if (a < m) {
          if (fwd) {
            w[e][q] = acc[e][q];
            stg[(int64_t)j * m + a] = acc[e][q];
          } else {
            const T x = csub(stg[(int64_t)j * m + a], acc[e][q]);
            w[e][q] = x;
            stg[(int64_t)j * m + a] = x;
          }
        }
      }
    }
  }
}

// One axis of the smoothing function beta_ij (Remark after Eq. (pc)) at cell x of a box
// [e0, e1) owning [o0, o1): 1 on the owned cells, else the C^2 step
// S(t) = t^3 (10 - 15 t + 6 t^2) of t = 1 - d / (W + 1), d the distance from the owned
// cells and W the width of the band on that side (so beta reaches 0 just past the box).
template <typename R> __device__ __forceinline__ R smooth_beta(int x, const AxisDev &a) {
  if (x >= a.o0 && x < a.o1) return (R)1;
  const R t = x < a.o0 ? (R)1 - (R)(a.o0 - x) / (R)(a.o0 - a.e0 + 1) : (R)1 - (R)(x - a.o1 + 1) / (R)(a.e1 - a.o1 + 1);
  return t * t * t * ((R)10 - (R)15 * t + (R)6 * t * t);
}

// The sum runs in the compute precision of the local solutions (FP32 for the c64
// modes: one conversion per cell instead of one per contribution, since the FP64
// pipe is the scarce one on this GPU) and is written out as complex128.
//
// A block covers 256 consecutive cells of GR grid rows.  The boxes that can cover them
// (per row: the boxes whose extent holds the row; per column: box columns nearx - 1 ..
// nearx + 1 of each cell) are looked up once per block into shared memory with their
// staging row offsets, so a thread's staging loads for its GR cells are independent
// (no chain of table, box and staging loads per cell).  Contributions are added in the
// same order as a per-cell walk (box rows, then box columns, ascending): the result does
// not depend on the blocking.  A span with more candidate box columns than GXC (boxes
// under about 40 cells wide) takes the per-cell walk.
constexpr int GR = 4, GXC = 8;
template <typename R, bool SMOOTH>
__global__ void __launch_bounds__(256)
k_gather(const SubDev *__restrict__ subs, const AxisDev *__restrict__ axx, const AxisDev *__restrict__ axy,
         const int32_t *__restrict__ nearx, const int32_t *__restrict__ neary, int nbx, int nby,
         const C<R> *__restrict__ staging_all, int64_t stg_stride, double2 *__restrict__ z_all, int64_t vec_stride,
         int NX, int NY) {
  __shared__ int ylist[GR][3], yoff[GR][3], ny_s[GR];
  __shared__ R ybeta[GR][3];
  __shared__ AxisDev xax[GXC];
  __shared__ int xj[GXC], ncx;
  __shared__ int64_t rowbase[GR][3][GXC];   // staging offset of (row, box row q, candidate c), less e0 of c
  const int t = threadIdx.x;
  const int gx0 = blockIdx.x * 256, gy0 = blockIdx.y * GR;
  if (t < GR) {
    // boxes whose extent covers grid row gy (at most 3, in practice 1 or 2)
    const int gy = gy0 + t;
    int cnt = 0;
    if (gy < NY) {
      const int iy = neary[gy];
      for (int jy = max(iy - 1, 0); jy <= min(iy + 1, nby - 1); ++jy) {
        const AxisDev ay = axy[jy];
        if (gy >= ay.e0 && gy < ay.e1) {
          ylist[t][cnt] = jy;
          yoff[t][cnt] = gy - ay.e0;
          if (SMOOTH) ybeta[t][cnt] = smooth_beta<R>(gy, ay);
          ++cnt;
        }
      }
    }
    ny_s[t] = cnt;
  } else if (t == 32) {
    // candidate box columns of the block's cells, ascending
    const int gx1 = min(gx0 + 256, NX) - 1;
    const int jlo = max(nearx[gx0] - 1, 0), jhi = min(nearx[gx1] + 1, nbx - 1);
    int c = 0;
    for (int jx = jlo; jx <= jhi; ++jx) {
      const AxisDev ax = axx[jx];
      if (ax.e1 <= gx0 || ax.e0 > gx1) continue;
      if (c == GXC) { c = -1; break; }
      xax[c] = ax;
      xj[c] = jx;
      ++c;
    }
    ncx = c;
  }
  __syncthreads();
  const int nc = ncx;
  if (nc >= 0) {
    for (int k = t; k < GR * 3 * GXC; k += 256) {
      const int row = k / (3 * GXC), q = (k / GXC) % 3, c = k % GXC;
      if (q < ny_s[row] && c < nc) {
        const AxisDev ax = xax[c];
        rowbase[row][q][c] = subs[ylist[row][q] * nbx + xj[c]].soff + (int64_t)yoff[row][q] * (ax.e1 - ax.e0) - ax.e0;
      }
    }
  }
  __syncthreads();
  const int gx = gx0 + t;
  if (gx >= NX) return;
  const C<R> *staging = staging_all + (int64_t)blockIdx.z * stg_stride;
  double2 *z = z_all + (int64_t)blockIdx.z * vec_stride;
  const int ix = nearx[gx];
  const int jx0 = max(ix - 1, 0), jx1 = min(ix + 1, nbx - 1);
#pragma unroll
  for (int row = 0; row < GR; ++row) {
    const int gy = gy0 + row;
    if (gy >= NY) break;
    C<R> acc = mk<C<R>>(0, 0);
    for (int q = 0; q < ny_s[row]; ++q) {
      if (nc >= 0) {
        for (int c = 0; c < nc; ++c) {
          const AxisDev ax = xax[c];
          if (xj[c] < jx0 || xj[c] > jx1 || gx < ax.e0 || gx >= ax.e1) continue;
          const C<R> v = staging[rowbase[row][q][c] + gx];
          if (SMOOTH) {   // beta_ij u_ij (Remark after Eq. (pc))
            const R b = mul_rn(ybeta[row][q], smooth_beta<R>(gx, ax));
            acc = mk<C<R>>(fma_rn(b, v.x, acc.x), fma_rn(b, v.y, acc.y));
          } else {
            acc = cadd(acc, v);
          }
        }
      } else {   // per-cell walk
        const int jy = ylist[row][q], ry = yoff[row][q];
        for (int jx = jx0; jx <= jx1; ++jx) {
          const AxisDev ax = axx[jx];
          if (gx < ax.e0 || gx >= ax.e1) continue;
          const C<R> v = staging[subs[jy * nbx + jx].soff + (int64_t)ry * (ax.e1 - ax.e0) + (gx - ax.e0)];
          if (SMOOTH) {
            const R b = mul_rn(ybeta[row][q], smooth_beta<R>(gx, ax));
            acc = mk<C<R>>(fma_rn(b, v.x, acc.x), fma_rn(b, v.y, acc.y));
          } else {
            acc = cadd(acc, v);
          }
        }
      }
    }
    z[(int64_t)gy * NX + gx] = make_double2((double)acc.x, (double)acc.y);
  }
}

// Ring depth: as deep as shared memory allows for the CTAs that share an SM.
template <typename T, typename S>
static int ring_stages(const hd_ctx *ctx, int ldmax, int nr, int groups) {
  int dev = 0, sms = 152;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int64_t ctas = (int64_t)ctx->nsub * groups;
  const int per_sm = (int)std::min<int64_t>(7, (ctas + sms - 1) / sms);
  const size_t budget = (size_t)200 * 1024 / (size_t)std::max(1, per_sm);
  const size_t stage = (size_t)chunk_cols<S>() * ldmax * sizeof(S);
  const size_t fixed = (size_t)nr * ldmax * sizeof(T) + 64;
  int ns = budget > fixed ? (int)((budget - fixed) / stage) : 2;
  return std::min(32, std::max(2, ns));
}

// Right-hand sides per CTA: one factor read serves NR vectors.
static int rhs_per_cta(int nrhs) { return nrhs >= 8 ? 8 : (nrhs >= 4 ? 4 : (nrhs >= 2 ? 2 : 1)); }

static int ld_max(const hd_ctx *ctx) { return (ctx->max_m + 3) & ~3; }

template <typename R, typename S, int CT, int NR>
static cudaError_t launch_subst(hd_ctx *ctx, const double2 *r, int nrhs, int64_t vec_stride, void *staging,
                                int64_t stg_stride, cudaStream_t st) {
  constexpr int NA = CT >= 192 ? 1 : 2;   // outputs per consumer thread
  using T = C<R>;
  const int ldmax = ld_max(ctx);
  const int groups = (nrhs + NR - 1) / NR;
  const int ns = (NR == 1 && ctx->tune_ns > 0) ? ctx->tune_ns : ring_stages<T, S>(ctx, ldmax, NR, groups);
  const size_t smem = subst_smem<T, S>(ns, ldmax, NR);
  cudaError_t e = allow_smem(k_subst<R, S, CT, NA, NR>, smem);
  if (e != cudaSuccess) return e;
  dim3 grid(groups, ctx->nsub);   // a box's source groups run side by side and share its factor reads in L2
  k_subst<R, S, CT, NA, NR><<<grid, CT + 32, smem, st>>>(ctx->d_subs, ctx->d_lpool,
                                                        reinterpret_cast<const S *>(ctx->factor), r, ctx->NX,
                                                        vec_stride, reinterpret_cast<T *>(staging), stg_stride, nrhs,
                                                        ns, ldmax, ctx->d_status);
  return cudaGetLastError();
}

template <typename R, typename S, int CT>
static cudaError_t launch_subst_nr(hd_ctx *ctx, const double2 *r, int nrhs, int64_t vs, void *stg, int64_t ss,
                                   cudaStream_t st) {
  switch (rhs_per_cta(nrhs)) {
    case 8: return launch_subst<R, S, CT, 8>(ctx, r, nrhs, vs, stg, ss, st);
    case 4: return launch_subst<R, S, CT, 4>(ctx, r, nrhs, vs, stg, ss, st);
    case 2: return launch_subst<R, S, CT, 2>(ctx, r, nrhs, vs, stg, ss, st);
    default: return launch_subst<R, S, CT, 1>(ctx, r, nrhs, vs, stg, ss, st);
  }
}

template <typename R, typename S>
static cudaError_t launch_apply_r(hd_ctx *ctx, const double2 *r, int64_t rs, double2 *z, int64_t zs, int nrhs,
                                  void *staging, cudaStream_t st) {
  if (ctx->tc || ctx->sym) {
    tic(ctx, T_SUBST, st);
    cudaError_t e = ctx->tc3  ? launch_subst_x3(ctx, r, nrhs, rs, staging, ctx->staging_elems, st)
                    : ctx->tc ? launch_subst_tc(ctx, r, nrhs, rs, staging, ctx->staging_elems, st)
                              : launch_subst_sym(ctx, r, nrhs, rs, staging, ctx->staging_elems, st);
    toc(ctx, T_SUBST, st, 1);
    if (e != cudaSuccess) return e;
    dim3 grid((ctx->NX + 255) / 256, (ctx->NY + GR - 1) / GR, nrhs);
    tic(ctx, T_GATHER, st);
    auto gather = ctx->smooth ? k_gather<R, true> : k_gather<R, false>;
    gather<<<grid, 256, 0, st>>>(ctx->d_subs, ctx->d_axx, ctx->d_axy, ctx->d_nearx, ctx->d_neary, ctx->nbx,
                                      ctx->nby, reinterpret_cast<const C<R> *>(staging), ctx->staging_elems, z, zs,
                                      ctx->NX, ctx->NY);
    toc(ctx, T_GATHER, st, 1);
    return cudaGetLastError();
  }
  tic(ctx, T_SUBST, st);
  // consumer threads: 96 or 192 cover boxes up to 192 wide, 128 or 256 up to 256
  int ct = ctx->tune_ct ? ctx->tune_ct : (ctx->max_m <= 192 ? 96 : 128);
  if (ct == 96 || ct == 192) ct = ctx->max_m <= 192 ? ct : (ct == 96 ? 128 : 256);
  cudaError_t e;
  switch (ct) {
    case 96: e = launch_subst_nr<R, S, 96>(ctx, r, nrhs, rs, staging, ctx->staging_elems, st); break;
    case 192: e = launch_subst_nr<R, S, 192>(ctx, r, nrhs, rs, staging, ctx->staging_elems, st); break;
    case 256: e = launch_subst_nr<R, S, 256>(ctx, r, nrhs, rs, staging, ctx->staging_elems, st); break;
    default: e = launch_subst_nr<R, S, 128>(ctx, r, nrhs, rs, staging, ctx->staging_elems, st); break;
  }
  toc(ctx, T_SUBST, st, 1);
  if (e != cudaSuccess) return e;
  dim3 grid((ctx->NX + 255) / 256, (ctx->NY + GR - 1) / GR, nrhs);
  tic(ctx, T_GATHER, st);
  auto gather = ctx->smooth ? k_gather<R, true> : k_gather<R, false>;
  gather<<<grid, 256, 0, st>>>(ctx->d_subs, ctx->d_axx, ctx->d_axy, ctx->d_nearx, ctx->d_neary, ctx->nbx,
                                    ctx->nby, reinterpret_cast<const C<R> *>(staging), ctx->staging_elems, z, zs,
                                    ctx->NX, ctx->NY);
  toc(ctx, T_GATHER, st, 1);
  return cudaGetLastError();
}

int run_apply(hd_ctx *ctx, const double2 *r, int64_t rs, double2 *z, int64_t zs, int nrhs, void *staging,
              cudaStream_t st) {
  cudaError_t e = ctx->prec == HD_C64    ? launch_apply_r<float, float2>(ctx, r, rs, z, zs, nrhs, staging, st)
                  : ctx->prec == HD_C64_H ? launch_apply_r<float, __half2>(ctx, r, rs, z, zs, nrhs, staging, st)
                  : ctx->prec == HD_C64_B ? launch_apply_r<float, __nv_bfloat162>(ctx, r, rs, z, zs, nrhs, staging, st)
                                          : launch_apply_r<double, double2>(ctx, r, rs, z, zs, nrhs, staging, st);
  if (e != cudaSuccess) return cuda_fail(e, "preconditioner launch");
  return HD_OK;
}

// z += c over nrhs strided vectors (grid.y = right-hand side)
__global__ void k_add(double2 *__restrict__ z, int64_t zs, const double2 *__restrict__ c, int64_t cs, int64_t n) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  double2 *zr = z + (int64_t)blockIdx.y * zs;
  const double2 a = zr[i], b = c[(int64_t)blockIdx.y * cs + i];
  zr[i] = make_double2(a.x + b.x, a.y + b.y);
}

// Multi-step overlapping DDM, Eq. (ddm0), (ddms), (sum), as residual correction:
// z = M r, then nsteps - 1 times  t = r - A z,  z += M t.
int run_apply_steps(hd_ctx *ctx, const double2 *r, int64_t rs, double2 *z, int64_t zs, int nrhs, int nsteps,
                    double2 *work, void *staging, cudaStream_t st) {
  int rc = run_apply(ctx, r, rs, z, zs, nrhs, staging, st);
  if (rc || nsteps <= 1) return rc;
  const int64_t n = (int64_t)ctx->NX * ctx->NY;
  double2 *t = work, *c = work + n * nrhs;
  for (int s = 1; s < nsteps; ++s) {
    tic(ctx, T_MATVEC, st);
    cudaError_t e = launch_residual_strided(ctx, r, rs, z, zs, t, n, nrhs, st);
    toc(ctx, T_MATVEC, st, 1);
    if (e != cudaSuccess) return cuda_fail(e, "multi-step residual");
    if ((rc = run_apply(ctx, t, n, c, n, nrhs, staging, st))) return rc;
    tic(ctx, T_GATHER, st);
    k_add<<<dim3((unsigned)((n + 255) / 256), nrhs), 256, 0, st>>>(z, zs, c, n, n);
    toc(ctx, T_GATHER, st, 1);
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "multi-step sum");
  }
  return HD_OK;
}

}  // namespace hd

// ---------------------------------------------------------------------------
// Autotuner of the substitution launch: consumer threads per CTA (full storage)
// and ring depth, timed with CUDA events on real applications; the winner is
// remembered per (precision, widest box, boxes, device) for the process.
#include <map>
#include <mutex>
#include <tuple>

namespace hd {

static std::mutex g_tune_mu;
static std::map<std::tuple<int, int, int, int, int>, std::pair<int, int>> g_tune_cache;

// Applies the launch shape an earlier autotune chose for this context's shape (same
// precision, storage, widest box, box count and device) in this process; false if none.
bool lookup_tuning(hd_ctx *ctx) {
  if (ctx->tc) return true;   // the tensor-core substitution has one launch shape
  int dev = 0;
  cudaGetDevice(&dev);
  const auto key = std::make_tuple(ctx->prec, ctx->sym ? 1 : 0, ctx->max_m, ctx->nsub, dev);
  std::lock_guard<std::mutex> lk(g_tune_mu);
  auto it = g_tune_cache.find(key);
  if (it == g_tune_cache.end()) return false;
  ctx->tune_ct = it->second.first;
  ctx->tune_ns = it->second.second;
  return true;
}

int autotune_subst(hd_ctx *ctx, const double2 *r, double2 *z, void *staging, cudaStream_t st, int *ct_out,
                   int *ns_out, float *ms_out) {
  if (ctx->tc) {   // the tensor-core substitution has one launch shape (ring sized by shared memory)
    if (ct_out) *ct_out = 128;
    if (ns_out) *ns_out = 0;
    if (ms_out) *ms_out = -1.f;
    return HD_OK;
  }
  int dev = 0;
  cudaGetDevice(&dev);
  const auto key = std::make_tuple(ctx->prec, ctx->sym ? 1 : 0, ctx->max_m, ctx->nsub, dev);
  {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    auto it = g_tune_cache.find(key);
    if (it != g_tune_cache.end()) {
      ctx->tune_ct = it->second.first;
      ctx->tune_ns = it->second.second;
      if (ct_out) *ct_out = ctx->tune_ct;
      if (ns_out) *ns_out = ctx->tune_ns;
      if (ms_out) *ms_out = -1.f;
      return HD_OK;
    }
  }
  const int ldmax = ld_max(ctx);
  // one ring stage of the full storage: chunk_cols<S>() columns of ldmax entries (64 bytes per row)
  int dev_optin = 0;
  cudaDeviceGetAttribute(&dev_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  // symmetric storage: threads follow from the number of boxes (launch_subst_sym), only the ring depth is timed
  std::vector<int> cts = ctx->sym ? std::vector<int>{subst_sym_threads(ctx)}
                                  : (ctx->max_m <= 192 ? std::vector<int>{96, 128, 192} : std::vector<int>{128, 256});
  std::vector<int> depths{2, 3, 4, 6, 8, 12, 16, 24, 32};
  if (ctx->sym) {   // up to the deepest ring that its launch can have
    const int deepest = subst_sym_stages(ctx);
    while (!depths.empty() && depths.back() >= deepest) depths.pop_back();
    depths.push_back(deepest);
  }
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  float best = 1e30f;
  int best_ct = 0, best_ns = 0;
  const bool prof = ctx->profiling;
  ctx->profiling = false;
  for (int ct : cts)
    for (int ns : depths) {
      if (!ctx->sym && (size_t)ns * ldmax * 64 + 8192 > (size_t)std::min(dev_optin, 224 * 1024)) continue;
      ctx->tune_ct = ct;
      ctx->tune_ns = ns;
      float tot = 0.f;
      bool ok = true;
      for (int rep = 0; rep < 3 && ok; ++rep) {
        cudaEventRecord(e0, st);
        ok = run_apply(ctx, r, 0, z, 0, 1, staging, st) == HD_OK;
        if (!ok) cudaGetLastError();   // a shape that does not fit leaves no error behind
        cudaEventRecord(e1, st);
        cudaEventSynchronize(e1);
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        if (rep > 0) tot += ms;   // the first run warms up
      }
      if (ok && tot < best) { best = tot; best_ct = ct; best_ns = ns; }
    }
  ctx->profiling = prof;
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  ctx->t_launch[T_SUBST] = 0;
  ctx->t_launch[T_GATHER] = 0;
  if (!best_ct) { set_error("hd_autotune: no substitution configuration ran"); return HD_ERR_CUDA; }
  ctx->tune_ct = best_ct;
  ctx->tune_ns = best_ns;
  {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    g_tune_cache[key] = {best_ct, best_ns};
  }
  if (ct_out) *ct_out = best_ct;
  if (ns_out) *ns_out = best_ns;
  if (ms_out) *ms_out = best / 2.f;
  return HD_OK;
}

}  // namespace hd

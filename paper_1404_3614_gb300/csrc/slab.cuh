// Fused y-x-y slab pass of the FP32 3D operator for an isotropic coefficient (one real
// coefficient value per double-grid point), transform length M = R * R on the x and y
// axes. One CTA owns one (right-hand side, component, z) slab of the field after the z
// inverse transform: it loads the Ny x Nh half-spectrum slab, runs the zero-padded
// inverse y transforms, the x row pass (Hermitian c2r of two real rows per complex FFT,
// pointwise coefficient A_M / |M|, r2c), and the truncating forward y transforms, all in
// shared memory, and writes the Ny x Nh slab back. This is the middle of the operator
// C u = Gamma P_N F_M (A_M/|M|) F_M^{-1} Pad(u) (Lemma double-grid, Eq. MBA_GA) with the
// intermediate double-grid slab never leaving the SM.
//
// Transforms are warp-level in-register Cooley-Tukey FFTs of length R * R: R lanes own
// one pencil; lane l loads x[l + R n2] (n2 < R), does a register DFT of length R, applies
// the twiddles w_M^(l k2), exchanges through shared memory, and does the second register
// DFT; lane l then holds X[l + R k1] (k1 < R). The output layout of the inverse x
// transform is the input layout of the forward one, so the coefficient product happens
// in registers between them. In the slab kernel every lane group transforms two pencils at
// once in packed FP32 arithmetic (fpair): two columns, or two pairs of rows.
#pragma once
#include <algorithm>

#include "fpair.cuh"
#include "kernels.cuh"

namespace homb {

// 15 warps, and, where a caller asks for more, a compilation for 20 (at 225 for 16: 20 warps' scratch
// exceeds the shared memory). One compilation for 16 warps costs the 15 of the automatic choice at
// 225 0.7 % (operator 382.8 -> 385.5 us).
constexpr int kSlabMaxThreads = 480;
constexpr int slab_wide_threads(int R) { return R < 15 ? 640 : 512; }

// Layout of the slab in shared memory: columns kx = l + R m and l + R (m + 1), m even, side by side
// (a column pair: one lane group's two pencils in the y passes, and two of a lane's values
// in the x pass), each y position one 16-byte group (re, re', im, im'). Rows m < slab_rows hold
// the Nh columns (those past Nh are zero); a pair's stride is odd and covers whole groups of four
// rows, so that the x pass, eight lanes on eight pairs, has no bank conflicts.
__host__ __device__ constexpr int slab_rows(int R, bool zb) {
  return zb ? ((R * R + 3) / 4 + R - 1) / R : (R + 1) / 2;   // ZeroBand<R>::lo, or all of M = N
}
__host__ __device__ constexpr int slab_pairs(int R, bool zb) { return (slab_rows(R, zb) + 1) / 2 * R; }
__host__ __device__ constexpr int slab_ld(int M) { return (M + 3) / 4 * 4 + 1; }

// Byte offset of the scratch / staging region of a slab CTA: after the barrier (16 bytes), two
// twiddle tables [M] and the column pairs (the bulk copy lands there).
__host__ __device__ inline size_t slab_scratch_offset(int R, bool zb) {
  return 16 + (size_t)((R * R + 1) / 2 * 2) * 16 + (size_t)slab_pairs(R, zb) * slab_ld(R * R) * 16;
}

// shared memory of one slab CTA with `warps` warps: the scratch region holds the x pass's double
// pencils or the staged input slab (Ny x Nh plus one element of alignment slack)
inline size_t slab_smem_bytes(int R, bool zb, int Ny, int Nh, int warps) {
  return slab_scratch_offset(R, zb) +
         std::max((size_t)warps * (32 / R) * R * R * 16, ((size_t)Ny * Nh + 2) * 8);
}

// First-stage DFT of a zero-padded inverse transform (inputs of the zero band not read) and
// last-stage DFT of a truncating forward one (outputs of the band not computed)
template <typename T, int R>
__device__ __forceinline__ void dft_reg_zin(cpx<T>* v, int dir) {
  if constexpr (R == 15) dft15_zin<T>(v, dir);
  else {
#pragma unroll
    for (int n = 0; n < R; ++n)
      if (ZeroBand<R>::in(n)) v[n] = mk<T>(T(0), T(0));
    dft_reg<T, R>(v, dir);
  }
}
template <typename T, int R>
__device__ __forceinline__ void dft_reg_zout(cpx<T>* v, int dir) {
  if constexpr (R == 15) dft15_zout<T>(v, dir);
  else dft_reg<T, R>(v, dir);
}

// In-place FFT of one contiguous pencil of length R*R by the R lanes of a lane group
// (lane index l < R). Every lane of the warp calls it (on = false: no memory access).
// Wt holds w_M^(l k) at [k][l].
template <typename T, int R>
__device__ __forceinline__ void pencil_fft_inplace(cpx<T>* p, int l, const cpx<T>* Wt, int dir, bool on) {
  cpx<T> v[R];
#pragma unroll
  for (int n = 0; n < R; ++n) v[n] = on ? p[l + R * n] : mk<T>(T(0), T(0));
  dft_reg<T, R>(v, dir);
#pragma unroll
  for (int k = 1; k < R; ++k) v[k] = mulc<T>(v[k], Wt[k * R + l], dir > 0);
  __syncwarp();
  if (on) {
#pragma unroll
    for (int k = 0; k < R; ++k) p[l + R * k] = st_norm<T>(v[k]);
  }
  __syncwarp();
#pragma unroll
  for (int n = 0; n < R; ++n) v[n] = on ? p[n + R * l] : mk<T>(T(0), T(0));
  dft_reg<T, R>(v, dir);
  __syncwarp();
  if (on) {
#pragma unroll
    for (int k = 0; k < R; ++k) p[l + R * k] = st_norm<T>(v[k]);
  }
  __syncwarp();
}

constexpr long long kSlabSpinLimit = 1LL << 22;   // polls of the staged-copy barrier

__device__ __forceinline__ uint32_t slab_smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Bounded wait for one phase of the staging barrier; false if it gave up.
__device__ __forceinline__ bool slab_wait(uint32_t mbar, uint32_t phase) {
  for (long long it = 0; it < kSlabSpinLimit; ++it) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(mbar), "r"(phase)
        : "memory");
    if (done) return true;
  }
  return false;
}

// Where the Ny x Nh input slab starting at global address `src` goes in the staging buffer
// and how it is copied: a bulk copy of the 16-byte aligned middle (`body` bytes from element
// `head`), plus at most one plain element in front (head = 1) and one behind (tail = 1).
struct SlabStage {
  int head, tail;
  unsigned body;
};
template <typename T>
__device__ __forceinline__ SlabStage slab_stage_plan(const cpx<T>* src, long long elems) {
  SlabStage st;
  st.head = (reinterpret_cast<uintptr_t>(src) & 15) ? 1 : 0;
  const long long bytes = (elems - st.head) * (long long)sizeof(cpx<T>);
  st.body = (unsigned)(bytes & ~15LL);
  st.tail = (int)((bytes - st.body) / (long long)sizeof(cpx<T>));
  return st;
}

// Persistent fused slab pass. Each CTA walks the slabs blockIdx.x, blockIdx.x + gridDim.x, ...
// (z-major, so the slabs in flight share few coefficient planes). The input of a slab is
// staged in shared memory by one bulk asynchronous copy (an mbarrier tracks its bytes),
// issued for the next slab as soon as the x pass of the current one has released the
// staging buffer, so the copy overlaps the forward y transforms and the stores. The inverse
// y transforms read the staged rows directly (zero padding implicit).
// pencil_fft_inplace for a truncating forward transform (dir = -1): the outputs of the zero
// band are neither computed nor stored
template <typename T, int R>
__device__ __forceinline__ void pencil_fft_fwd_trunc(cpx<T>* p, int l, const cpx<T>* Wt, bool on) {
  cpx<T> v[R];
#pragma unroll
  for (int n = 0; n < R; ++n) v[n] = on ? p[l + R * n] : mk<T>(T(0), T(0));
  dft_reg<T, R>(v, -1);
#pragma unroll
  for (int k = 1; k < R; ++k) v[k] = mulc<T>(v[k], Wt[k * R + l], false);
  __syncwarp();
  if (on) {
#pragma unroll
    for (int k = 0; k < R; ++k) p[l + R * k] = st_norm<T>(v[k]);
  }
  __syncwarp();
#pragma unroll
  for (int n = 0; n < R; ++n) v[n] = on ? p[n + R * l] : mk<T>(T(0), T(0));
  dft_reg_zout<T, R>(v, -1);
  __syncwarp();
  if (on) {
#pragma unroll
    for (int k = 0; k < R; ++k)
      if (!ZeroBand<R>::in(k)) p[l + R * k] = st_norm<T>(v[k]);
  }
  __syncwarp();
}

// pencil_fft_inplace for a zero-padded inverse transform (dir = +1): the zero band's inputs
// are not read
template <typename T, int R>
__device__ __forceinline__ void pencil_fft_pad_inv(cpx<T>* p, int l, const cpx<T>* Wt, bool on) {
  cpx<T> v[R];
#pragma unroll
  for (int n = 0; n < R; ++n)
    if (!ZeroBand<R>::in(n)) v[n] = on ? p[l + R * n] : mk<T>(T(0), T(0));
  dft_reg_zin<T, R>(v, +1);
#pragma unroll
  for (int k = 1; k < R; ++k) v[k] = mulc<T>(v[k], Wt[k * R + l], true);
  __syncwarp();
  if (on) {
#pragma unroll
    for (int k = 0; k < R; ++k) p[l + R * k] = st_norm<T>(v[k]);
  }
  __syncwarp();
#pragma unroll
  for (int n = 0; n < R; ++n) v[n] = on ? p[n + R * l] : mk<T>(T(0), T(0));
  dft_reg<T, R>(v, +1);
  __syncwarp();
  if (on) {
#pragma unroll
    for (int k = 0; k < R; ++k) p[l + R * k] = st_norm<T>(v[k]);
  }
  __syncwarp();
}

// Twiddles w_M^(l k) on the first-stage results (conj: inverse), both pencils alike
template <int R>
__device__ __forceinline__ void slab_twiddle(fpair2* v, const float2* Wt, int l, bool conj) {
#pragma unroll
  for (int k = 1; k < R; ++k) {
    const float2 w = Wt[k * R + l];
    v[k] = mulc<fpair>(v[k], mk<fpair>(fpair(w.x), fpair(w.y)), conj);
  }
}
// Transpose of a lane group's R x R values through its pencil of shared memory: v[k] of lane l
// goes to v[l] of lane k (own = false: nothing written, the values read are not used; S is then
// the pencil of another lane group of the same warp, which its barriers keep apart from writes)
template <int R>
__device__ __forceinline__ void slab_exchange(fpair2* v, fpair2* S, int l, bool own) {
  __syncwarp();
  if (own) {
#pragma unroll
    for (int k = 0; k < R; ++k) S[l + R * k] = v[k];
  }
  __syncwarp();
#pragma unroll
  for (int n = 0; n < R; ++n) v[n] = S[n + R * l];
}
__device__ __forceinline__ fpair slab_shfl(fpair a, int src) {
  return fpair(__shfl_sync(0xffffffffu, a.v.x, src), __shfl_sync(0xffffffffu, a.v.y, src));
}

// 225^3, 9 components: 0.311 -> 0.270 ms a launch (the 3-field operator 428 -> 383 us) against one
// pencil a lane group: 248 M -> 123 M warp instructions. Shared-memory accesses weigh most
// (71 % of the L1 data pipe; FP32 pipe 42 %, issue 37 %): a pencil passes through
// shared memory once between its two register DFTs, and once between the y and x passes. 128
// registers a thread (15 warps, one CTA an SM) leave 92 bytes of spills.
template <int R, bool ZB, int NT = kSlabMaxThreads>
__global__ void __launch_bounds__(NT) k_slab(SlabArgs a) {
  using F = fpair;
  constexpr int M = R * R;
  constexpr int LD = slab_ld(M);
  constexpr int PW = 32 / R;   // lane groups per warp, two pencils each
  constexpr int NM = slab_rows(R, ZB), NP = (NM + 1) / 2, NC = slab_pairs(R, ZB);
  extern __shared__ __align__(16) unsigned char smem[];
  uint64_t* mbar = reinterpret_cast<uint64_t*>(smem);
  float2* Wt = reinterpret_cast<float2*>(smem + 16);
  float2* Ws = Wt + (M + 1) / 2 * 2;   // the same times 1 / (2 |M|)
  fpair2* P = reinterpret_cast<fpair2*>(Ws + (M + 1) / 2 * 2);   // [NC][LD]
  // x-pass scratch [warps * PW][M] double pencils, and between x passes the staged next input
  float2* S = reinterpret_cast<float2*>(smem + slab_scratch_offset(R, ZB));
  const int Ny = a.Ny, Nh = a.Nh, half = (Ny - 1) / 2;
  const long long slab_elems = (long long)Ny * Nh;
  const long long nslabs = (long long)a.nrc * a.Mz;
  const float2* in = reinterpret_cast<const float2*>(a.in);
  float2* out = reinterpret_cast<float2*>(a.out);
  // twiddles w_M^(l k) stored at [k][l] so that the R lanes of a group read consecutive words
  const float2* W = reinterpret_cast<const float2*>(a.W);
  const float fs = 0.5f * (float)a.scale;   // 1 / |M| and the 1/2 of the split into rows
  for (int t = threadIdx.x; t < M; t += blockDim.x) {
    const int k = t / R;
    const float2 w = W[(t - k * R) * k];
    Wt[t] = w;
    Ws[t] = make_float2(fs * w.x, fs * w.y);
  }
  // the padding rows M .. LD - 1 of every column pair: zero, and never written
  for (int t = threadIdx.x; t < NC * (LD - M); t += blockDim.x) {
    const int c = t / (LD - M);
    P[c * LD + M + (t - c * (LD - M))] = mk<F>(F(0.f), F(0.f));
  }
  // slab q of the walk is (z, rc) = (q / nrc, q mod nrc) (z-major); in memory it is slab
  // rc * Mz + z of the [nrc][Mz][Ny][Nh] field
  auto mem = [&](long long q) {
    const long long z = q / a.nrc;
    return (q - z * a.nrc) * a.Mz + z;
  };
  auto active = [&](long long s) {
    if (a.cg == nullptr) return true;
    const int rc = (int)(s % a.nrc);
    return a.cg->active[rc / a.C] != 0;
  };
  auto next_active = [&](long long s) {
    do {
      s += gridDim.x;
    } while (s < nslabs && !active(s));
    return s;
  };
  long long s = blockIdx.x;
  if (s < nslabs && !active(s)) s = next_active(s);
  const uint32_t mb = slab_smem_u32(mbar);
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mb) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  // thread 0: start the staged copy of slab t; the plain end elements go to registers
  float2 edge0 = make_float2(0.f, 0.f), edge1 = make_float2(0.f, 0.f);
  auto issue = [&](long long t) {
    const float2* src = in + mem(t) * slab_elems;
    const SlabStage st = slab_stage_plan<float>(src, slab_elems);
    float2* stage = S + st.head;   // S is 16-byte aligned: element `head` lands aligned
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mb), "r"(st.body) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     slab_smem_u32(stage + st.head)),
                 "l"(src + st.head), "r"(st.body), "r"(mb)
                 : "memory");
    if (st.head) edge0 = src[0];
    if (st.tail) edge1 = src[slab_elems - 1];
  };
  if (threadIdx.x == 0 && s < nslabs) issue(s);
  uint32_t phase = 0;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarp = blockDim.x >> 5;
  // R = 15: one lane group to each half warp (the hardware serves a 64-bit access half by half:
  // groups on lanes 0-14 and 15-29 cost a third wavefront); else R lanes after one another
  // Lanes outside a group (act = false) read what lane 0 of their warp's last group, or of their half
  // warp, reads, and groups past the last pencil or rows (on = false) the last ones, which are
  // their own warp's then: no warp reads what another one writes, and no access needs a predicate.
  const int sub = R == 15 ? lane >> 4 : min(lane / R, PW - 1);
  const int l0 = R == 15 ? sub << 4 : sub * R;
  const bool act = lane - l0 < R;
  const int l = act ? lane - l0 : 0;
  const int lc = l > 0 ? R - l : 0;                      // the column of this lane's negative frequencies
  const int mirror = act && l > 0 ? l0 + lc : lane;      // and the lane that holds them
  const int slots = nwarp * PW;
  const int slot = warp * PW + sub;
  constexpr int nquad = (M + 3) / 4;     // groups of four rows (the last one holds M mod 4 = 1)
  static_assert(M % 4 == 1, "rows of the last group");
  fpair2* Sw = reinterpret_cast<fpair2*>(S) + (size_t)slot * M;

  while (s < nslabs) {
    const int z = (int)(s / a.nrc);
    const SlabStage st = slab_stage_plan<float>(in + mem(s) * slab_elems, slab_elems);
    const float2* stage = S + st.head;
    // ---- wait for the staged input (bounded), complete its plain end elements
    const bool ok = __syncthreads_and(slab_wait(mb, phase) ? 1 : 0) != 0;
    if (!ok) {
      // the copy never completed: report it, give it one more bounded wait, stop this CTA
      if (threadIdx.x == 0 && a.fault) atomicExch(a.fault, 1);
      slab_wait(mb, phase);
      return;
    }
    phase ^= 1u;
    if (threadIdx.x == 0) {
      if (st.head) const_cast<float2*>(stage)[0] = edge0;
      if (st.tail) const_cast<float2*>(stage)[slab_elems - 1] = edge1;
    }
    __syncthreads();

    // ---- inverse y transforms, a column pair to each lane group: input rows from the staged
    // slab (row-major [Ny][Nh]), zero padded to M; columns past Nh are zero
    for (int c0 = 0; c0 < NC; c0 += slots) {
      if (c0 + warp * PW >= NC) break;   // no pair for this warp in this or a later round
      const int c = min(c0 + slot, NC - 1);
      const bool on = act && c0 + slot < NC;
      const int mp = c / R;              // columns l' + R 2 mp and l' + R (2 mp + 1), l' = c mod R
      const int ka = c - mp * R + 2 * R * mp, kb = ka + R;
      const bool ona = on && ka < Nh, onb = on && kb < Nh;
      fpair2* p = P + (size_t)c * LD;
      fpair2 v[R];
#pragma unroll
      for (int n = 0; n < R; ++n) {
        if (ZB && ZeroBand<R>::in(n)) continue;   // padding rows only
        const int pos = l + R * n;
        const int y = pos <= half ? pos : (pos >= M - half ? pos - M + Ny : -1);
        float2 u = make_float2(0.f, 0.f), w = u;
        if (y >= 0 && ona) u = stage[y * Nh + ka];
        if (y >= 0 && onb) w = stage[y * Nh + kb];
        v[n] = mk<F>(F(u.x, w.x), F(u.y, w.y));
      }
      if constexpr (ZB) dft_reg_zin<F, R>(v, +1);
      else dft_reg<F, R>(v, +1);
      slab_twiddle<R>(v, Wt, l, true);   // inverse: conjugate twiddles
      slab_exchange<R>(v, p, l, on);
      dft_reg<F, R>(v, +1);
      __syncwarp();
      if (on) {
#pragma unroll
        for (int k = 0; k < R; ++k) p[l + R * k] = v[k];
      }
    }
    __syncthreads();

    // ---- x row pass: rows y0 .. y0 + 3 as two complex pencils Z = X_a + i X_b
    const float* coefz = reinterpret_cast<const float*>(a.coef) + (size_t)z * M * M;
    for (int q0 = 0; q0 < nquad; q0 += slots) {
      if (q0 + warp * PW >= nquad) break;   // no rows for this warp
      const bool on = act && q0 + slot < nquad;
      const int y0 = 4 * min(q0 + slot, nquad - 1);
      const bool four = y0 + 3 < M;         // else one row
      fpair2 v[R];
      {
        // columns l + R m (frequency k = l + R m, value m) and R - l + R m (frequency
        // -k' = M - (R - l) - R m, value R - 1 - m; lane 0: its columns R m are the frequencies
        // -R m, value R - m)
        const fpair2* pf = P + (size_t)l * LD + y0;
        const fpair2* pc = P + (size_t)lc * LD + y0;
        fpair2 zc[2 * NP];
#pragma unroll
        for (int h = 0; h < NP; ++h) {
          const fpair2 q[4] = {pf[h * R * LD], pf[h * R * LD + 1], pf[h * R * LD + 2], pf[h * R * LD + 3]};
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const int n = 2 * h + e;
            if (n >= NM) continue;
            float re[4], im[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
              re[r] = e ? q[r].x.v.y : q[r].x.v.x;
              im[r] = e ? q[r].y.v.y : q[r].y.v.x;
              if (n == 0 && l == 0) im[r] = 0.f;
            }
            v[n] = mk<F>(F(re[0] - im[1], re[2] - im[3]), F(im[0] + re[1], im[2] + re[3]));
          }
          const fpair2 c[4] = {pc[h * R * LD], pc[h * R * LD + 1], pc[h * R * LD + 2], pc[h * R * LD + 3]};
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            float re[4], im[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
              re[r] = e ? c[r].x.v.y : c[r].x.v.x;
              im[r] = e ? c[r].y.v.y : c[r].y.v.x;
            }
            zc[2 * h + e] = mk<F>(F(re[0] + im[1], re[2] + im[3]), F(re[1] - im[0], re[3] - im[2]));
          }
        }
#pragma unroll
        for (int m = 0; m < NM; ++m) {
          const fpair2 up = m + 1 < NM ? zc[m + 1] : mk<F>(F(0.f), F(0.f));
          const fpair2 w = l == 0 ? up : zc[m];
          if (R - 1 - m >= NM) v[R - 1 - m] = w;
          else if (R - 1 - m == m && l + R * m >= Nh) v[m] = w;   // M = N: the middle value, either side of Nh
        }
      }
      if constexpr (ZB) dft_reg_zin<F, R>(v, +1);
      else dft_reg<F, R>(v, +1);
      // the coefficient of the even rows (real parts): loaded before the second half of the
      // transform, so that it overlaps the exchange
      const float* cy = coefz + (size_t)y0 * M + l;
      const float* cy2 = four ? cy + 2 * M : cy;
      F ce[R];
#pragma unroll
      for (int k = 0; k < R; ++k) ce[k] = F(__ldg(cy + R * k), __ldg(cy2 + R * k));
      slab_twiddle<R>(v, Wt, l, true);
      slab_exchange<R>(v, Sw, l, act);
      dft_reg<F, R>(v, +1);
      // v[k1] = z(x = l + R k1): real parts rows y0, y0 + 2, imaginary parts rows y0 + 1, y0 + 3
      // (a group of one row has zeros in the others)
#pragma unroll
      for (int k = 0; k < R; ++k) v[k].x = v[k].x * ce[k];
      const float* cy1 = four ? cy + M : cy;
      const float* cy3 = four ? cy + 3 * M : cy;
#pragma unroll
      for (int k = 0; k < R; ++k) ce[k] = F(__ldg(cy1 + R * k), __ldg(cy3 + R * k));
#pragma unroll
      for (int k = 0; k < R; ++k) v[k].y = v[k].y * ce[k];
      // forward transform: lane l holds x[l + R n2] with n2 = k1; the kept frequencies only
      dft_reg<F, R>(v, -1);
      slab_twiddle<R>(v, Wt, l, false);
      slab_exchange<R>(v, Sw, l, act);
      if constexpr (ZB) dft_reg_zout<F, R>(v, -1);
      else dft_reg<F, R>(v, -1);
      // split Z into its rows: Z(M - k), k = l + R n, is value R - 1 - n of the lane R - l, and of
      // lane 0 its own value R - n
      fpair2* d = P + (size_t)l * LD + y0;
#pragma unroll
      for (int h = 0; h < NP; ++h) {
        float re[4][2], im[4][2];   // [row][column of the pair]
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int n = 2 * h + e;
          if (n >= NM) {
#pragma unroll
            for (int r = 0; r < 4; ++r) re[r][e] = im[r][e] = 0.f;
            continue;
          }
          fpair2 zm;
          zm.x = slab_shfl(v[R - 1 - n].x, mirror);
          zm.y = slab_shfl(v[R - 1 - n].y, mirror);
          if (l == 0) zm = v[n == 0 ? 0 : R - n];
          const fpair2 zk = v[n];
          re[0][e] = zk.x.v.x + zm.x.v.x;
          im[0][e] = zk.y.v.x - zm.y.v.x;
          re[1][e] = zk.y.v.x + zm.y.v.x;
          im[1][e] = zm.x.v.x - zk.x.v.x;
          re[2][e] = zk.x.v.y + zm.x.v.y;
          im[2][e] = zk.y.v.y - zm.y.v.y;
          re[3][e] = zk.y.v.y + zm.y.v.y;
          im[3][e] = zm.x.v.y - zk.x.v.y;
        }
        if (on) {
#pragma unroll
          for (int r = 0; r < 4; ++r)
            if (r == 0 || four) d[h * R * LD + r] = mk<F>(F(re[r][0], re[r][1]), F(im[r][0], im[r][1]));
        }
      }
      __syncwarp();
    }
    // ---- the staging buffer is free: start the copy of the next slab's input (the async
    // proxy writes where the generic proxy just read and wrote: every thread orders its own
    // accesses before it, then the barrier, then one thread issues the copy)
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    const long long sn = next_active(s);
    if (threadIdx.x == 0 && sn < nslabs) issue(sn);

    // ---- forward y transforms in place (truncated; with ZB the zero band's rows are neither
    // computed nor stored)
    for (int c0 = 0; c0 < NC; c0 += slots) {
      if (c0 + warp * PW >= NC) break;
      const bool on = act && c0 + slot < NC;
      fpair2* p = P + (size_t)min(c0 + slot, NC - 1) * LD;
      fpair2 v[R];
#pragma unroll
      for (int n = 0; n < R; ++n) v[n] = p[l + R * n];
      dft_reg<F, R>(v, -1);
      slab_twiddle<R>(v, Ws, l, false);
      v[0] = scl<F>(v[0], F(fs));
      slab_exchange<R>(v, p, l, on);
      if constexpr (ZB) dft_reg_zout<F, R>(v, -1);
      else dft_reg<F, R>(v, -1);
      __syncwarp();
      if (on) {
#pragma unroll
        for (int k = 0; k < R; ++k)
          if (!(ZB && ZeroBand<R>::in(k))) p[l + R * k] = v[k];
      }
    }
    __syncthreads();
    float2* o = out + mem(s) * slab_elems;
    for (int kx = lane; kx < Nh; kx += 32) {
      const int m = kx / R;
      const float* pk = reinterpret_cast<const float*>(P + (size_t)(m / 2 * R + kx - m * R) * LD) + (m & 1);
#pragma unroll 4
      for (int y = warp; y < Ny; y += nwarp) {
        const int pos = y <= half ? y : y - Ny + M;
        o[(size_t)y * Nh + kx] = make_float2(pk[4 * pos], pk[4 * pos + 2]);
      }
    }
    __syncthreads();   // P is rewritten by the next slab's inverse y transforms
    s = sn;
  }
}

template <int R, bool ZB, int NT> cudaError_t launch_slab_nt(const SlabArgs& a, int warps, cudaStream_t s) {
  const size_t smem = slab_smem_bytes(R, ZB, a.Ny, a.Nh, warps);
  static std::atomic<int> cache[kAttrDevices] = {};
  cudaError_t e = smem_attr(k_slab<R, ZB, NT>, smem, cache);
  if (e != cudaSuccess) return e;
  // persistent: as many CTAs as are resident at once, at most one per slab
  int dev = 0, sms = 0, per = 0;
  e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_slab<R, ZB, NT>, warps * 32, smem);
  if (e != cudaSuccess) return e;
  if (per < 1) return cudaErrorInvalidConfiguration;
  const long long nslabs = (long long)a.nrc * a.Mz;
  const int grid = (int)std::min<long long>(nslabs, (long long)sms * per);
  k_slab<R, ZB, NT><<<grid, warps * 32, smem, s>>>(a);
  return cudaGetLastError();
}

template <int R, bool ZB> cudaError_t launch_slab_rz(const SlabArgs& a, int warps, cudaStream_t s) {
  if (warps * 32 > kSlabMaxThreads) return launch_slab_nt<R, ZB, slab_wide_threads(R)>(a, warps, s);
  return launch_slab_nt<R, ZB, kSlabMaxThreads>(a, warps, s);
}

// The zero band applies when the y rows (Ny stored around 0) and the Hermitian x extension
// (2 Nh - 1 frequencies around 0) leave it empty: a zero-padded double grid M >= 2N - 1; not
// when the transforms are as long as the data (GaNi on the N grid, M = N)
inline bool slab_band_free(int M, int Ny, int Nh) {
  auto f = [M](int n) {
    const int half = (n - 1) / 2, top = n - 1 - half;
    return half < (M + 3) / 4 && M - top > (3 * M - 3) / 4;
  };
  return f(Ny) && f(2 * Nh - 1);
}

template <int R> cudaError_t launch_slab_r(const SlabArgs& a, int warps, cudaStream_t s) {
  return slab_band_free(a.M, a.Ny, a.Nh) ? launch_slab_rz<R, true>(a, warps, s) : launch_slab_rz<R, false>(a, warps, s);
}

// Warps per slab CTA, or 0 when the slab pass does not apply (length not R*R with R in
// {3, 5, 9, 15}, or the slab does not fit in shared memory).
template <typename T> int slab_warps(int M, int Ny, int Nh) {
  int R = 0;
  for (int r : {3, 5, 9, 15})
    if (r * r == M) R = r;
  // FP64 stays on the separate passes: it is bound by the FP64 pipe, and lane groups of R
  // leave 32 mod R lanes of every warp issuing FP64 work on zeros
  if (R == 0 || sizeof(T) == 8) return 0;
  // the warps with the least idle lane groups over the rounds (two rounds of column pairs, weight 1
  // each, and of row groups, weight 2.2), more warps where that ties: zero-padded 225: 15, 81: 7, 25: 1,
  // 9: 1; as long as the data 81: 9, 25: 2, 9: 1
  const bool zb = slab_band_free(M, Ny, Nh);
  const int PW = 32 / R, nc = slab_pairs(R, zb), nquad = (M + 3) / 4;
  int best = 0;
  double best_cost = 1e30;
  for (int w = 1; w * 32 <= kSlabMaxThreads; ++w) {
    if (slab_smem_bytes(R, zb, Ny, Nh, w) > 220 * 1024) break;
    const int slots = w * PW;
    const double cost = w * (2.0 * ((nc + slots - 1) / slots) + 2.2 * ((nquad + slots - 1) / slots)) *
                        (w < 4 && M >= 81 ? 2.0 : 1.0);
    if (cost <= best_cost + 1e-9) {
      best_cost = cost;
      best = w;
    }
  }
  return best;
}

// The same with a caller's choice of warps (0: none), taken where it fits
template <typename T> int slab_warps_asked(int M, int Ny, int Nh, int asked) {
  const int warps = slab_warps<T>(M, Ny, Nh);
  if (warps == 0 || asked <= 0) return warps;
  const int r = M == 225 ? 15 : (M == 81 ? 9 : (M == 25 ? 5 : 3));
  const bool fits = asked * 32 <= slab_wide_threads(r) &&
                    slab_smem_bytes(r, slab_band_free(M, Ny, Nh), Ny, Nh, asked) <= 227 * 1024;
  return fits ? asked : warps;
}

template <typename T> cudaError_t launch_slab(const SlabArgs& a, cudaStream_t s) {
  if constexpr (sizeof(T) != 4) {
    return cudaErrorNotSupported;
  } else {
    const int warps = slab_warps_asked<T>(a.M, a.Ny, a.Nh, a.warps);
    switch (warps ? a.M : 0) {
      case 9: return launch_slab_r<3>(a, warps, s);
      case 25: return launch_slab_r<5>(a, warps, s);
      case 81: return launch_slab_r<9>(a, warps, s);
      case 225: return launch_slab_r<15>(a, warps, s);
      default: return cudaErrorNotSupported;
    }
  }
}

}  // namespace homb

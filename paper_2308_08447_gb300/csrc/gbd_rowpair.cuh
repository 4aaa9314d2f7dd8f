// x-row kernel of the demag convolution for FP32 meshes with open x (Sec. II, Eq. 1; the xFFT_R2C /
// xFFT_C2R steps of Appendix A with one GPU) with the fused exchange (Eq. 4) + LLG (Eq. 5) + RK
// stage epilogue (Sec. III): the arithmetic of row_kernel on two rows at a time.
//
// A thread transforms the same position of two adjacent rows, with the rows' values in the halves of
// f32x2 registers (cpair): half the instructions, shared-memory accesses and twiddle loads per
// value, at the same FMA-pipe time. A block takes NPR row pairs (three pair lines each) and
// 3 NPR L / 16 threads of 16 pair values. Rows are paired along the flattened (z, y) index; a pair's
// spectrum is one 16-byte vector of the [kx][y] spectrum where the two rows are adjacent there.
// Every operation rounds as row_kernel's, so that a mesh may run its transforms in one kernel and its
// stages in the other: a run split over calls equals the unsplit run.
#pragma once
#include "gbd_row.cuh"

namespace gbd {

// Row pairs per block: 192 threads (240 and 288 for lengths 5 * 2^k and 3 * 2^k; more for L above 1024).
__host__ __device__ constexpr int pair_npr(int L) { return 1024 / pow2_floor(L) > 0 ? 1024 / pow2_floor(L) : 1; }
__host__ __device__ constexpr int pair_threads(int L, int npr) { return 3 * npr * L / GBD_E; }
// Blocks per SM: the epilogue's instances at 12 to 16 warps (168 or 128 registers; at 96 they spill and
// the film's stage takes 62 us instead of 47), the transform-only ones at 18 (96 registers; 512x512x64
// forward 238 us at 16 warps, 194 at 18).
__host__ __device__ constexpr int pair_blocks(int T, int kind) {
  const int warps = kind != 1 ? 16 : 18, w = (T + 31) / 32;
  return warps / w < 1 ? 1 : warps / w;
}
template <int L, int NPR>
__host__ __device__ constexpr size_t pair_smem() {
  return (size_t)3 * NPR * line_stride<L, true>() * sizeof(cpair);
}

// The epilogue of the cells (x0, x0 + 1) of the rows y, y + 1 of plane z (linear index idx of the
// first), with the demag field in hd, for every mode but ROW_H: all loads first, then epilogue_pair's
// arithmetic, term for term. Returns true with the next stage's m in mn ([row][cell][component]) for
// the RK stages that have one. Even nx, 8-byte aligned fields, open x. RK4: the modes ROW_RK1 .. 4, or
// the others (one function for both costs the RK4 stages registers).
template <bool RK4>
__device__ __forceinline__ bool epilogue_rows2(const RowArgs& a, int mode, int z, int y, long long idx, int x0,
                                               const float (&hd)[2][2][3], float (&mn)[2][2][3]) {
  const long long N = a.N;
  const int nx = a.nx, ny = a.ny;
  const long long sz = (long long)nx * ny;
  const long long wy = (long long)(ny - 1) * nx, wz = (long long)(a.nz - 1) * sz;
  const long long oym = y > 0 ? -(long long)nx : ((a.per & 2) ? wy : 0);             // below row y
  const long long oyp = y + 1 < ny - 1 ? 2LL * nx : ((a.per & 2) ? nx - wy : nx);    // above row y + 1
  const long long ozm = z > 0 ? -sz : ((a.per & 4) ? wz : 0);
  const long long ozp = z < a.nz - 1 ? sz : ((a.per & 4) ? -wz : 0);
  const int oxl = x0 > 0 ? -1 : 0, oxr = x0 + 2 < nx ? 2 : 1;   // free x boundary
  const bool rk_acc = RK4 && mode != ROW_RK1;
  const bool rkg = !RK4 && mode == ROW_RKG;
  float mv[2][2][3], lap[2][2][3];
  float2 q0[2][3], qa[2][3];   // step-start m; k-sum, or (ROW_RKG) the weighted sum of earlier slopes
  auto ld2 = [](const float* p) { return *reinterpret_cast<const float2*>(p); };
  auto st2 = [](float* p, float x, float y) { *reinterpret_cast<float2*>(p) = make_float2(x, y); };
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float* __restrict__ p = a.ms + c * N + idx;
    const float2 r[4] = {ld2(p + oym), ld2(p), ld2(p + nx), ld2(p + oyp)};
    const float left[2] = {p[oxl], p[nx + oxl]}, right[2] = {p[oxr], p[nx + oxr]};
    float2 zm[2] = {r[1], r[2]}, zp[2] = {r[1], r[2]};
    if (a.nz > 1) {
      zm[0] = ld2(p + ozm);
      zm[1] = ld2(p + ozm + nx);
      zp[0] = ld2(p + ozp);
      zp[1] = ld2(p + ozp + nx);
    }
    if (rk_acc) {
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        q0[u][c] = ld2(a.m0 + c * N + idx + u * nx);
        qa[u][c] = ld2(a.acc + c * N + idx + u * nx);
      }
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const float2 cc = r[u + 1], ym = r[u], yp = r[u + 2];
      mv[u][0][c] = cc.x;
      mv[u][1][c] = cc.y;
      lap[u][0][c] = laplacian(a, cc.x, left[u], cc.y, ym.x, yp.x, zm[u].x, zp[u].x);
      lap[u][1][c] = laplacian(a, cc.y, cc.x, right[u], ym.y, yp.y, zm[u].y, zp[u].y);
    }
  }
  const float hs = rkg && a.hdev ? *a.hdev : 1.f;   // step size on the device, or folded into kw
  if (rkg && a.mnext) {
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int c = 0; c < 3; ++c) q0[u][c] = ld2(a.m0 + c * N + idx + u * nx);
    for (int j = 0; j < a.nk; ++j) {
      const float* kj = a.kin[j] + idx;
      const float w = a.kw[j] * hs;
      float2 k[2][3];
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int c = 0; c < 3; ++c) k[u][c] = ld2(kj + c * N + u * nx);
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          q0[u][c].x = fmaf(w, k[u][c].x, q0[u][c].x);
          q0[u][c].y = fmaf(w, k[u][c].y, q0[u][c].y);
        }
    }
  }
  if (a.hrec) {
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int c = 0; c < 3; ++c) st2(a.hrec + c * N + idx + u * nx, hd[u][0][c], hd[u][1][c]);
  }
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    float m0v[2][3] = {}, accv[2][3] = {}, ao[2][3], res[2][3];
    if (rk_acc) {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        m0v[0][c] = q0[u][c].x;
        m0v[1][c] = q0[u][c].y;
        accv[0][c] = qa[u][c].x;
        accv[1][c] = qa[u][c].y;
      }
    }
    const int lm = rkg ? (int)ROW_RHS : mode;
#pragma unroll
    for (int v = 0; v < 2; ++v)
      llg_update(a, lm, hd[u][v], mv[u][v], lap[u][v], m0v[v], accv[v], mn[u][v], ao[v], res[v]);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const long long o = c * N + idx + u * nx;
      if (!RK4 && !rkg) {
        st2(a.out + o, res[0][c], res[1][c]);
      } else if (rkg) {
        st2(a.kout + o, res[0][c], res[1][c]);
        if (a.mnext) {
          const float w = a.kw[a.nk] * hs;
          mn[u][0][c] = fmaf(w, res[0][c], q0[u][c].x);
          mn[u][1][c] = fmaf(w, res[1][c], q0[u][c].y);
          st2(a.mnext + o, mn[u][0][c], mn[u][1][c]);
        }
      } else if (mode == ROW_RK4) {   // m0_out may alias m0: each cell is read, then written, by one thread
        st2(a.m0_out + o, mn[u][0][c], mn[u][1][c]);
      } else {
        st2(a.acc + o, ao[0][c], ao[1][c]);
        st2(a.mnext + o, mn[u][0][c], mn[u][1][c]);
      }
    }
  }
  return RK4 || (rkg && a.mnext);
}

// KIND 0: the RK4 stages; KIND 1: the forward transform, and the inverse transform to hscale * H_d;
// KIND 2: the other epilogues (H_eff, dm/dt, general RK stages; in one instance with the RK4 stages
// their code costs those 3 %).
template <int L, int NPR, int KIND>
__global__ void __launch_bounds__(pair_threads(L, NPR), pair_blocks(pair_threads(L, NPR), KIND))
    row_pair_kernel(const __grid_constant__ RowArgs a, const float2* __restrict__ tw) {
  constexpr int LINES = 3 * NPR;
  constexpr int T = pair_threads(L, NPR);
  constexpr int LS = line_stride<L, true>();
  constexpr int NP = npasses(L, false);
  constexpr int HX = L + 1, HALF = L / 2, LT = L / GBD_E;
  constexpr int R0 = radix_at(L, false, 0);
  extern __shared__ cpair smp[];
  const int r0 = blockIdx.x * 2 * NPR;
  const long long N = a.N;
  const int mode = a.mode, nx = a.nx, ny = a.ny;
  const int tid = threadIdx.x;
  if constexpr (KIND == 0) __builtin_assume(mode >= ROW_RK1 && mode <= ROW_RK4);
  if constexpr (KIND == 2) __builtin_assume(mode == ROW_HEFF || mode == ROW_RHS || mode == ROW_RKG);
  // transform items: pair line (g, c) and positions jj + i L/16
  const int tg = tid % NPR, tt = tid / NPR, jj = tt % LT, tc = tt / LT;
  cpair* const tl = smp + (tc * NPR + tg) * LS;
  const bool vec = (ny & 1) == 0;   // the rows of a pair are adjacent in the spectrum
  const int rowa = r0 + 2 * tg;
  const bool oka = rowa < a.rows, okb = rowa + 1 < a.rows;
  float2 *Sa, *Sb;                  // the rows' spectra of component tc, at k = 0
  {
    const int za = rowa / ny, ya = rowa - za * ny;
    const int zb = ya + 1 < ny ? za : za + 1, yb = ya + 1 < ny ? ya + 1 : 0;
    Sa = a.S + (long long)(tc * a.nz + za) * HX * ny + ya;
    Sb = a.S + (long long)(tc * a.nz + zb) * HX * ny + yb;
  }
  auto sload = [&](long long o) {
    cpair v = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
    if (vec) {
      if (oka) {
        const float4 q = *reinterpret_cast<const float4*>(Sa + o);
        v = {make_float2(q.x, q.z), make_float2(q.y, q.w)};
      }
    } else {
      if (oka) {
        const float2 q = Sa[o];
        v.x.x = q.x;
        v.y.x = q.y;
      }
      if (okb) {
        const float2 q = Sb[o];
        v.x.y = q.x;
        v.y.y = q.y;
      }
    }
    return v;
  };
  auto sstore = [&](long long o, cpair v) {
    if (vec) {
      if (oka) *reinterpret_cast<float4*>(Sa + o) = make_float4(v.x.x, v.y.x, v.x.y, v.y.y);
    } else {
      if (oka) Sa[o] = make_float2(v.x.x, v.y.x);
      if (okb) Sb[o] = make_float2(v.x.y, v.y.y);
    }
  };
  auto conj = [](cpair v) { return cpair{v.x, pneg(v.y)}; };
  const long long kstep = (long long)LT * ny;
  pdl_wait_then_release();

  if (KIND != 1 || mode != ROW_FWD) {
    if (KIND == 1 || !a.extrap) {
      // 1. X[k], X[L - k] -> Z[k], Z[L - k], k = jj + i L/16 < L/2 (k = 0 with X[L], and X[L/2] alone):
      //    every thread issues all its loads before using any
      constexpr int NI = GBD_E / 2;
      cpair A[NI], B[NI];
#pragma unroll
      for (int i = 0; i < NI; ++i) {
        A[i] = sload(jj * (long long)ny + i * kstep);
        B[i] = sload((L - jj) * (long long)ny - i * kstep);
      }
      cpair M;
      if (jj == 0) M = sload((long long)HALF * ny);
#pragma unroll
      for (int i = 0; i < NI; ++i) {
        const int k = jj + i * LT;
        const float2 wp = twiddle_at<-1>(tw, 2 * L, k);
        const cpair s1 = cadd(A[i], conj(B[i])), d1 = csub(A[i], conj(B[i]));
        if (i == 0 && jj == 0) {
          tl[pad(0)] = cadd_i<1>(s1, d1);
          tl[pad(HALF)] = cadd_i<1>(cadd(M, conj(M)), cmul(cconj(twiddle_at<-1>(tw, 2 * L, HALF)), csub(M, conj(M))));
        } else {
          // with t = W^-k (A - B*): Z[k] = s1 + i t, Z[L - k] = (s1 - i t)*
          const cpair t = cmul(cconj(wp), d1);
          tl[pad(k)] = cadd_i<1>(s1, t);
          tl[pad(L - k)] = conj(cadd_i<-1>(s1, t));
        }
      }
      __syncthreads();
      // 2. unnormalised inverse FFT: adjoint passes, the last one keeping the lower half
      adj_passes_smem<1, L, false, LINES, false, LS, NP, 1, 0>(smp, tw);
      if constexpr (R0 % 2 == 0) {
        stockham_pass_sm<1, true, L, R0, 1, LINES, false, LS, true>(smp, tw);
      } else {
        stockham_pass<1, true, L, R0, 1, LINES, false, true>(
            tw, [&](int l, int i) { return smp[l * LS + pad(i)]; },
            [&](int l, int i, cpair v) {
              if (i < HALF) smp[l * LS + pad(i)] = v;
            });
      }
      __syncthreads();
    }
    // 3. epilogue
    if constexpr (KIND == 1) {   // ROW_H
      const int NX2 = (nx + 1) / 2;
      const bool v8 = (nx & 1) == 0 && a.vec8;
      for (int e = tid; e < LINES * NX2; e += T) {
        const int line = e / NX2, p = e - line * NX2;
        const int c = line / NPR, row = r0 + 2 * (line - c * NPR);
        const cpair h = smp[line * LS + pad(p)];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          if (row + u >= a.rows) continue;
          const float2 v = u == 0 ? make_float2(h.x.x * a.hscale, h.y.x * a.hscale)
                                  : make_float2(h.x.y * a.hscale, h.y.y * a.hscale);
          const long long idx = c * N + (long long)(row + u) * nx + 2 * p;
          if (v8) {
            if (a.hrec) *reinterpret_cast<float2*>(a.hrec + idx) = v;
            *reinterpret_cast<float2*>(a.out + idx) = v;
          } else {
            if (a.hrec) a.hrec[idx] = v.x;
            a.out[idx] = v.x;
            if (2 * p + 1 < nx) {
              if (a.hrec) a.hrec[idx + 1] = v.y;
              a.out[idx + 1] = v.y;
            }
          }
        }
      }
      return;
    } else {
      auto field = [&](int g, int p, float (&hd)[2][2][3]) {   // [row][cell][component]
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const cpair h = smp[(c * NPR + g) * LS + pad(p)];
          hd[0][0][c] = h.x.x * a.hscale;
          hd[1][0][c] = h.x.y * a.hscale;
          hd[0][1][c] = h.y.x * a.hscale;
          hd[1][1][c] = h.y.y * a.hscale;
        }
      };
      if ((nx & 1) == 0 && a.vec8) {
        const int NP2 = nx / 2;
        for (int e = tid; e < NPR * NP2; e += T) {
          const int g = NPR == 1 ? 0 : e / NP2, p = e - g * NP2;
          const int row = r0 + 2 * g;
          if (row >= a.rows) continue;
          const int z = row / ny, y = row - z * ny;
          const long long idx = (long long)row * nx + 2 * p;
          float hd[2][2][3], mn[2][2][3] = {};
          if (!a.extrap) field(g, p, hd);
          bool next = a.fwd_after != 0;
          if (!a.extrap && y + 1 < ny) {
            next = epilogue_rows2<KIND == 0>(a, mode, z, y, idx, 2 * p, hd, mn) && next;
          } else {
#pragma unroll 1
            for (int u = 0; u < 2; ++u) {
              if (row + u >= a.rows) break;
              const int yu = y + u < ny ? y + u : 0, zu = y + u < ny ? z : z + 1;
              float h1[2][3], m1[2][3];
#pragma unroll
              for (int v = 0; v < 2; ++v)
#pragma unroll
                for (int c = 0; c < 3; ++c) h1[v][c] = u == 0 ? hd[0][v][c] : hd[1][v][c];
              if (a.extrap) extrap_pair(a, idx + u * nx, h1);
              next = epilogue_pair<false>(a, mode, zu, yu, idx + u * nx, 2 * p, 0, h1, m1) && next;
#pragma unroll
              for (int v = 0; v < 2; ++v)
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                  if (u == 0)
                    mn[0][v][c] = m1[v][c];
                  else
                    mn[1][v][c] = m1[v][c];
                }
            }
          }
          if (next) {
#pragma unroll
            for (int c = 0; c < 3; ++c)
              smp[(c * NPR + g) * LS + pad(p)] = {make_float2(mn[0][0][c], mn[1][0][c]), make_float2(mn[0][1][c], mn[1][1][c])};
          }
        }
      } else {
        // general path: one cell per item
        for (int e = tid; e < 2 * NPR * nx; e += T) {
          const int rr = e / nx, x = e - rr * nx, row = r0 + rr;
          if (row >= a.rows) continue;
          const int z = row / ny, y = row - z * ny;
          const long long idx = (long long)row * nx + x;
          float* at = reinterpret_cast<float*>(smp + (rr >> 1) * LS + pad(x >> 1)) + 2 * (x & 1) + (rr & 1);
          constexpr int CS = 4 * NPR * LS;   // floats between components
          float hd[3], mn[3];
          if (a.extrap) {
            extrap_cell(a, idx, hd);
          } else {
#pragma unroll
            for (int c = 0; c < 3; ++c) hd[c] = at[c * CS] * a.hscale;
          }
          if (epilogue_cell(a, mode, z, y, x, idx, hd, mn) && a.fwd_after) {
#pragma unroll
            for (int c = 0; c < 3; ++c) at[c * CS] = mn[c];
          }
        }
      }
      if (!a.fwd_after) return;   // uniform over the grid
    }
  } else {
    // the input rows
    const int NX2 = (nx + 1) / 2;
    const bool v8 = (nx & 1) == 0 && a.vec8;
    constexpr int U = 4;
    for (int e0 = tid; e0 < LINES * NX2; e0 += U * T) {
      cpair v[U];
#pragma unroll
      for (int i = 0; i < U; ++i) {
        const int e = e0 + i * T;
        v[i] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
        if (e < LINES * NX2) {
          const int line = e / NX2, p = e - line * NX2;
          const int c = line / NPR, row = r0 + 2 * (line - c * NPR);
          const float* in = a.in + c * N + (long long)row * nx + 2 * p;
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            if (row + u >= a.rows) continue;
            float2 q;
            if (v8)
              q = *reinterpret_cast<const float2*>(in + u * nx);
            else
              q = make_float2(in[u * nx], 2 * p + 1 < nx ? in[u * nx + 1] : 0.f);
            if (u == 0) {
              v[i].x.x = q.x;
              v[i].y.x = q.y;
            } else {
              v[i].x.y = q.x;
              v[i].y.y = q.y;
            }
          }
        }
      }
#pragma unroll
      for (int i = 0; i < U; ++i) {
        const int e = e0 + i * T;
        if (e < LINES * NX2) {
          const int line = e / NX2;
          smp[line * LS + pad(e - line * NX2)] = v[i];
        }
      }
    }
  }
  // 4. zero what the forward transform reads beyond the data (cells nx .. L - 1; rows past the last)
  {
    const int p0 = KIND == 1 ? (nx + 1) / 2 : nx / 2;   // first element with a zero cell
    for (int line = 0; line < LINES; ++line) {
      float4* fl = reinterpret_cast<float4*>(smp + line * LS);
      for (int p = p0 + tid; p < HALF; p += T) {
        if (2 * p < nx) {   // the last cell of an odd row, and one zero
          float2* q = reinterpret_cast<float2*>(fl + pad(p));
          q[1] = make_float2(0.f, 0.f);
        } else {
          fl[pad(p)] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
      }
    }
    if (KIND != 1 && r0 + 2 * NPR > a.rows) {
      for (int rr = 0; rr < 2 * NPR; ++rr)
        if (r0 + rr >= a.rows)
          for (int c = 0; c < 3; ++c)
            for (int x = tid; x < nx; x += T)
              reinterpret_cast<float*>(smp + (c * NPR + (rr >> 1)) * LS + pad(x >> 1))[2 * (x & 1) + (rr & 1)] = 0.f;
    }
  }
  __syncthreads();
  // 5. forward FFT; the first pass reads the lower half only
  if constexpr (R0 % 2 == 0) {
    stockham_pass_sm<-1, false, L, R0, 1, LINES, false, LS, true>(smp, tw);
  } else {
    stockham_pass<-1, false, L, R0, 1, LINES, false, true>(
        tw,
        [&](int l, int i) {
          return i < HALF ? smp[l * LS + pad(i)] : cpair{make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
        },
        [&](int l, int i, cpair v) { smp[l * LS + pad(i)] = v; });
  }
  __syncthreads();
  fwd_passes_smem<-1, L, false, LINES, false, LS, 1, NP, 0>(smp, tw);
  // 6. Z -> X pairwise and store the half spectrum
#pragma unroll 2
  for (int i = 0; i < GBD_E / 2; ++i) {
    const int k = jj + i * LT;
    const long long oa = jj * (long long)ny + i * kstep, ob = (L - jj) * (long long)ny - i * kstep;
    const cpair A = tl[pad(k)];
    if (i == 0 && jj == 0) {
      const float2 zero = make_float2(0.f, 0.f);
      sstore(oa, {padd(A.x, A.y), zero});   // X[0]
      sstore(ob, {psub(A.x, A.y), zero});   // X[L]
      const cpair Mz = tl[pad(HALF)];       // X[L/2], of one Z
      sstore((long long)HALF * ny,
             cscale(cadd_i<-1>(cadd(Mz, conj(Mz)), cmul(twiddle_at<-1>(tw, 2 * L, HALF), csub(Mz, conj(Mz)))), 0.5f));
    } else {
      const cpair B = tl[pad(L - k)];
      const float2 wp = twiddle_at<-1>(tw, 2 * L, k);
      // with s = A + B*, t = W^k (A - B*): X[k] = (s - i t)/2, X[L - k] = ((s + i t)/2)*
      const cpair s1 = cadd(A, conj(B)), t = cmul(wp, csub(A, conj(B)));
      sstore(oa, cscale(cadd_i<-1>(s1, t), 0.5f));
      sstore(ob, conj(cscale(cadd_i<1>(s1, t), 0.5f)));
    }
  }
}

// ---- launcher --------------------------------------------------------------------------------
// Calls f(std::integral_constant<int, L>) for a power-of-two (G = 0) or mixed (G = 1) length with
// kernels; false for any other.
template <int G, class F>
static bool pair_switch(int L, F f) {
#define GBD_PAIR_LEN(N)                  \
  case N:                                \
    f(std::integral_constant<int, N>()); \
    return true;
  if constexpr (G == 0) {
    switch (L) {
      GBD_PAIR_LEN(32)
      GBD_PAIR_LEN(64)
      GBD_PAIR_LEN(128)
      GBD_PAIR_LEN(256)
      GBD_PAIR_LEN(512)
      GBD_PAIR_LEN(1024)
      GBD_PAIR_LEN(2048)
      default: return false;
    }
  } else {
    switch (L) {
      GBD_PAIR_LEN(96)
      GBD_PAIR_LEN(160)
      GBD_PAIR_LEN(192)
      GBD_PAIR_LEN(320)
      GBD_PAIR_LEN(384)
      GBD_PAIR_LEN(640)
      GBD_PAIR_LEN(768)
      GBD_PAIR_LEN(1280)
      GBD_PAIR_LEN(1536)
      GBD_PAIR_LEN(2560)
      GBD_PAIR_LEN(3072)
      default: return false;
    }
  }
#undef GBD_PAIR_LEN
}

template <int L, int NPR, int KIND>
static void pair_launch_t(const RowArgs* a, const float2* tw, cudaStream_t st) {
  constexpr size_t smem = pair_smem<L, NPR>();
  prep(row_pair_kernel<L, NPR, KIND>, smem);
  if (a) launch_pdl(row_pair_kernel<L, NPR, KIND>, (a->rows + 2 * NPR - 1) / (2 * NPR), pair_threads(L, NPR), smem, st, *a, tw);
}

// Launches (a == nullptr: prepares) the kernel of length L and kind KIND. The transform-only launches
// halve a tile of four or more pairs that would leave SMs without a block (192x224x8 demag 54.9 ->
// 51.7 us, 64x64x64 36.7 -> 34.6); a tile of one pair reads half sectors and is slower (512x512x1 23.3
// -> 29.6), and the RK stages keep the larger tile (128x128x16 33.7 us, halved 37.1).
template <int L, int KIND>
static void pair_launch(const RowArgs* a, const float2* tw, cudaStream_t st) {
  constexpr int P = pair_npr(L);
  if constexpr (KIND == 1 && P >= 4) {
    const bool few = a && (a->rows + 2 * P - 1) / (2 * P) < kTileBlocks;
    if (!a || few) pair_launch_t<L, P / 2, KIND>(a, tw, st);
    if (few) return;
  }
  pair_launch_t<L, P, KIND>(a, tw, st);
}

}  // namespace gbd

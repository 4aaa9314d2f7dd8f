// Kernels for meshes too small to fill the GPU (FP32): the x rows (Sec. II, Eq. 1; xFFT_R2C /
// xFFT_C2R of Appendix A, with the exchange + LLG + RK stage epilogue of Sec. III) and the
// convolution along y and z in one launch.
//
// On such meshes a launch of row_kernel or of the convolution kernels takes as long as one of its
// blocks: a few thousand instructions of straight-line code per thread, each fetched once from
// L2 and waited for. These kernels shorten that chain instead of raising throughput:
//   - 8 complex values per thread and pass (radix 8), so a thread runs about a third of the
//     instructions, on blocks of one or two rows or one kx column, so that every SM has work;
//   - the transform lengths are run-time values and the passes a loop, so one small body is
//     fetched once for all passes of both directions;
//   - the passes go back and forth between two shared-memory buffers: one barrier per pass;
//   - what does not depend on the launch before -- twiddles (copied to shared memory) and, for the
//     RK stages, the field rows (bulk copies) -- is requested before the dependent-launch wait;
//   - y FFT, z FFT, product and the inverses of one kx run in one block with the z transform in
//     registers, so the y spectrum never leaves shared memory (one launch instead of three).
// The arithmetic does not depend on the tile variant or on how the rows are grouped.
#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "gbd_row.cuh"

namespace gbd {

// Radix passes of length L = r 2^k (r in {1, 3, 5}, 2^k >= 16): the odd radix, as in the other kernels,
// then radix 8 and 4. (The odd radix last keeps Ns a power of two, but costs accuracy: 150x150x6 field,
// rms error 1.57e-7 against 1.30e-7.)
struct FftPlan {
  int L, np;
  int ls;                    // float2 slots per line
  int radix[6], ns[6];
  int twoff[6];              // first of the pass's twiddles in the shared table
  unsigned kdiv[6];          // floor(j / Ns) = umulhi(j, kdiv) for j < 2^16 (0: Ns = 1)
  unsigned mdiv[6];          // floor(b / (L / R)) = umulhi(b, mdiv) for b < 2^16
  int ntw;                   // shared twiddles of all passes
};
// Element i of a line sits at i + i / 16, or, where the first radix is odd (ODD), at i: the writes of a
// first pass of radix 8 or 4 then miss each other's banks, and so do those of radix 3 or 5, of which the
// pad would put five into one bank (320x320x4 field 64.9 -> 62.9 us).
template <bool ODD>
__host__ __device__ __forceinline__ constexpr int at(int i) {
  return ODD ? i : i + (i >> 4);
}
static unsigned magic_div(unsigned d) { return d <= 1 ? 0u : (unsigned)((0x100000000ull + d - 1) / d); }
__device__ __forceinline__ int fast_div(int b, unsigned m) { return m ? (int)__umulhi((unsigned)b, m) : b; }

static bool make_fft_plan(int L, FftPlan& f) {
  const int r = odd_part(L);
  if (L < 16 || r > 5 || (r > 1 && L / r < 16)) return false;
  f.L = L;
  f.np = 0;
  if (r > 1) f.radix[f.np++] = r;
  int k = ilog2(L / r);
  while (k > 0) {
    const int b = (k == 4 || k == 2) ? 2 : 3;   // k >= 4: ends 8, 8 4 or 4 4, never with a radix 2
    f.radix[f.np++] = 1 << b;
    k -= b;
  }
  int ns = 1, off = 0;
  for (int p = 0; p < f.np; ++p) {
    f.ns[p] = ns;
    f.twoff[p] = off;
    if (p > 0) off += (f.radix[p] - 1) * ns;
    f.mdiv[p] = magic_div(L / f.radix[p]);
    f.kdiv[p] = magic_div(ns);
    ns *= f.radix[p];
  }
  f.ntw = off;
  // unpadded lines start L / 8 banks of two apart, so that the radix-8 reads of a half warp run on from one
  // line to the next (L = 96: 1.28 wavefronts per access instead of 1.60)
  f.ls = r > 1 ? L + std::max(1, (L / 8 - L) & 15) : at<false>(L) | 1;
  return true;
}

// Copies the passes' twiddles into shared memory: pass p holds w^e, 0 < e < R, at [e - 1][k], w =
// exp(-2 pi i / (Ns R)). Every power comes from the table: products of powers (three loads instead of
// seven for R = 8) add their own roundings (32x32x8 field, rms error 1.89e-7 against 1.55e-7) at the same
// time.
__device__ __forceinline__ void load_twiddles(const FftPlan& f, float2* stw, const float2* __restrict__ tw) {
  for (int p = 1; p < f.np; ++p) {
    const int R = f.radix[p], ns = f.ns[p], n = (R - 1) * ns;
    const float2* lev = tw + tw_base(ns * R);
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      const int e = fast_div(i, f.kdiv[p]);
      stw[f.twoff[p] + i] = __ldg(lev + (i - e * ns) * (e + 1));
    }
  }
}

__device__ __forceinline__ void prefetch_l1(const void* p) { asm volatile("prefetch.global.L1 [%0];\n" ::"l"(p)); }

// One radix-R butterfly: twiddles from the shared table (sign S), DFT.
template <int S, int R>
__device__ __forceinline__ void small_butterfly(float2* v, const float2* __restrict__ t, int k, int ns) {
  if (ns > 1) {
#pragma unroll
    for (int e = 1; e < R; ++e) {
      const float2 w = t[(e - 1) * ns + k];
      v[e] = cmul(v[e], S < 0 ? w : cconj(w));
    }
  }
  dft<R, S>(v);
}

// Pass p over `lines` lines: LD(line, i) -> element i, ST(line, i, v). Stockham: reads j + r L/R,
// writes (j - k) R + k + q Ns.
template <int S, int R, bool ODD, class LD, class ST>
__device__ __forceinline__ void small_pass_r(const FftPlan& f, int p, int lines, const float2* __restrict__ stw, LD ld, ST st) {
  const int LR = f.L / R, ns = f.ns[p];
  for (int b = threadIdx.x; b < lines * LR; b += blockDim.x) {
    const int line = fast_div(b, f.mdiv[p]);
    const int j = b - line * LR;
    const int k = ODD ? j - fast_div(j, f.kdiv[p]) * ns : j & (ns - 1);
    float2 v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = ld(line, j + r * LR);
    small_butterfly<S, R>(v, stw + f.twoff[p], k, ns);
    const int base = (j - k) * R + k;
#pragma unroll
    for (int q = 0; q < R; ++q) st(line, base + q * ns, v[q]);
  }
}
template <int S, bool ODD, class LD, class ST>
__device__ __forceinline__ void small_pass(const FftPlan& f, int p, int lines, const float2* __restrict__ stw, LD ld, ST st) {
  const int R = f.radix[p];
  if (R == 8)
    small_pass_r<S, 8, ODD>(f, p, lines, stw, ld, st);
  else if (!ODD || R == 4)
    small_pass_r<S, 4, ODD>(f, p, lines, stw, ld, st);
  else if (R == 3)
    small_pass_r<S, 3, ODD>(f, p, lines, stw, ld, st);
  else
    small_pass_r<S, 5, ODD>(f, p, lines, stw, ld, st);
}
// Passes [p0, p1) between the buffers, starting from x; returns the buffer that holds the result.
// A barrier precedes each pass.
template <int S, bool ODD>
__device__ __forceinline__ float2* small_passes(const FftPlan& f, int p0, int p1, int lines, const float2* __restrict__ stw,
                                                float2* x, float2* y) {
  for (int p = p0; p < p1; ++p) {
    __syncthreads();
    const float2* src = x;
    float2* dst = y;
    small_pass<S, ODD>(f, p, lines, stw, [&](int l, int i) { return src[l * f.ls + at<ODD>(i)]; },
                  [&](int l, int i, float2 v) { dst[l * f.ls + at<ODD>(i)] = v; });
    y = x;
    x = dst;
  }
  return x;
}

// ---- x rows --------------------------------------------------------------------------------

struct SmallRowArgs {
  RowArgs a;
  FftPlan f;
  int rb_log;            // rows per block = 2^rb_log
  unsigned mhalf;        // division by Lx / 2 + 1
  unsigned mnp2, mnx;    // division by nx / 2 and nx
  unsigned mpad;         // division by the zero padding of a line, L - nx
  unsigned mny;          // division by ny (0: ny = 1), rows < 2^16
  int staged;            // the RK stage's field rows come by bulk copies: bit 0 the stage input's rows,
                         // bit 1 those of the planes below and above, bit 2 step-start m and k-sum
};

// Staged rows of a block (floats [row][3][nx]): stage input m on the rows y0 - 1 .. y0 + RB, on the
// RB rows of the planes below and above (nz > 1), step-start m and k-sum on the RB rows (stages 2-4).
__host__ __device__ __forceinline__ int small_stage_rows(int RB, int staged) {
  return (staged & 1) ? RB + 2 + ((staged & 2) ? 2 * RB : 0) + ((staged & 4) ? 2 * RB : 0) : 0;
}

// ODD: Lx is 3 * 2^k or 5 * 2^k.
template <bool ODD>
__global__ void __launch_bounds__(384, 2) small_row_kernel(const __grid_constant__ SmallRowArgs s, const float2* __restrict__ tw) {
  const RowArgs& a = s.a;
  const FftPlan& f = s.f;
  const int T = blockDim.x, tid = threadIdx.x;
  const int RB = 1 << s.rb_log, L = f.L, HALF = L / 2, HX = L + 1, lines = 3 * RB;
  const int nx = a.nx, ny = a.ny, mode = a.mode;
  const long long N = a.N;
  const bool xper = (a.per & 1) != 0;
  extern __shared__ float2 sm[];
  float2* X = sm;
  float2* Y = X + lines * f.ls;
  float2* stw = Y + lines * f.ls;
  float2* shw = stw + f.ntw;                                   // exp(-2 pi i k / Px), k <= L / 2
  float* sF = reinterpret_cast<float*>(sm + ((2 * lines * f.ls + f.ntw + HALF + 2) & ~1));   // staged rows, 16-byte aligned
  const int r0 = blockIdx.x << s.rb_log;
  const int zb = s.mny ? (int)__umulhi((unsigned)r0, s.mny) : r0, yb = r0 - zb * ny;
  auto row_zy = [&](int rr, int& z, int& y) {
    y = yb + rr;
    z = zb;
    while (y >= ny) {
      y -= ny;
      ++z;
    }
  };
  const bool rk_acc = mode != ROW_RK1;
  // staged launches: ny a multiple of RB, so the block's rows lie in plane zb
  float* sZ = sF + (RB + 2) * 3 * nx;                          // planes zb - 1, zb + 1
  float* sA = sZ + ((s.staged & 2) ? 2 * RB * 3 * nx : 0);           // m0, k-sum
  unsigned long long* sbar = reinterpret_cast<unsigned long long*>(sF + small_stage_rows(RB, s.staged) * 3 * nx);
  if (s.staged && tid == 0) {
    // written by x-row launches before the preceding convolution launch, so complete once this
    // block runs (gbd_launch.cuh): requested before the wait for the preceding launch
    mbar_init(sbar, 1);
    mbar_expect_tx(sbar, (unsigned)(small_stage_rows(RB, s.staged) * 3 * nx * 4) + a.stage_extra);
    const long long plane = (long long)zb * ny;
    const unsigned bytes = (unsigned)(nx * 4);
    for (int c = 0; c < 3; ++c) {
      const float* p = a.ms + c * N;
      for (int q = 0; q < RB + 2; ++q) {
        int y = yb - 1 + q;
        if (y < 0) y = (a.per & 2) ? ny - 1 : 0;
        if (y >= ny) y = (a.per & 2) ? 0 : ny - 1;
        bulk_g2s(sF + (q * 3 + c) * nx, p + (plane + y) * nx, bytes, sbar);
      }
      for (int q = 0; q < RB; ++q) {
        const long long row = plane + yb + q;
        if (s.staged & 2) {
          const int zm = zb > 0 ? zb - 1 : ((a.per & 4) ? a.nz - 1 : 0);
          const int zp = zb < a.nz - 1 ? zb + 1 : ((a.per & 4) ? 0 : a.nz - 1);
          bulk_g2s(sZ + (q * 3 + c) * nx, p + ((long long)zm * ny + yb + q) * nx, bytes, sbar);
          bulk_g2s(sZ + ((RB + q) * 3 + c) * nx, p + ((long long)zp * ny + yb + q) * nx, bytes, sbar);
        }
        if (s.staged & 4) {
          bulk_g2s(sA + (q * 3 + c) * nx, a.m0 + c * N + row * nx, bytes, sbar);
          bulk_g2s(sA + ((RB + q) * 3 + c) * nx, a.acc + c * N + row * nx, bytes, sbar);
        }
      }
    }
  }
  load_twiddles(f, stw, tw);
  for (int k = tid; k <= HALF; k += T) shw[k] = __ldg(tw + tw_base(2 * L) + k);
  pdl_wait_then_release();
  __syncthreads();

  if (mode != ROW_FWD && !a.extrap) {
    // 1. X[k], X[L - k] (global, [kx][y] layout) -> Z in the lines; all loads of a thread first
    constexpr int IPT = 5;   // covers T >= 3 RB L / 8; a block with more threads runs fewer
    const int items = lines * (HALF + 1), rounds = (items + T - 1) / T;
    for (int e0 = tid; e0 < items; e0 += IPT * T) {
      float2 A[IPT], B[IPT];
#pragma unroll
      for (int i = 0; i < IPT; ++i) {
        if (i >= rounds) break;
        const int e = e0 + i * T;
        A[i] = B[i] = make_float2(0.f, 0.f);
        if (e < items) {
          const int rr = e & (RB - 1), t2 = e >> s.rb_log;
          const int c = fast_div(t2, s.mhalf), k = t2 - c * (HALF + 1);
          if (r0 + rr < a.rows) {
            int z, y;
            row_zy(rr, z, y);
            const float2* base = a.S + (long long)(c * a.nz + z) * HX * ny + y;
            A[i] = base[(long long)k * ny];
            B[i] = base[(long long)(L - k) * ny];
          }
        }
      }
#pragma unroll
      for (int i = 0; i < IPT; ++i) {
        if (i >= rounds) break;
        const int e = e0 + i * T;
        if (e < items) {
          const int rr = e & (RB - 1), t2 = e >> s.rb_log;
          const int c = fast_div(t2, s.mhalf), k = t2 - c * (HALF + 1);
          const float2 wp = shw[k], wm = cconj(wp);
          const float2 Au = A[i], Bu = B[i];
          float2* D = X + (c * RB + rr) * f.ls;
          if (k == 0) {
            D[at<ODD>(0)] = cadd(cadd(Au, cconj(Bu)), cmul_i<1>(csub(Au, cconj(Bu))));
          } else {
            D[at<ODD>(k)] = cadd(cadd(Au, cconj(Bu)), cmul_i<1>(cmul(wm, csub(Au, cconj(Bu)))));
            if (k != L - k) D[at<ODD>(L - k)] = csub(cadd(Bu, cconj(Au)), cmul_i<1>(cmul(wp, csub(Bu, cconj(Au)))));
          }
        }
      }
    }
    // 2. unnormalised inverse FFT
    float2* R = small_passes<1, ODD>(f, 0, f.np, lines, stw, X, Y);
    if (R != X) {
      Y = X;
      X = R;
    }
    __syncthreads();
  }
  if (mode != ROW_FWD) {
    if (s.staged && !mbar_wait(sbar, 0, GBD_WAIT_LIMIT_NS) && a.status) atomicOr(a.status, GBD_DEV_WAIT_TIMEOUT);
    // 3. epilogue; element x of a row is float 2 at<ODD>(x / 2) + (x & 1) of its line
    if (s.staged) {
      const int NP2 = nx / 2;
      const long long sz = (long long)nx * ny;
      const long long ozm = zb > 0 ? -sz : ((a.per & 4) ? (a.nz - 1) * sz : 0);
      const long long ozp = zb < a.nz - 1 ? sz : ((a.per & 4) ? -(a.nz - 1) * sz : 0);
      for (int e = tid; e < RB * NP2; e += T) {
        const int rr = fast_div(e, s.mnp2), xp = e - rr * NP2, x0 = 2 * xp;
        const long long idx = (long long)(r0 + rr) * nx + x0;
        float hd[2][3], mv[2][3], lap[2][3], m0v[2][3] = {}, accv[2][3] = {}, mn[2][3], ao[2][3], res[2][3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const float2 h2 = X[(c * RB + rr) * f.ls + at<ODD>(xp)];
          hd[0][c] = h2.x * a.hscale;
          hd[1][c] = h2.y * a.hscale;
          if (a.hrec) *reinterpret_cast<float2*>(a.hrec + c * N + idx) = make_float2(hd[0][c], hd[1][c]);
          auto at = [&](const float* b, int row) { return *reinterpret_cast<const float2*>(b + (row * 3 + c) * nx + x0); };
          const float* rc = sF + ((rr + 1) * 3 + c) * nx;
          const float2 cc = at(sF, rr + 1), ym = at(sF, rr), yp = at(sF, rr + 2);
          const float left = x0 > 0 ? rc[x0 - 1] : cc.x;          // free x boundary
          const float right = x0 + 2 < nx ? rc[x0 + 2] : cc.y;
          float2 zm = cc, zp = cc;
          if (s.staged & 2) {
            zm = at(sZ, rr);
            zp = at(sZ, RB + rr);
          } else if (a.nz > 1) {
            zm = *reinterpret_cast<const float2*>(a.ms + c * N + idx + ozm);
            zp = *reinterpret_cast<const float2*>(a.ms + c * N + idx + ozp);
          }
          mv[0][c] = cc.x;
          mv[1][c] = cc.y;
          lap[0][c] = laplacian(a, cc.x, left, cc.y, ym.x, yp.x, zm.x, zp.x);
          lap[1][c] = laplacian(a, cc.y, cc.x, right, ym.y, yp.y, zm.y, zp.y);
          if (rk_acc) {
            const float2 q0 = (s.staged & 4) ? at(sA, rr) : *reinterpret_cast<const float2*>(a.m0 + c * N + idx);
            const float2 qa = (s.staged & 4) ? at(sA, RB + rr) : *reinterpret_cast<const float2*>(a.acc + c * N + idx);
            m0v[0][c] = q0.x;
            m0v[1][c] = q0.y;
            accv[0][c] = qa.x;
            accv[1][c] = qa.y;
          }
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) llg_update(a, mode, hd[u], mv[u], lap[u], m0v[u], accv[u], mn[u], ao[u], res[u]);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const float2 v = make_float2(mn[0][c], mn[1][c]);
          if (mode == ROW_RK4) {
            *reinterpret_cast<float2*>(a.m0_out + c * N + idx) = v;
          } else {
            *reinterpret_cast<float2*>(a.acc + c * N + idx) = make_float2(ao[0][c], ao[1][c]);
            *reinterpret_cast<float2*>(a.mnext + c * N + idx) = v;
          }
          X[(c * RB + rr) * f.ls + at<ODD>(xp)] = v;
        }
      }
    } else if (mode == ROW_H) {
      for (int e = tid; e < lines * nx; e += T) {
        const int line = fast_div(e, s.mnx), x = e - line * nx;
        const int rr = line & (RB - 1), c = line >> s.rb_log;
        if (r0 + rr >= a.rows) continue;
        const float v = reinterpret_cast<const float*>(X + line * f.ls)[2 * at<ODD>(x >> 1) + (x & 1)] * a.hscale;
        const long long idx = c * N + (long long)(r0 + rr) * nx + x;
        if (a.hrec) a.hrec[idx] = v;
        a.out[idx] = v;
      }
    } else if ((nx & 1) == 0 && a.vec8) {
      const int NP2 = nx / 2;
      for (int e = tid; e < RB * NP2; e += T) {
        const int rr = fast_div(e, s.mnp2), xp = e - rr * NP2;
        if (r0 + rr >= a.rows) continue;
        int z, y;
        row_zy(rr, z, y);
        const long long idx = (long long)(r0 + rr) * nx + 2 * xp;
        float hd[2][3], mn[2][3];
        if (a.extrap) {
          extrap_pair(a, idx, hd);
        } else {
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            const float2 h2 = X[(c * RB + rr) * f.ls + at<ODD>(xp)];
            hd[0][c] = h2.x * a.hscale;
            hd[1][c] = h2.y * a.hscale;
          }
        }
        if (epilogue_pair<false>(a, mode, z, y, idx, 2 * xp, 0, hd, mn) && a.fwd_after) {
#pragma unroll
          for (int c = 0; c < 3; ++c) X[(c * RB + rr) * f.ls + at<ODD>(xp)] = make_float2(mn[0][c], mn[1][c]);
        }
      }
    } else {
      for (int e = tid; e < RB * nx; e += T) {
        const int rr = fast_div(e, s.mnx), x = e - rr * nx;
        if (r0 + rr >= a.rows) continue;
        int z, y;
        row_zy(rr, z, y);
        const long long idx = (long long)(r0 + rr) * nx + x;
        const int fpos = 2 * at<ODD>(x >> 1) + (x & 1);
        float hd[3], mn[3];
        if (a.extrap) {
          extrap_cell(a, idx, hd);
        } else {
#pragma unroll
          for (int c = 0; c < 3; ++c) hd[c] = reinterpret_cast<const float*>(X + (c * RB + rr) * f.ls)[fpos] * a.hscale;
        }
        if (epilogue_cell(a, mode, z, y, x, idx, hd, mn) && a.fwd_after) {
#pragma unroll
          for (int c = 0; c < 3; ++c) reinterpret_cast<float*>(X + (c * RB + rr) * f.ls)[fpos] = mn[c];
        }
      }
    }
    if (!a.fwd_after) return;   // uniform over the grid
  } else {
    for (int e = tid; e < lines * nx; e += T) {
      const int line = fast_div(e, s.mnx), x = e - line * nx;
      const int rr = line & (RB - 1), c = line >> s.rb_log;
      float v = 0.f;
      if (r0 + rr < a.rows) v = a.in[c * N + (long long)(r0 + rr) * nx + x];
      reinterpret_cast<float*>(X + line * f.ls)[2 * at<ODD>(x >> 1) + (x & 1)] = v;
    }
  }
  // 4. zeros beyond the data: up to the middle of the line (open x; the first pass takes the upper
  //    half as zero), rows past the last one of the mesh
  if (const int pad_x = (xper ? 2 * L : L) - nx; pad_x > 0)
    for (int e = tid; e < lines * pad_x; e += T) {
      const int line = fast_div(e, s.mpad), x = nx + e - line * pad_x;
      reinterpret_cast<float*>(X + line * f.ls)[2 * at<ODD>(x >> 1) + (x & 1)] = 0.f;
    }
  if (r0 + RB > a.rows)
    for (int line = 0; line < lines; ++line)
      if (r0 + (line & (RB - 1)) >= a.rows)
        for (int x = tid; x < nx; x += T) reinterpret_cast<float*>(X + line * f.ls)[2 * at<ODD>(x >> 1) + (x & 1)] = 0.f;
  __syncthreads();
  // 5. forward FFT
  {
    const float2* src = X;
    float2* dst = Y;
    small_pass<-1, ODD>(f, 0, lines, stw,
                   [&](int l, int i) { return (xper || i < HALF) ? src[l * f.ls + at<ODD>(i)] : make_float2(0.f, 0.f); },
                   [&](int l, int i, float2 v) { dst[l * f.ls + at<ODD>(i)] = v; });
  }
  const float2* Z = small_passes<-1, ODD>(f, 1, f.np, lines, stw, Y, X);
  __syncthreads();
  // 6. Z -> X pairwise and store the half spectrum
  const int items = lines * (HALF + 1);
  for (int e = tid; e < items; e += T) {
    const int rr = e & (RB - 1), t2 = e >> s.rb_log;
    const int c = fast_div(t2, s.mhalf), k = t2 - c * (HALF + 1);
    if (r0 + rr >= a.rows) continue;
    const float2* Lz = Z + (c * RB + rr) * f.ls;
    const float2 wp = shw[k], wm = cconj(wp);
    float2 xk, xl;
    if (k == 0) {
      const float2 A = Lz[at<ODD>(0)];
      xk = make_float2(A.x + A.y, 0.f);
      xl = make_float2(A.x - A.y, 0.f);
    } else {
      const float2 A = Lz[at<ODD>(k)], B = Lz[at<ODD>(L - k)];
      xk = cscale(csub(cadd(A, cconj(B)), cmul_i<1>(cmul(wp, csub(A, cconj(B))))), 0.5f);
      xl = cscale(cadd(cadd(B, cconj(A)), cmul_i<1>(cmul(wm, csub(B, cconj(A))))), 0.5f);
    }
    int z, y;
    row_zy(rr, z, y);
    float2* base = a.S + (long long)(c * a.nz + z) * HX * ny + y;
    base[(long long)k * ny] = xk;
    if (k == 0 || L - k != k) base[(long long)(k == 0 ? L : L - k) * ny] = xl;
  }
}

// ---- convolution along y (and z) -------------------------------------------------------------

struct SmallConvArgs {
  ColArgs a;
  FftPlan f;
  float2* S;               // x spectrum [3][nz][Hx][ny]
  float2* T;               // y spectrum [3][nz][Hx][Py], used when the phases run as launches of their own
  int phases;              // 1 y FFT, 2 z FFT + product + z IFFT, 4 y IFFT; 7: all in one launch
};

// The z FFT of the zero-padded nz <= PZ / 2 values of three components, the kernel product and the
// inverse z FFT, in registers. With NZ = PZ / 2 and w = exp(-2 pi i / PZ), the even frequencies are
// DFT_NZ(x[n]) and the odd ones DFT_NZ(x[n] w^n); the inverse adds the two inverse DFT_NZ, the
// second times w^-n. Each half is complete under the product (kz and PZ - kz have one parity).
template <int PZ, class KF>
__device__ __forceinline__ void z_in_registers(float2 (&x)[3][PZ / 2], KF kfetch) {
  constexpr int NZ = PZ / 2;
  float2 u[3][NZ], r[3][NZ];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
#pragma unroll
      for (int n = 0; n < NZ; ++n) u[c][n] = (h == 0 || n == 0) ? x[c][n] : (4 * n == PZ) ? cmul_i<-1>(x[c][n]) : cmul(x[c][n], wr<-1, PZ>(n));
      dft<NZ, -1>(u[c]);
    }
#pragma unroll
    for (int m = 0; m < NZ; ++m) {
      const int kz = 2 * m + h;
      float K[6];
      kfetch(kz <= NZ ? kz : PZ - kz, K);
      const float sz = kz <= NZ ? 1.f : -1.f;
      const float kxz = sz * K[4], kyz = sz * K[5];
      const float2 a = u[0][m], b = u[1][m], c = u[2][m];
      u[0][m] = make_float2(K[0] * a.x + K[3] * b.x + kxz * c.x, K[0] * a.y + K[3] * b.y + kxz * c.y);
      u[1][m] = make_float2(K[3] * a.x + K[1] * b.x + kyz * c.x, K[3] * a.y + K[1] * b.y + kyz * c.y);
      u[2][m] = make_float2(kxz * a.x + kyz * b.x + K[2] * c.x, kxz * a.y + kyz * b.y + K[2] * c.y);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      dft<NZ, 1>(u[c]);
#pragma unroll
      for (int n = 0; n < NZ; ++n) {
        if (h == 0)
          r[c][n] = u[c][n];
        else
          x[c][n] = cadd(r[c][n], n == 0 ? u[c][0] : (4 * n == PZ) ? cmul_i<1>(u[c][n]) : cmul(u[c][n], wr<1, PZ>(n)));
      }
    }
  }
}

// The z transforms of 16 points take 128 registers or more: TWO runs them at two blocks of 256 threads
// per SM, otherwise at one of 384. ODD: Py is 3 * 2^k or 5 * 2^k.
__host__ __device__ constexpr int small_conv_threads(int PZ, bool two) { return PZ >= 16 && two ? 256 : 384; }
template <int PZ, bool ODD, bool TWO = true>
__global__ void __launch_bounds__(small_conv_threads(PZ, TWO), TWO ? 2 : 1) small_conv_kernel(const __grid_constant__ SmallConvArgs s, const float2* __restrict__ tw) {
  const ColArgs& a = s.a;
  const FftPlan& f = s.f;
  const int T = blockDim.x, tid = threadIdx.x;
  const int L = f.L, nz = a.nz, lines = 3 * nz, ny = a.ny, KY = L / 2 + 1;
  const int kx = blockIdx.x;
  extern __shared__ float2 sm[];
  float2* X = sm;
  float2* Y = X + lines * f.ls;
  float2* stw = Y + lines * f.ls;
  if (s.phases & 5) load_twiddles(f, stw, tw);
  // a film's kernel entry of the thread's first column towards L1, ahead of the wait (with layers, the
  // dozen entries per thread displace more than they save: 480x240x2 stage 33.6 -> 34.5 us)
  if (PZ == 1 && tid < L) prefetch_l1(a.Kf + (long long)kx * KY + (tid > L / 2 ? L - tid : tid));
  pdl_wait_then_release();
  __syncthreads();
  auto gS = [&](int l) { return s.S + ((long long)l * a.Hx + kx) * ny; };
  auto gT = [&](int l) { return s.T + ((long long)l * a.Hx + kx) * L; };
  auto from_T = [&]() {
    for (int l = 0; l < lines; ++l)
      for (int i = tid; i < L; i += T) X[l * f.ls + at<ODD>(i)] = gT(l)[i];
    __syncthreads();
  };
  auto to_T = [&]() {
    for (int l = 0; l < lines; ++l)
      for (int i = tid; i < L; i += T) gT(l)[i] = X[l * f.ls + at<ODD>(i)];
  };
  if (s.phases & 1) {
    float2* dst = X;
    small_pass<-1, ODD>(f, 0, lines, stw, [&](int l, int i) { return i < ny ? gS(l)[i] : make_float2(0.f, 0.f); },
                   [&](int l, int i, float2 v) { dst[l * f.ls + at<ODD>(i)] = v; });
    float2* R = small_passes<-1, ODD>(f, 1, f.np, lines, stw, X, Y);
    if (R != X) {
      Y = X;
      X = R;
    }
    __syncthreads();
    if (s.phases == 1) {
      to_T();
      return;
    }
  } else {
    from_T();
  }
  if (s.phases & 2) {
    for (int ky = tid; ky < L; ky += T) {
      const bool up = ky > L / 2;
      const int kyp = up ? L - ky : ky;
      const float sy = up ? -1.f : 1.f;
      float2* col = X + at<ODD>(ky);
      if constexpr (PZ == 1) {
        const float4 k4 = __ldg(a.Kf + (long long)kx * KY + kyp);
        const float kxy = sy * k4.w;
        const float2 m0 = col[0], m1 = col[f.ls], m2 = col[2 * f.ls];
        col[0] = make_float2(k4.x * m0.x + kxy * m1.x, k4.x * m0.y + kxy * m1.y);
        col[f.ls] = make_float2(kxy * m0.x + k4.y * m1.x, kxy * m0.y + k4.y * m1.y);
        col[2 * f.ls] = make_float2(k4.z * m2.x, k4.z * m2.y);
      } else {
        const int kpl = a.Hx * KY;   // entries per plane of the kernel
        const float2* kb = a.K3 + kx * KY + kyp;
        float2 x[3][PZ / 2];
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
          for (int z = 0; z < PZ / 2; ++z) x[c][z] = z < nz ? col[(c * nz + z) * f.ls] : make_float2(0.f, 0.f);
        z_in_registers<PZ>(x, [&](int kz, float (&K)[6]) {
          const float2* kp = kb + 3LL * kz * kpl;
          const float2 k01 = __ldg(kp), k23 = __ldg(kp + kpl), k45 = __ldg(kp + 2 * kpl);
          K[0] = k01.x;
          K[1] = k01.y;
          K[2] = k23.x;
          K[3] = sy * k23.y;
          K[4] = k45.x;
          K[5] = sy * k45.y;
        });
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
          for (int z = 0; z < PZ / 2; ++z)
            if (z < nz) col[(c * nz + z) * f.ls] = x[c][z];
      }
    }
    if (s.phases == 2) {
      __syncthreads();
      to_T();
      return;
    }
  }
  float2* R = small_passes<1, ODD>(f, 0, f.np - 1, lines, stw, X, Y);
  __syncthreads();
  const float2* src = R;
  small_pass<1, ODD>(f, f.np - 1, lines, stw, [&](int l, int i) { return src[l * f.ls + at<ODD>(i)]; },
                [&](int l, int i, float2 v) {
                  if (i < ny) gS(l)[i] = v;
                });
}

// ---- launchers -------------------------------------------------------------------------------

constexpr size_t kSmallSmem = 232448;   // dynamic shared memory of a block
constexpr int kSmallThreads = 384;

// Threads of a block: one per x-row item or y frequency while the blocks leave SMs to spare (96x64x1
// stage 10.4 -> 9.1 us), else one per eight values (4 % of the eight-mesh batch).
static int small_threads(int blocks, int items, int values, int most = kSmallThreads) {
  const int t = blocks <= 2 * kTileBlocks ? items : values / 8;
  return std::min(most, (t + 31) / 32 * 32);
}

static size_t small_row_smem(const FftPlan& f, int RB, int nx, int stage_rows) {
  return (size_t)((2 * 3 * RB * f.ls + f.ntw + f.L / 2 + 2) & ~1) * sizeof(float2) + (size_t)stage_rows * 3 * nx * 4 + 16;
}

// A staged RK stage: free x boundary, 16-byte aligned field rows, all rows of a block in one plane.
static bool small_stage_applies(const RowArgs& a, int RB) {
  auto al16 = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; };
  if (a.mode < ROW_RK1 || a.mode > ROW_RK4 || a.extrap || (a.per & 1) || a.nx % 4 != 0 || !a.vec8) return false;
  if (a.ny % RB != 0 || !al16(a.ms)) return false;
  return a.mode == ROW_RK1 || (al16(a.m0) && al16(a.acc));
}

// The x rows run here up to kSmallRowWork complex values per component (lengths 3 * 2^k, 5 * 2^k:
// kSmallRowMixed): beyond, the fewer instructions per value of row_kernel (row_pair_kernel) win over
// the shorter chain. RK stage of the whole mesh, us, row_kernel / this kernel: 64x64x1 13.7 / 10.9,
// 32x32x8 18.5 / 12.5, 128x128x1 14.5 / 11.8, 256x256x1 15.0 / 19.0; mixed lengths, row_pair_kernel /
// this kernel: 150x150x6 41.8 / 32.4, 600x333x1 demag 44.9 / 38.8, 320x320x4 62.4 / 72.3. From L = 768, where
// two rows fill half of an SM's shared memory, up to 200,000 values (row_kernel / this kernel: 700x320x1
// demag 33.9 / 38.5, 1200x200x1 30.3 / 32.6, 700x256x1 27.8 / 26.0).
// One row per block up to 64 rows or kSmallRowOne values, else two (a 16-byte piece of the spectrum):
// 128x128x1 11.8 / 12.5 us, 256x128x1 15.0 / 13.4, 200x150x1 18.9 / 14.3.
constexpr long long kSmallRowWork = 40960, kSmallRowMixed = 262144, kSmallRowMixed2 = 200000, kSmallRowOne = 20480;

bool small_row_ok(int Lx, int rows) {
  FftPlan f;
  const long long most = !mixed_len(Lx) ? kSmallRowWork : Lx >= 768 ? kSmallRowMixed2 : kSmallRowMixed;
  return Lx <= 1280 && rows < 65536 && (long long)rows * Lx <= most && make_fft_plan(Lx, f);
}

bool launch_small_row(int Lx, const RowArgs& a, const float2* tw, cudaStream_t st) {
  SmallRowArgs s;
  s.a = a;
  if (!make_fft_plan(Lx, s.f)) return false;
  s.rb_log = a.rows > 64 && (long long)a.rows * Lx > kSmallRowOne ? 1 : 0;
  const int RB = 1 << s.rb_log;
  s.mhalf = magic_div(Lx / 2 + 1);
  s.mnp2 = magic_div(a.nx / 2);
  s.mnx = magic_div(a.nx);
  s.mpad = magic_div(std::max(1, Lx - a.nx));
  s.mny = magic_div(a.ny);
  // stage the input rows where they fit, the others while that leaves room for two blocks per SM
  auto smem_of = [&](int staged) { return small_row_smem(s.f, RB, a.nx, small_stage_rows(RB, staged)); };
  s.staged = 0;
  if (small_stage_applies(a, RB) && smem_of(1) <= kSmallSmem) {
    s.staged = 1;
    // (not where the next stage's input replaces m0: the autotuner's repeated launch, without a
    // convolution in between, would read what the launch before writes)
    if (a.mode != ROW_RK1 && a.m0 != a.mnext && smem_of(s.staged | 4) <= kSmallSmem / 2) s.staged |= 4;
    if (a.nz > 1 && smem_of(s.staged | 2) <= kSmallSmem / 2) s.staged |= 2;
  }
  const size_t smem = smem_of(s.staged);
  const int blocks = (a.rows + RB - 1) >> s.rb_log;
  launch_pdl(mixed_len(Lx) ? small_row_kernel<true> : small_row_kernel<false>, (unsigned)blocks, (unsigned)small_threads(blocks, 3 * RB * (Lx / 2 + 1), 3 * RB * Lx), smem, st, s, tw);
  return true;
}

static size_t small_conv_smem(const FftPlan& f, int nz) { return (size_t)(2 * 3 * nz * f.ls + f.ntw) * sizeof(float2); }

// In one launch: 3D meshes of up to 8 layers whose lines of one kx fit a block's shared memory
// (demag against three launches, us: 32x64x4 21 -> 14.5, 480x240x2 42 -> 34, 320x320x4 70 -> 59), films up
// to kSmallFilm values (96x64x1 stage 13.5 -> 12.9; 200x150x1 17.1 -> 16.0; 256x256x1 equal). Only for
// lines below 1024 values: one block takes all lines of a kx, and with longer lines its passes and their
// barriers outlast the launches that it saves (100x512x1 demag 15.6 us by film_conv_kernel, 18.9 here;
// 512x400x2 47.8 in three launches, 58.6 here; 32x400x4 21.3, 31.0).
constexpr long long kSmallFilm = 300000;
bool small_conv_ok(int Hx, int Py, int Pz, int nz, int per) {
  FftPlan f;
  if (Py >= 1024 || !make_fft_plan(Py, f) || (per & 4) || nz > 8 || Pz == 2) return false;
  return (nz > 1 || 3LL * Hx * Py <= kSmallFilm) && small_conv_smem(f, nz) <= kSmallSmem;
}

bool launch_small_conv(const ColArgs& a, float2* S, float2* T, int phases, const float2* tw, cudaStream_t st) {
  SmallConvArgs s;
  s.a = a;
  s.S = S;
  s.T = T;
  s.phases = phases;
  if (!make_fft_plan(a.Py, s.f)) return false;
  const size_t smem = small_conv_smem(s.f, a.nz);
  // 5 to 8 layers: two blocks per SM where shared memory and the number of blocks allow (201x117x5 stage
  // 37.6 -> 33.9 us, 512x128x6 49.8 -> 44.6; 256x256x8, whose lines fill an SM, 49.4 -> 54.1, and
  // 128x128x8, with fewer blocks than SMs, 24.3 -> 27.2)
  const bool two = smem <= kSmallSmem / 2 && a.Hx > kTileBlocks;
  const int values = 3 * a.nz * a.Py;
  const unsigned threads = (unsigned)small_threads(a.Hx, std::max(a.Py, values / 8), values, small_conv_threads(a.Pz, two));
  auto go = [&](auto pz, auto two_per_sm) {
    constexpr int PZ = decltype(pz)::value;
    constexpr bool TWO = decltype(two_per_sm)::value;
    launch_pdl(mixed_len(a.Py) ? small_conv_kernel<PZ, true, TWO> : small_conv_kernel<PZ, false, TWO>, a.Hx, threads, smem, st, s, tw);
    return true;
  };
  switch (a.Pz) {
    case 1: return go(std::integral_constant<int, 1>(), std::true_type());
    case 4: return go(std::integral_constant<int, 4>(), std::true_type());
    case 8: return go(std::integral_constant<int, 8>(), std::true_type());
    case 16:
      return two ? go(std::integral_constant<int, 16>(), std::true_type()) : go(std::integral_constant<int, 16>(), std::false_type());
    default: return false;
  }
}

template <bool ODD>
static void prepare_small_t() {
  prep(small_row_kernel<ODD>, kSmallSmem);
  prep(small_conv_kernel<1, ODD>, kSmallSmem);
  prep(small_conv_kernel<4, ODD>, kSmallSmem);
  prep(small_conv_kernel<8, ODD>, kSmallSmem);
  prep(small_conv_kernel<16, ODD, true>, kSmallSmem);
  prep(small_conv_kernel<16, ODD, false>, kSmallSmem);
}
void prepare_small() {
  prepare_small_t<false>();
  prepare_small_t<true>();
}

}  // namespace gbd

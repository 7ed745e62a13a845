// Host launchers of the kernels in kernels.cuh: degree dispatch, grid sizing
// and the per-context tables.  Included once per value type (inst_f64.cu,
// inst_f32.cu).
#pragma once
#include <cmath>
#include <cstring>
#include <algorithm>
#include <new>
#include <type_traits>
#include <vector>

#include "ffsweep.cuh"
#include "kernels.cuh"
#include "mvs.cuh"
#include "mvs3.cuh"
#include "mvs_fx.cuh"
#include "sweep_fx.cuh"

namespace bh {

template <typename T, int K>
struct HostTables {
  Tables<T, K> t;
  MvsTab<T, K> mvs;  // operator + FDM tables for the fused MVS kernel
  CanonTab<T, K> canon;  // the interior tiles' part of mvs (batched FP32 kernel parameter)
  Tables<T, K>* dev = nullptr;  // device copy of t (batched kernels read it from memory)
  T* dinv = nullptr;  // device, 4^d slots x m^d reciprocals of the eigenvalue sums
  // FP32 tables only: the operator's class tables as hi + lo FP32 parts for the
  // compensated defect (ffsweep.cuh), host copy and device copy
  FfTab<K>* ff = nullptr;
  FfTab<K>* dev_ff = nullptr;
  // FP64 tables only: the fixed-point tables (fx.cuh), the interior ones on the
  // host (a kernel parameter), the others in device memory with D behind them
  FxCanon<K>* fx = nullptr;
  FxBand<K> band;
  FxFull<K>* dev_fx = nullptr;
  int2* dev_fxd = nullptr;
  int d = 0;
};

template <typename T, int K>
static void free_host_tables(HostTables<T, K>* h) {
  cudaFree(h->dinv);
  cudaFree(h->dev);
  cudaFree(h->dev_ff);
  cudaFree(h->dev_fx);
  delete h->ff;
  delete h->fx;
  delete h;
}

// limbs of L bits of an integer
static inline int2 fx_host(long long v, int L) {
  const long long hi = (v + (1ll << (L - 1))) >> L;
  return make_int2((int)hi, (int)(v - hi * (1ll << L)));
}

// a / b 2^f rounded to nearest, as limbs: the quotient as a sum of two doubles (long
// double is emulated in software on some hosts, and made this the larger part of a
// context's creation)
static inline int2 fx_host_quotient(double a, double b, int f, int L) {
  const double hi = a / b, lo = std::fma(-hi, b, a) / b;
  const double v = std::ldexp(hi, f), w = std::rint(v);
  return fx_host((long long)w + std::llrint((v - w) + std::ldexp(lo, f)), L);
}

// A row c 2^f (c times a power of two: exact in FP64) as band limbs whose sum is
// rounded too: entries are rounded to nearest, and then as many of those rounded
// furthest the other way as bring the sum within half a unit.  The sum's error is
// what a smooth vector sees.
static inline void fx_host_row(const double* c, int n, double factor, int f, int2* out) {
  double v[4 * kMaxK + 1], d[4 * kMaxK + 1], err = 0;
  int order[4 * kMaxK + 1];
  const double scale = std::ldexp(factor, f);
  for (int t = 0; t < n; ++t) {
    const double x = c[t] * scale;
    v[t] = std::rint(x);
    d[t] = x - v[t];
    err += d[t];
    order[t] = t;
  }
  const int miss = (int)std::lround(err), step = miss < 0 ? -1 : 1;
  if (miss) std::sort(order, order + n, [&](int x, int y) { return step * d[x] > step * d[y]; });
  for (int i = 0; i < std::abs(miss) && i < n && d[order[i]] != 0; ++i) v[order[i]] += step;
  for (int t = 0; t < n; ++t) out[t] = fx_host((long long)v[t], kFxBand);
}

// smallest e with v < 2^e, v a little enlarged: a coefficient's high limb has to
// stay below 2^31
static inline int fx_ceil_exp(double v) {
  int e;
  std::frexp(v * (1.0 + 1e-8), &e);
  return e;
}

// The scales of fx.cuh for a set of rows and patch types, and the fixed-point
// coefficients at them.  Row sums: at most 2^kFxCoef in the band tables.
struct FxScales {
  int fx[3];  // x-split scale per operator (M, L, B)
  int gy;     // y-combination, common to B on T_M, 2 L on T_L, M on T_B
  double wy[3];  // factor of operator o in the y-combination, relative to its 1D matrix
  double cf, cb;  // largest absolute sums of the forward and backward eigenvector lines
};

// exponent e_c of the forward lines' column scale 2^-e_c (about l_c^(-1/2)).  The
// eigenvalues are 20 and more with the default penalty; with a small one they may
// be negative or near zero.
static inline int fx_col_exp(double lam) {
  return (int)std::lround(0.5 * std::log2(std::max(std::fabs(lam), 1.0)));
}

template <int K>
static FxScales fx_scales(const OpTab<double, K>& op, const FdmTab<double, K>& fdm, int classes,
                          int types) {
  constexpr int BW = 4 * K + 1, M = 2 * K - 1;
  const double(*tab[3])[BW] = {op.M, op.L, op.B};
  FxScales s{};
  double sum[3][3 * K + 1];
  for (int o = 0; o < 3; ++o) {
    double top = 0.0;
    for (int c = 0; c < classes; ++c) {
      sum[o][c] = 0.0;
      for (int t = 0; t < BW; ++t) sum[o][c] += std::fabs(tab[o][c][t]);
      top = std::max(top, sum[o][c]);
    }
    s.fx[o] = kFxCoef - fx_ceil_exp(top);
  }
  // T_P = Y_P 2^(kFxCoef - fx[P]): the operator that acts on T_M is B, on T_L
  // 2 L, on T_B M
  s.wy[0] = std::ldexp(1.0, kFxCoef - s.fx[2]);
  s.wy[1] = std::ldexp(2.0, kFxCoef - s.fx[1]);
  s.wy[2] = std::ldexp(1.0, kFxCoef - s.fx[0]);
  double top = 0.0;
  for (int c = 0; c < classes; ++c)
    top = std::max(top, s.wy[0] * sum[0][c] + s.wy[1] * sum[1][c] + s.wy[2] * sum[2][c]);
  s.gy = kFxCoef - fx_ceil_exp(top);
  s.cf = s.cb = 0.0;
  for (int ty = 0; ty < types; ++ty)
    for (int i = 0; i < M; ++i) {
      double row = 0.0, col = 0.0;
      for (int j = 0; j < M; ++j) {
        row += std::fabs(fdm.S[ty][i][j]);
        col += std::fabs(fdm.S[ty][j][i]);
      }
      s.cb = std::max(s.cb, row);
      s.cf = std::max(s.cf, std::ldexp(col, -fx_col_exp(fdm.lam[ty][i])));
    }
  s.cf *= 1.0 + 1e-9;
  s.cb *= 1.0 + 1e-9;
  return s;
}

// The sweeps' tables (every row at its own scale) and, in 2D, those of the patch
// smoother, which is the fixed-point form only there.
template <int K>
static bool make_fx(HostTables<double, K>* h, const std::vector<double>& dinv, int md, int slots,
                    int d) {
  constexpr int BW = 4 * K + 1, M = 2 * K - 1, NC = 3 * K + 1;
  const OpTab<double, K>& op = h->t.op;
  const FdmTab<double, K>& fdm = h->t.fdm;
  const double(*tab[3])[BW] = {op.M, op.L, op.B};
  h->fx = new (std::nothrow) FxCanon<K>();
  // FxFull<K> and, behind it, the division of the patch smoother's combinations
  const size_t nD = d == 2 ? dinv.size() : 0, bytes = sizeof(FxFull<K>) + nD * sizeof(int2);
  std::vector<unsigned char> buf(bytes);
  if (!h->fx) return false;
  auto* full = new (buf.data()) FxFull<K>();
  int2* D = reinterpret_cast<int2*>(buf.data() + sizeof(FxFull<K>));
  int2* bx[3] = {h->band.M, h->band.L, h->band.B};
  float* ba[3] = {h->band.aM, h->band.aL, h->band.aB};
  for (int o = 0; o < 3; ++o)
    for (int c = 0; c < NC; ++c) {
      double sum = 0.0;
      for (int t = 0; t < BW; ++t) sum += std::fabs(tab[o][c][t]);
      const int f = kFxCoef - fx_ceil_exp(sum);
      full->f[o][c] = f;
      fx_host_row(tab[o][c], BW, 1.0, f, full->s[o][c]);
      if (c >= K) continue;
      h->band.f[o][c] = f;
      const double scale = std::ldexp(1.0, f - kFxCoef);
      for (int t = band_lo(o, c, K); t <= band_hi(o, c, K); ++t) {
        bx[o][FxIdx<K>::at(o, c, t)] = full->s[o][c][t + 2 * K];
        ba[o][FxIdx<K>::at(o, c, t)] = (float)(std::fabs(tab[o][c][t + 2 * K]) * scale);
      }
    }
  full->band = h->band;
  if (d == 2) {
    // interior: canonical rows 0..K-1, patch type 0
    FxScales s = fx_scales<K>(op, fdm, K, 1);
    int2* cx[3] = {h->fx->xM, h->fx->xL, h->fx->xB};
    int2* cy[3] = {h->fx->yM, h->fx->yL, h->fx->yB};
    for (int o = 0; o < 3; ++o)
      for (int q = 0; q < K; ++q) {
        const int lo = band_lo(o, q, K), n = band_hi(o, q, K) - lo + 1, at = FxIdx<K>::at(o, q, lo);
        fx_host_row(&tab[o][q][lo + 2 * K], n, 1.0, s.fx[o], cx[o] + at);
        fx_host_row(&tab[o][q][lo + 2 * K], n, s.wy[o], s.gy, cy[o] + at);
      }
    int ce[4][M];  // exponents of the forward lines' columns
    for (int ty = 0; ty < 4; ++ty)
      for (int c = 0; c < M; ++c) ce[ty][c] = fx_col_exp(fdm.lam[ty][c]);
    auto fwd = [&](int ty, int j, int c) {
      return fx_host_quotient(fdm.S[ty][j][c], s.cf, 2 * kFxLine - ce[ty][c], kFxLine);
    };
    auto bwd = [&](int ty, int j, int c) {
      return fx_host_quotient(fdm.S[ty][j][c], s.cb, 2 * kFxLine, kFxLine);
    };
    for (int j = 0; j < K; ++j)
      for (int c = 0; c < M; ++c) {
        h->fx->Sf[j][c] = fwd(0, j, c);
        h->fx->Sb[j][c] = bwd(0, j, c);
      }
    h->fx->eax = -s.gy;
    h->fx->corr = std::pow(s.cf * s.cb, d);
    full->canon = *h->fx;
    // every class and type
    s = fx_scales<K>(op, fdm, NC, 4);
    for (int o = 0; o < 3; ++o)
      for (int c = 0; c < NC; ++c) {
        fx_host_row(tab[o][c], BW, 1.0, s.fx[o], full->x[o][c]);
        fx_host_row(tab[o][c], BW, s.wy[o], s.gy, full->y[o][c]);
      }
    for (int ty = 0; ty < 4; ++ty)
      for (int j = 0; j < M; ++j)
        for (int c = 0; c < M; ++c) {
          full->Sf[ty][j][c] = fwd(ty, j, c);
          full->Sb[ty][j][c] = bwd(ty, j, c);
        }
    full->eax = -s.gy;
    full->corr = std::pow(s.cf * s.cb, d);
    double ds[M * M];  // the division, with the column scales taken back
    for (int slot = 0; slot < slots; ++slot) {
      const int *e0 = ce[slot % 4], *e1 = ce[slot / 4];
      double top = 0.0;
      for (int l = 0; l < md; ++l) {
        ds[l] = std::ldexp(dinv[(size_t)slot * md + l], e0[l % M] + e1[l / M]);
        top = std::max(top, std::fabs(ds[l]));
      }
      full->cD[slot] = top * (1.0 + 1e-9);
      for (int l = 0; l < md; ++l)
        D[(size_t)slot * md + l] = fx_host_quotient(ds[l], full->cD[slot], 2 * kFxLine, kFxLine);
    }
  }
  if (cudaMalloc(&h->dev_fx, bytes) != cudaSuccess ||
      cudaMemcpy(h->dev_fx, buf.data(), bytes, cudaMemcpyHostToDevice) != cudaSuccess)
    return false;
  h->dev_fxd = reinterpret_cast<int2*>(h->dev_fx + 1);
  return true;
}

template <typename T, int K>
static void* make_tables_k(const Setup1D& s, int d) {
  auto* h = new (std::nothrow) HostTables<T, K>();
  if (!h) return nullptr;
  const int nc = 3 * K + 1, bw = 4 * K + 1, m = 2 * K - 1;
  for (int c = 0; c < nc; ++c)
    for (int t = 0; t < bw; ++t) {
      h->t.op.M[c][t] = (T)s.tabM[c * bw + t];
      h->t.op.L[c][t] = (T)s.tabL[c * bw + t];
      h->t.op.B[c][t] = (T)s.tabB[c * bw + t];
    }
  for (int ty = 0; ty < 4; ++ty) {
    for (int i = 0; i < m; ++i) {
      for (int j = 0; j < m; ++j) h->t.fdm.S[ty][i][j] = (T)s.fdmS[ty][i * m + j];
      h->t.fdm.lam[ty][i] = (T)s.fdmLam[ty][i];
    }
  }
  for (int r = 0; r < 2 * K; ++r)
    for (int q = 0; q <= K; ++q) h->t.xfer.P[r][q] = (T)s.prolong[r * (K + 1) + q];
  h->mvs.op = h->t.op;
  h->mvs.fdm = h->t.fdm;
  for (int q = 0; q < K; ++q)
    for (int t = 0; t < bw; ++t) {
      h->canon.M[q][t] = h->t.op.M[q][t];
      h->canon.L[q][t] = h->t.op.L[q][t];
      h->canon.B[q][t] = h->t.op.B[q][t];
    }
  for (int i = 0; i < m; ++i)
    for (int j = 0; j < m; ++j) h->canon.S[0][i][j] = h->t.fdm.S[0][i][j];
  // reciprocal eigenvalue sums per type combination (FP64, then converted)
  int md = 1, slots = 1;
  for (int a = 0; a < d; ++a) {
    md *= m;
    slots *= 4;
  }
  std::vector<T> dinv((size_t)slots * md);
  for (int slot = 0; slot < slots; ++slot)
    for (int l = 0; l < md; ++l) {
      double sum = 0.0;
      int ll = l, ss = slot;
      for (int a = 0; a < d; ++a) {
        sum += s.fdmLam[ss % 4][ll % m];
        ll /= m;
        ss /= 4;
      }
      dinv[(size_t)slot * md + l] = (T)(1.0 / sum);
    }
  h->d = d;
  if constexpr (sizeof(T) == 4) {
    h->ff = new (std::nothrow) FfTab<K>();
    if (!h->ff) {
      delete h;
      return nullptr;
    }
    const double* src[3] = {s.tabM.data(), s.tabL.data(), s.tabB.data()};
    float(*hi[3])[4 * K + 1] = {h->ff->hi.M, h->ff->hi.L, h->ff->hi.B};
    float(*lo[3])[4 * K + 1] = {h->ff->lo.M, h->ff->lo.L, h->ff->lo.B};
    for (int o = 0; o < 3; ++o)
      for (int c = 0; c < nc; ++c)
        for (int t = 0; t < bw; ++t) {
          const double v = src[o][c * bw + t];
          const float vh = (float)v;
          hi[o][c][t] = vh;
          lo[o][c][t] = (float)(v - (double)vh);
        }
    if (cudaMalloc(&h->dev_ff, sizeof(FfTab<K>)) != cudaSuccess ||
        cudaMemcpy(h->dev_ff, h->ff, sizeof(FfTab<K>), cudaMemcpyHostToDevice) != cudaSuccess) {
      free_host_tables(h);
      return nullptr;
    }
  } else if (!make_fx<K>(h, dinv, md, slots, d)) {
    free_host_tables(h);
    return nullptr;
  }
  if (cudaMalloc(&h->dev, sizeof(Tables<T, K>)) != cudaSuccess ||
      cudaMemcpy(h->dev, &h->t, sizeof(Tables<T, K>), cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMalloc(&h->dinv, dinv.size() * sizeof(T)) != cudaSuccess ||
      cudaMemcpy(h->dinv, dinv.data(), dinv.size() * sizeof(T), cudaMemcpyHostToDevice) !=
          cudaSuccess) {
    free_host_tables(h);
    return nullptr;
  }
  return h;
}

#define BH_K_DISPATCH(k, CALL) \
  switch (k) {                 \
    case 2: CALL(2); break;    \
    case 3: CALL(3); break;    \
    case 4: CALL(4); break;    \
    case 5: CALL(5); break;    \
    case 6: CALL(6); break;    \
    case 7: CALL(7); break;    \
    default: return cudaErrorInvalidValue; \
  }

inline unsigned grid_for(int64_t threads, int block) {
  return (unsigned)((threads + block - 1) / block);
}

template <typename T>
void* Ops<T>::make_tables(const Setup1D& s, int d) {
  switch (s.k) {
    case 2: return make_tables_k<T, 2>(s, d);
    case 3: return make_tables_k<T, 3>(s, d);
    case 4: return make_tables_k<T, 4>(s, d);
    case 5: return make_tables_k<T, 5>(s, d);
    case 6: return make_tables_k<T, 6>(s, d);
    case 7: return make_tables_k<T, 7>(s, d);
  }
  return nullptr;
}

template <typename T, int K>
static void free_tables_k(void* p) {
  free_host_tables(static_cast<HostTables<T, K>*>(p));
}

template <typename T, int K>
static DevTables device_tables_k(const void* p) {
  const auto* h = static_cast<const HostTables<T, K>*>(p);
  return DevTables{h->dev, h->dinv, h->dev_fx, h->dev_fxd};
}

template <typename T>
DevTables Ops<T>::device_tables(const void* p, int k) {
  switch (k) {
    case 2: return device_tables_k<T, 2>(p);
    case 3: return device_tables_k<T, 3>(p);
    case 4: return device_tables_k<T, 4>(p);
    case 5: return device_tables_k<T, 5>(p);
    case 6: return device_tables_k<T, 6>(p);
    case 7: return device_tables_k<T, 7>(p);
  }
  return DevTables{nullptr, nullptr, nullptr, nullptr};
}

template <typename T, int K>
static const void* host_mvs_tables_k(const void* p, size_t* bytes) {
  const auto* h = static_cast<const HostTables<T, K>*>(p);
  if constexpr (sizeof(T) == 8) {
    *bytes = sizeof(FxCanon<K>);
    return h->fx;
  }
  *bytes = sizeof(CanonTab<T, K>);
  return &h->canon;
}

template <typename T>
const void* Ops<T>::host_mvs_tables(const void* p, int k, size_t* bytes) {
  switch (k) {
    case 2: return host_mvs_tables_k<T, 2>(p, bytes);
    case 3: return host_mvs_tables_k<T, 3>(p, bytes);
    case 4: return host_mvs_tables_k<T, 4>(p, bytes);
    case 5: return host_mvs_tables_k<T, 5>(p, bytes);
    case 6: return host_mvs_tables_k<T, 6>(p, bytes);
    case 7: return host_mvs_tables_k<T, 7>(p, bytes);
  }
  *bytes = 0;
  return nullptr;
}

template <typename T>
void Ops<T>::free_tables(void* p, int k) {
  if (!p) return;
  switch (k) {
    case 2: free_tables_k<T, 2>(p); break;
    case 3: free_tables_k<T, 3>(p); break;
    case 4: free_tables_k<T, 4>(p); break;
    case 5: free_tables_k<T, 5>(p); break;
    case 6: free_tables_k<T, 6>(p); break;
    case 7: free_tables_k<T, 7>(p); break;
  }
}

template <typename T, int K, int KIND>
static cudaError_t launch_sweep(const HostTables<T, K>& h, const SweepArgs<T>& a, cudaStream_t st) {
  const int block = 128;
  // FP64 on the integer pipe from one block per SM (152) on: apply of Q2 on 256^2 and
  // 32^3 cells 31.7 and 56.2 -> 27.7 and 51.6 us, Q3 on 16^3 41.7 -> 31.6, Q7 on 8^3
  // 124 -> 69.  Below, the FP64 form's little code is faster at Q2 (8^3 and 16^3 23.1
  // and 24.4 against 29.8 and 29.6), even at Q3 and Q4, and slower from Q5 on on uniform
  // values only (2D Q7 16^2 49.5 against 37.7): where rows are formed again, a launch of
  // few blocks waits for them (a step with the exact solver on smoothed data, Q7 on
  // 32^2, 1153 against 1250 to 1460, Q4 on 64^2 444 against 518).
  bool fx = false;
  if constexpr (sizeof(T) == 8) {
    fx = split_blocks(a.lines, a.N) >= 152;
    if (fx)
      fxs_sweep_kernel<K, KIND><<<(unsigned)split_blocks(a.lines, a.N), block, 0, st>>>(
          h.band, h.dev_fx, h.dev, a);
  }
  if (!fx)
    sweep_kernel<T, K, KIND><<<grid_for(sweep_launch_threads(KIND, a.lines, a.N), block), block, 0,
                               st>>>(h.t.op, a);
  g_kernel_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError();
}

template <typename T, int K>
static cudaError_t apply_k(const void* tabp, const LevelGeom& g, const T* x, const T* b, T* y,
                           double scale, int mode, T* scratch, cudaStream_t st) {
  const auto& tab = *static_cast<const HostTables<T, K>*>(tabp);
  SweepArgs<T> a{};
  a.d = g.d;
  a.N = g.N;
  a.n = g.n;
  a.lines = g.nd / g.n;
  a.scale = scale;
  a.mode = mode;
  a.b = b;
  T* s[6];
  for (int i = 0; i < 6; ++i) s[i] = scratch + (int64_t)i * g.nd;
  // pass x: split into M x, L x, B x
  a.axis = 0;
  a.stride = 1;
  a.in[0] = x;
  a.out[0] = s[0];
  a.out[1] = s[1];
  a.out[2] = s[2];
  cudaError_t e = launch_sweep<T, K, 0>(tab, a, st);
  if (e != cudaSuccess) return e;
  if (g.d == 2) {
    a.axis = 1;
    a.stride = g.n;
    a.in[0] = s[0];
    a.in[1] = s[1];
    a.in[2] = s[2];
    a.out[0] = y;
    return launch_sweep<T, K, 2>(tab, a, st);
  }
  a.axis = 1;
  a.stride = g.n;
  a.in[0] = s[0];
  a.in[1] = s[1];
  a.in[2] = s[2];
  a.out[0] = s[3];
  a.out[1] = s[4];
  a.out[2] = s[5];
  e = launch_sweep<T, K, 1>(tab, a, st);
  if (e != cudaSuccess) return e;
  a.axis = 2;
  a.stride = (int64_t)g.n * g.n;
  a.in[0] = s[3];
  a.in[1] = s[4];
  a.in[2] = s[5];
  a.out[0] = y;
  return launch_sweep<T, K, 3>(tab, a, st);
}

template <typename T>
cudaError_t Ops<T>::apply(const void* tab, const LevelGeom& g, const T* x, const T* b, T* y,
                          double scale, int mode, T* scratch, cudaStream_t st) {
#define BH_CALL(KK) return apply_k<T, KK>(tab, g, x, b, y, scale, mode, scratch, st)
  BH_K_DISPATCH(g.k, BH_CALL)
#undef BH_CALL
  return cudaErrorInvalidValue;
}

template <typename T, int D, int K>
static cudaError_t patch_fdm_k(const void* tabp, const LevelGeom& g, const T* r, T* x,
                               const int* verts, int count, double scale, bool atomic,
                               cudaStream_t st) {
  if (count <= 0) return cudaSuccess;
  const auto* h = static_cast<const HostTables<T, K>*>(tabp);
  PatchArgs<T> a{};
  a.r = r;
  a.x = x;
  a.verts = verts;
  a.count = count;
  a.N = g.N;
  a.n = g.n;
  a.scale = scale;
  a.dinv = h->dinv;
  constexpr int PB = PatchCfg<T, D, K>::PB;
  const unsigned grid = (unsigned)((count + PB - 1) / PB);
  if (atomic)
    patch_fdm_kernel<T, D, K, true><<<grid, 256, 0, st>>>(h->t.fdm, a);
  else
    patch_fdm_kernel<T, D, K, false><<<grid, 256, 0, st>>>(h->t.fdm, a);
  g_kernel_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError();
}

template <typename T>
cudaError_t Ops<T>::patch_fdm(const void* tab, const LevelGeom& g, const T* r, T* x,
                              const int* verts, int count, double scale, bool atomic,
                              cudaStream_t st) {
  if (g.d == 2) {
#define BH_CALL(KK) return patch_fdm_k<T, 2, KK>(tab, g, r, x, verts, count, scale, atomic, st)
    BH_K_DISPATCH(g.k, BH_CALL)
#undef BH_CALL
  } else {
#define BH_CALL(KK) return patch_fdm_k<T, 3, KK>(tab, g, r, x, verts, count, scale, atomic, st)
    BH_K_DISPATCH(g.k, BH_CALL)
#undef BH_CALL
  }
  return cudaErrorInvalidValue;
}

// Patches per block of the fused MVS kernels at which one smoothing step (FP64)
// or one V-cycle (FP32) at the paper's sizes (2D: 512^2 cells for k <= 4, 256^2
// above; 3D: 128^3 for k <= 3, 64^3 above) ran fastest on GB300; the automatic
// choice is min(ceil(count / (2 * 152)), this, the shared-memory limit), so
// levels with few patches still spread over the SMs (0: no cap).  In FP32 the
// 3D kernel's shared memory, not its FMAs, sets the pace: smaller tiles leave
// room for more blocks per SM.
constexpr int kMvs3TileF64[8] = {0, 0, 12, 16, 16, 16, 16, 16};
constexpr int kMvs2TileF32[8] = {0, 0, 0, 0, 0, 0, 0, 0};
constexpr int kMvs3TileF32[8] = {0, 0, 12, 8, 4, 3, 0, 0};

template <typename T>
inline int auto_tile(int count, int pref_f64, int pref_f32) {
  int pb = (count + 2 * 152 - 1) / (2 * 152);
  const int pref = sizeof(T) == 8 ? pref_f64 : pref_f32;
  if (pref > 0 && pb > pref) pb = pref;
  return pb;
}

template <typename T, int K>
static cudaError_t mvs_color_k(const void* tabp, const LevelGeom& g, T* x, const T* b,
                               const int* verts, int count, double ascale, double pscale,
                               int pb_req, cudaStream_t st) {
  if (count <= 0) return cudaSuccess;
  const auto* h = static_cast<const HostTables<T, K>*>(tabp);
  MvsArgs<T> a{};
  a.x = x;
  a.b = b;
  a.verts = verts;
  a.count = count;
  a.N = g.N;
  a.n = g.n;
  a.ascale = ascale;
  a.pscale = pscale;
  a.dinv = h->dinv;
  a.dtab = h->dev;
  a.fx = h->dev_fx;
  a.fx_dinv = h->dev_fxd;
  // FP64 on the integer pipe (mvs_fx.cuh), FP32 on its own
  using C = std::conditional_t<sizeof(T) == 8, Fx2Cfg<K>, Mvs2Cfg<T, K>>;
  // patches per block: enough blocks for two waves on 152 SMs, at most PB_MAX
  int pb = pb_req > 0 ? pb_req : auto_tile<T>(count, kFx2Tile[K], kMvs2TileF32[K]);
  pb = pb < 1 ? 1 : (pb > C::PB_MAX ? C::PB_MAX : pb);
  a.pb = pb;
  const unsigned grid = (unsigned)((count + pb - 1) / pb);
  // opt in to the dynamic shared memory once per instantiation (thread-safe static init)
  if constexpr (sizeof(T) == 8) {
    if (count <= kFx2SmallCount && pb_req <= 0) {
      static const cudaError_t attr = cudaFuncSetAttribute(
          mvs2_fx_small_kernel<K>, cudaFuncAttributeMaxDynamicSharedMemorySize,
          (int)C::smem_bytes(1));
      if (attr != cudaSuccess) return attr;
      a.pb = 1;
      mvs2_fx_small_kernel<K><<<(unsigned)count, 256, C::smem_bytes(1), st>>>(a);
    } else {
      static const cudaError_t attr =
          cudaFuncSetAttribute(mvs2_fx_kernel<K>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)C::smem_bytes(C::PB_MAX));
      if (attr != cudaSuccess) return attr;
      mvs2_fx_kernel<K><<<grid, C::THREADS, C::smem_bytes(pb), st>>>(*h->fx, a);
    }
  } else {
    static const cudaError_t attr = cudaFuncSetAttribute(
        mvs2_color_kernel<T, K>, cudaFuncAttributeMaxDynamicSharedMemorySize,
        (int)C::smem_bytes(C::PB_MAX));
    if (attr != cudaSuccess) return attr;
    mvs2_color_kernel<T, K><<<grid, 256, C::smem_bytes(pb), st>>>(h->mvs, a);
  }
  g_kernel_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError();
}

template <typename T, int K>
static cudaError_t mvs3_color_k(const void* tabp, const LevelGeom& g, T* x, const T* b,
                                const int* verts, int count, double ascale, double pscale,
                                int pb_req, cudaStream_t st) {
  if (count <= 0) return cudaSuccess;
  const auto* h = static_cast<const HostTables<T, K>*>(tabp);
  MvsArgs<T> a{};
  a.x = x;
  a.b = b;
  a.verts = verts;
  a.count = count;
  a.N = g.N;
  a.n = g.n;
  a.ascale = ascale;
  a.pscale = pscale;
  a.dinv = h->dinv;
  a.dtab = h->dev;
  using C = Mvs3Cfg<T, K>;
  int pb = pb_req > 0 ? pb_req : auto_tile<T>(count, kMvs3TileF64[K], kMvs3TileF32[K]);
  pb = pb < 1 ? 1 : (pb > C::PB_MAX ? C::PB_MAX : pb);
  a.pb = pb;
  static const cudaError_t attr = cudaFuncSetAttribute(
      mvs3_color_kernel<T, K>, cudaFuncAttributeMaxDynamicSharedMemorySize,
      (int)C::smem_bytes(C::PB_MAX));
  if (attr != cudaSuccess) return attr;
  mvs3_color_kernel<T, K><<<(unsigned)((count + pb - 1) / pb), C::THREADS, C::smem_bytes(pb), st>>>(
      h->mvs, a);
  g_kernel_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError();
}

template <typename T>
cudaError_t Ops<T>::mvs_color(const void* tab, const LevelGeom& g, T* x, const T* b,
                              const int* verts, int count, double ascale, double pscale, int pb,
                              cudaStream_t st) {
  if (g.d == 2) {
#define BH_CALL(KK) return mvs_color_k<T, KK>(tab, g, x, b, verts, count, ascale, pscale, pb, st)
    BH_K_DISPATCH(g.k, BH_CALL)
#undef BH_CALL
  } else {
#define BH_CALL(KK) \
  return mvs3_color_k<T, KK>(tab, g, x, b, verts, count, ascale, pscale, pb, st)
    BH_K_DISPATCH(g.k, BH_CALL)
#undef BH_CALL
  }
  return cudaErrorInvalidValue;
}

template <typename T, int D, int K>
static cudaError_t patch_exact_k(const LevelGeom& g, const T* ainv, const T* r, T* x,
                                 const int* verts, int count, double scale, bool atomic,
                                 cudaStream_t st) {
  if (count <= 0) return cudaSuccess;
  PatchArgs<T> a{};
  a.r = r;
  a.x = x;
  a.verts = verts;
  a.count = count;
  a.N = g.N;
  a.n = g.n;
  a.scale = scale;
  a.ainv = ainv;
  constexpr int PB = PatchCfg<T, D, K>::PB;
  const unsigned grid = (unsigned)((count + PB - 1) / PB);
  if (atomic)
    patch_exact_kernel<T, D, K, true><<<grid, 256, 0, st>>>(a);
  else
    patch_exact_kernel<T, D, K, false><<<grid, 256, 0, st>>>(a);
  g_kernel_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError();
}

template <typename T>
cudaError_t Ops<T>::patch_exact(const LevelGeom& g, const T* Ainv, const T* r, T* x,
                                const int* verts, int count, double scale, bool atomic,
                                cudaStream_t st) {
  if (g.d == 2) {
#define BH_CALL(KK) return patch_exact_k<T, 2, KK>(g, Ainv, r, x, verts, count, scale, atomic, st)
    BH_K_DISPATCH(g.k, BH_CALL)
#undef BH_CALL
  } else {
#define BH_CALL(KK) return patch_exact_k<T, 3, KK>(g, Ainv, r, x, verts, count, scale, atomic, st)
    BH_K_DISPATCH(g.k, BH_CALL)
#undef BH_CALL
  }
  return cudaErrorInvalidValue;
}

template <typename T, int D, int K>
static cudaError_t patch_gather_k(const LevelGeom& g, const T* r, const int* verts, int count,
                                  T* R, cudaStream_t st) {
  if (count <= 0) return cudaSuccess;
  const int64_t tot = (int64_t)count * PatchCfg<T, D, K>::MD;
  patch_gather_kernel<T, D, K><<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(r, verts, count,
                                                                            g.N, g.n, R);
  g_kernel_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError();
}

template <typename T, int D, int K>
static cudaError_t patch_scatter_k(const LevelGeom& g, const T* Y, const int* verts, int count,
                                   T* x, bool atomic, cudaStream_t st) {
  if (count <= 0) return cudaSuccess;
  const int64_t tot = (int64_t)count * PatchCfg<T, D, K>::MD;
  const unsigned grid = (unsigned)((tot + 255) / 256);
  if (atomic)
    patch_scatter_kernel<T, D, K, true><<<grid, 256, 0, st>>>(Y, verts, count, g.N, g.n, x);
  else
    patch_scatter_kernel<T, D, K, false><<<grid, 256, 0, st>>>(Y, verts, count, g.N, g.n, x);
  g_kernel_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError();
}

template <typename T>
cudaError_t Ops<T>::patch_gather(const LevelGeom& g, const T* r, const int* verts, int count,
                                 T* R, cudaStream_t st) {
  if (g.d == 2) {
#define BH_CALL(KK) return patch_gather_k<T, 2, KK>(g, r, verts, count, R, st)
    BH_K_DISPATCH(g.k, BH_CALL)
#undef BH_CALL
  } else {
#define BH_CALL(KK) return patch_gather_k<T, 3, KK>(g, r, verts, count, R, st)
    BH_K_DISPATCH(g.k, BH_CALL)
#undef BH_CALL
  }
  return cudaErrorInvalidValue;
}

template <typename T>
cudaError_t Ops<T>::patch_scatter(const LevelGeom& g, const T* Y, const int* verts, int count,
                                  T* x, bool atomic, cudaStream_t st) {
  if (g.d == 2) {
#define BH_CALL(KK) return patch_scatter_k<T, 2, KK>(g, Y, verts, count, x, atomic, st)
    BH_K_DISPATCH(g.k, BH_CALL)
#undef BH_CALL
  } else {
#define BH_CALL(KK) return patch_scatter_k<T, 3, KK>(g, Y, verts, count, x, atomic, st)
    BH_K_DISPATCH(g.k, BH_CALL)
#undef BH_CALL
  }
  return cudaErrorInvalidValue;
}

// one transfer pass along `axis`; shapes per axis given for input and output
template <typename T, int K, bool PROLONG>
static cudaError_t xfer_pass(const XferTab<T, K>& tab, int d, int axis, const int* din,
                             const int* dout, int Nc, int nc, int nf, const T* in, T* out,
                             bool add, cudaStream_t st, float* out32 = nullptr) {
  XferArgs<T> a{};
  a.in = in;
  a.out = out;
  a.out32 = out32;
  a.d = d;
  a.axis = axis;
  a.Nc = Nc;
  a.nc = nc;
  a.nf = nf;
  a.add = add;
  int64_t si = 1, so = 1, lines = 1;
  for (int i = 0; i < 3; ++i) {
    a.dims_in[i] = i < d ? din[i] : 1;
    a.dims_out[i] = i < d ? dout[i] : 1;
    a.str_in[i] = si;
    a.str_out[i] = so;
    si *= a.dims_in[i];
    so *= a.dims_out[i];
    if (i < d && i != axis) lines *= din[i];
  }
  a.lines = lines;
  const int block = 128;
  if (PROLONG)
    prolong_kernel<T, K><<<grid_for(lines * Nc, block), block, 0, st>>>(tab, a);
  else
    restrict_kernel<T, K><<<grid_for(lines * Nc, block), block, 0, st>>>(tab, a);
  g_kernel_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError();
}

template <typename T, int K, bool PROLONG>
static cudaError_t transfer_k(const void* tabp, const LevelGeom& fine, const T* in, T* out,
                              T* s0, T* s1, cudaStream_t st, float* out32 = nullptr) {
  const auto& tab = static_cast<const HostTables<T, K>*>(tabp)->t.xfer;
  const int d = fine.d, Nc = fine.N / 2, nc = K * Nc - 1, nf = fine.n;
  int dims[3];
  for (int i = 0; i < 3; ++i) dims[i] = PROLONG ? nc : nf;
  const T* src = in;
  T* bufs[2] = {s0, s1};
  for (int axis = 0; axis < d; ++axis) {
    int dn[3] = {dims[0], dims[1], dims[2]};
    dn[axis] = PROLONG ? nf : nc;
    const bool last = axis == d - 1;
    T* dst = last ? out : bufs[axis % 2];
    cudaError_t e =
        xfer_pass<T, K, PROLONG>(tab, d, axis, dims, dn, Nc, nc, nf, src, dst, PROLONG && last, st,
                                 last ? out32 : nullptr);
    if (e != cudaSuccess) return e;
    for (int i = 0; i < 3; ++i) dims[i] = dn[i];
    src = dst;
  }
  return cudaSuccess;
}

template <typename T>
cudaError_t Ops<T>::prolongate_add(const void* tab, const LevelGeom& fine, const T* xc, T* xf,
                                   T* s0, T* s1, cudaStream_t st) {
#define BH_CALL(KK) return transfer_k<T, KK, true>(tab, fine, xc, xf, s0, s1, st)
  BH_K_DISPATCH(fine.k, BH_CALL)
#undef BH_CALL
  return cudaErrorInvalidValue;
}

template <typename T>
cudaError_t Ops<T>::restrict_(const void* tab, const LevelGeom& fine, const T* rf, T* bc, T* s0,
                              T* s1, cudaStream_t st, float* bc32) {
#define BH_CALL(KK) return transfer_k<T, KK, false>(tab, fine, rf, bc, s0, s1, st, bc32)
  BH_K_DISPATCH(fine.k, BH_CALL)
#undef BH_CALL
  return cudaErrorInvalidValue;
}

template <typename T>
cudaError_t Ops<T>::add(T* y, const T* x, int64_t n, cudaStream_t st) {
  int64_t g = (n + 255) / 256;
  if (g > 152 * 32) g = 152 * 32;
  add_kernel<T><<<(unsigned)(g < 1 ? 1 : g), 256, 0, st>>>(y, x, n);
  g_kernel_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError();
}

template <typename T>
cudaError_t Ops<T>::dense_symv(int n, const double* A, const T* in, T* out, double scale,
                               cudaStream_t st) {
  dense_symv_kernel<T><<<grid_for(n, 128), 128, 0, st>>>(n, A, in, out, scale);
  g_kernel_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError();
}

}  // namespace bh

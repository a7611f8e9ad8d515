// The subdomain operators of the fast-diagonalization (FDM) local solver, one CTA per subdomain:
//   SCHUR     y_i = (K_GG - K_GI K_II^{-1} K_IG) x_i            (eq. 6)
//   CONDENSE  y_i = -K_GI K_II^{-1} f_I                          (Sect. 3.1)
//   RECOVER   x_I = K_II^{-1} (f_I - K_IG x_G), x_G copied       (Sect. 3.1)
// and the same for a block of ensemble members. Single Schur applications in df64 on 8^3 subdomains
// keep their own kernel (k_schur_fused), which forms the brick entries on chip: these rows stream 77 KB
// of coefficients per subdomain, which a block of members shares and a single vector does not.
//
// K_IG, K_GI and K_GG are applied as assembled rows of the local stiffness matrix ("local rows"),
// formed once at setup in FP64. The matrix-free form summed over the up to eight bricks of a node:
// 18.6k multiply-adds per 8^3 subdomain in the two passes, of which more than half met a zero
// interior value or a brick entry that another brick of the same node pair could have been added to;
// the assembled rows take 8.8k. K_II^{-1} = V D^{-1} V^T, V = Vz (x) Vy (x) Vx, is six contractions along
// lines: a thread holds a line's values in registers and forms several outputs from broadcast
// quads of V, so the shared-memory traffic per multiply-add falls from two loads to less than
// one (the per-output form ran at 25 % of the df64 ALU rate, bound by shared memory).
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <map>
#include <vector>

#include "batch.h"
#include "device.h"
#include "local.h"
#include "policy.cuh"

namespace dd {

// ---------------------------------------------------------------------------
// setup
// ---------------------------------------------------------------------------
LocalRowsHost build_local_rows(const Mesh1& M, const Level& L, bool boundary_only) {
  LocalRowsHost R;
  const int S = M.S, NLx = M.NLx, NLy = M.NLy, NLz = M.NLz;
  struct Entry {
    int16_t a, b;  // local nodes of the row and of the neighbour
  };
  std::vector<std::vector<Entry>> ell;  // per type: (row node, neighbour node) in storage order, a < 0: padding
  std::map<std::vector<int8_t>, int> types;
  std::vector<int8_t> pat(M.NL);
  R.type.resize(S);
  for (int s = 0; s < S; ++s) {
    const int16_t* code = M.lidx.data() + (size_t)s * M.NL;
    for (int l = 0; l < M.NL; ++l) pat[l] = code[l] >= 0 ? 1 : (code[l] == INT16_MIN ? 0 : 2);
    auto it = types.find(pat);
    if (it != types.end()) {
      R.type[s] = it->second;
      continue;
    }
    const int t = (int)types.size();
    types.emplace(pat, t);
    R.type[s] = t;
    const int nG = (int)(L.goff[s + 1] - L.goff[s]);
    // interior unknowns next to the interface, and their rank among these
    std::vector<int> rank(M.NL, -1);
    R.bnd.emplace_back();
    for (int l = 0; l < M.NL; ++l) {
      if (pat[l] != 1) continue;
      const int a = l % NLx, b = (l / NLx) % NLy, c = l / (NLx * NLy);
      bool next = false;
      for (int z = std::max(c - 1, 0); z <= std::min(c + 1, NLz - 1); ++z)
        for (int y = std::max(b - 1, 0); y <= std::min(b + 1, NLy - 1); ++y)
          for (int x = std::max(a - 1, 0); x <= std::min(a + 1, NLx - 1); ++x)
            next = next || pat[x + NLx * (y + NLy * z)] == 2;
      if (!next) continue;
      rank[l] = (int)R.bnd[t].size();
      R.bnd[t].push_back(code[l]);
    }
    auto compact = [&](int l) {
      if (code[l] < 0) return -1 - code[l];
      return nG + (boundary_only ? rank[l] : code[l]);
    };
    ell.emplace_back();
    const int nb_base = (int)R.nb.size();
    int range[4];
    for (int pass = 0; pass < 2; ++pass) {
      std::vector<std::pair<int, std::vector<int>>> rows;  // row node, neighbours
      for (int l = 0; l < M.NL; ++l) {
        if (pat[l] != (pass == 0 ? 1 : 2)) continue;
        const int a = l % NLx, b = (l / NLx) % NLy, c = l / (NLx * NLy);
        // corner neighbours first, the node itself last: its product, the largest, is not carried through
        // the roundings of the others. Interface rows of a uniform 4^3 subdomain in df64, 2-norm: 4.1e-15
        // in lexicographic order, 3.3e-15 in this one, 2.8e-15 with the chains renormalized before
        // they are added (apply_rows); brick by brick 2.8e-15.
        std::vector<int> nbs;
        for (int far = 3; far >= 0; --far)
          for (int dz = -1; dz <= 1; ++dz)
            for (int dy = -1; dy <= 1; ++dy)
              for (int dx = -1; dx <= 1; ++dx) {
                if ((dx != 0) + (dy != 0) + (dz != 0) != far) continue;
                const int x = a + dx, y = b + dy, z = c + dz;
                if (x < 0 || y < 0 || z < 0 || x >= NLx || y >= NLy || z >= NLz) continue;
                const int q = x + NLx * (y + NLy * z);
                if (pat[q] == 2 || (pass == 1 && pat[q] == 1)) nbs.push_back(q);
              }
        if (!nbs.empty()) rows.emplace_back(l, std::move(nbs));
      }
      // rows of similar length share a slice of 32
      std::stable_sort(rows.begin(), rows.end(), [](const auto& x, const auto& y) { return x.second.size() > y.second.size(); });
      range[2 * pass] = (int)R.sl_w.size();
      for (size_t i0 = 0; i0 < rows.size(); i0 += 32) {
        const int w = (int)rows[i0].second.size();
        R.sl_w.push_back(w);
        R.sl_off.push_back((int)ell[t].size());
        for (int u = 0; u < 32; ++u) {
          const bool in = i0 + u < rows.size();
          R.sl_out.push_back(in ? (int16_t)compact(rows[i0 + u].first) : (int16_t)-1);
          R.sl_cnt.push_back(in ? (int16_t)rows[i0 + u].second.size() : (int16_t)0);
        }
        for (int q = 0; q < w; ++q)
          for (int u = 0; u < 32; ++u) {
            const bool in = i0 + u < rows.size() && q < (int)rows[i0 + u].second.size();
            ell[t].push_back(in ? Entry{(int16_t)rows[i0 + u].first, (int16_t)rows[i0 + u].second[q]} : Entry{-1, -1});
            R.nb.push_back(in ? (int16_t)compact(rows[i0 + u].second[q]) : (int16_t)0);
          }
      }
      range[2 * pass + 1] = (int)R.sl_w.size();
    }
    R.trange.insert(R.trange.end(), range, range + 4);
    R.trange.push_back(nb_base);
  }
  R.coff.resize(S + 1);
  R.coff[0] = 0;
  for (int s = 0; s < S; ++s) R.coff[s + 1] = R.coff[s] + (int64_t)ell[R.type[s]].size();
  R.coef.assign((size_t)R.coff[S], 0.0);
#pragma omp parallel for schedule(static)
  for (int s = 0; s < S; ++s) {
    const std::vector<Entry>& E = ell[R.type[s]];
    const int I = s % M.Sx, J = (s / M.Sx) % M.Sy, K = s / (M.Sx * M.Sy);
    double* dst = R.coef.data() + R.coff[s];
    for (size_t t = 0; t < E.size(); ++t) {
      if (E[t].a < 0) continue;
      int p[3], d[3], lo[3], hi[3], sgn = 0;
      const int dim[3] = {M.sx, M.sy, M.sz};
      const int ia[3] = {E[t].a % NLx, (E[t].a / NLx) % NLy, E[t].a / (NLx * NLy)};
      const int ib[3] = {E[t].b % NLx, (E[t].b / NLx) % NLy, E[t].b / (NLx * NLy)};
      for (int a = 0; a < 3; ++a) {
        p[a] = ia[a];
        d[a] = ib[a] - ia[a];
        lo[a] = d[a] > 0 ? p[a] : p[a] - 1;  // elements that hold both nodes along this axis
        hi[a] = d[a] < 0 ? p[a] - 1 : p[a];
        lo[a] = std::max(lo[a], 0);
        hi[a] = std::min(hi[a], dim[a] - 1);
        if (d[a]) sgn |= 1 << a;
      }
      const double sx = (sgn & 1) ? -1.0 : 1.0, mx = (sgn & 1) ? 1.0 : 2.0;
      const double sy = (sgn & 2) ? -1.0 : 1.0, my = (sgn & 2) ? 1.0 : 2.0;
      const double sz = (sgn & 4) ? -1.0 : 1.0, mz = (sgn & 4) ? 1.0 : 2.0;
      double v = 0.0;
      for (int ec = lo[2]; ec <= hi[2]; ++ec)
        for (int eb = lo[1]; eb <= hi[1]; ++eb)
          for (int ea = lo[0]; ea <= hi[0]; ++ea) {
            const size_t e = (size_t)(I * M.sx + ea) + (size_t)M.nx * ((J * M.sy + eb) + (size_t)M.ny * (K * M.sz + ec));
            v += M.ecx[e] * (sx * my * mz) + M.ecy[e] * (mx * sy * mz) + M.ecz[e] * (mx * my * sz);
          }
      dst[t] = v;
    }
  }
  return R;
}

// ---------------------------------------------------------------------------
// device pieces
// ---------------------------------------------------------------------------
constexpr int VST = 10;           // stride of the staged 1-D bases (16-byte rows)
constexpr int VMAT = 9 * VST;     // one staged basis
template <class V>
struct alignas(16) Two {
  V a, b;
};

// Vs[2 a] = V_a by rows (out_j = sum_i V(i, j) x_i reads row i), Vs[2 a + 1] = V_a^T
template <class P>
__device__ __forceinline__ void stage_bases(const DevMesh& m, int s, typename P::V* Vs) {
  for (int t = threadIdx.x; t < 243; t += blockDim.x) {
    const typename P::V v = ld_fdm<P>(m.fdm_V, (int64_t)s * 243 + t);
    const int a = t / 81, i = (t % 81) / 9, j = t % 9;
    Vs[2 * a * VMAT + i * VST + j] = v;
    Vs[(2 * a + 1) * VMAT + j * VST + i] = v;
  }
  // the tenth column pads the rows to 16 bytes
  for (int t = threadIdx.x; t < 54; t += blockDim.x) Vs[(t / 9) * VMAT + (t % 9) * VST + 9] = P::zero();
}

// out[j] = sum_i A(i, j0 + j) x_i, j < NJ (j0 even), over na <= NI values of a line; two chains per
// output (even and odd i). FULL: the chains are renormalized before they are added (six df64
// contractions of 7^3 values 8.7e-15 -> 7.7e-15 from the exact ones). Ensembles do without: their kernels
// before had one chain per output, 9.7e-15.
template <class P, int NI, int NJ, bool FULL>
__device__ __forceinline__ void line_products(const typename P::V* A, int na, int j0, const typename P::V* x,
                                              typename P::V* out) {
  using V = typename P::V;
  typename P::Acc acc[2][NJ];
#pragma unroll
  for (int j = 0; j < NJ; ++j) {
    P::init(acc[0][j]);
    P::init(acc[1][j]);
  }
#pragma unroll
  for (int i = 0; i < NI; ++i) {
    if (i < na) {
#pragma unroll
      for (int j = 0; j + 1 < NJ; j += 2) {
        const Two<V> a = *reinterpret_cast<const Two<V>*>(A + i * VST + j0 + j);
        P::fma(acc[i & 1][j], a.a, x[i]);
        P::fma(acc[i & 1][j + 1], a.b, x[i]);
      }
      if (NJ & 1) P::fma(acc[i & 1][NJ - 1], A[i * VST + j0 + NJ - 1], x[i]);
    }
  }
#pragma unroll
  for (int j = 0; j < NJ; ++j) {
    if (FULL) {
      out[j] = P::add(P::get(acc[0][j]), P::get(acc[1][j]));
    } else {
      P::merge(acc[0][j], acc[1][j]);
      out[j] = P::get(acc[0][j]);
    }
  }
}

__device__ __forceinline__ void line_geom(int ax, const int* n, int l, int& base, int& stride) {
  if (ax == 0) {
    base = n[0] * l;
    stride = 1;
  } else if (ax == 1) {
    base = l % n[0] + n[0] * n[1] * (l / n[0]);
    stride = n[0];
  } else {
    base = l;
    stride = n[0] * n[1];
  }
}

// one contraction of a single vector, from `in` to `out`; a line's outputs are shared by two
// threads (0-3 and the rest) of different warps: threads 0-63 and 64-127, one of the 49 lines each.
// EPI 0: store; 1: times D^{-1}; 2: negate; 3: hand to `fin(index, value)`
template <class P, int NI, int NJ, int EPI, class Fin>
__device__ __forceinline__ void line_out(const typename P::V* A, int na, int j0, const typename P::V* x, int base,
                                         int stride, typename P::V* out, const void* dinv, int64_t io, Fin fin) {
  using V = typename P::V;
  V o[NJ], dv[NJ];
  if (EPI == 1) {
#pragma unroll
    for (int j = 0; j < NJ; ++j)
      if (j0 + j < na) dv[j] = ld_fdm<P>(dinv, io + base + (j0 + j) * stride);
  }
  line_products<P, NI, NJ, true>(A, na, j0, x, o);
#pragma unroll
  for (int j = 0; j < NJ; ++j) {
    if (j0 + j >= na) break;
    const int idx = base + (j0 + j) * stride;
    if (EPI == 0) {
      out[idx] = o[j];
    } else if (EPI == 1) {
      typename P::Acc d;
      P::init(d);
      P::fma(d, o[j], dv[j]);
      out[idx] = P::get(d);
    } else if (EPI == 2) {
      out[idx] = P::neg(o[j]);
    } else {
      fin(idx, o[j]);
    }
  }
}

template <class P, int N7, int EPI, class Fin>
__device__ __forceinline__ void contract1(const typename P::V* A, int ax, const int* nr, const typename P::V* in,
                                          typename P::V* out, const void* dinv, int64_t io, Fin fin) {
  using V = typename P::V;
  const int n7[3] = {7, 7, 7};
  const int* n = N7 ? n7 : nr;
  const int na = N7 ? 7 : (ax == 0 ? n[0] : (ax == 1 ? n[1] : n[2]));
  const int nl = N7 ? 49 : (ax == 0 ? n[1] * n[2] : (ax == 1 ? n[0] * n[2] : n[0] * n[1]));
  constexpr int NI = N7 ? 7 : 9;
  const int part = threadIdx.x >> 6;
  if (part > 1) return;
  for (int l = threadIdx.x & 63; l < nl; l += 64) {
    int base, stride;
    line_geom(ax, n, l, base, stride);
    V x[NI];
#pragma unroll
    for (int i = 0; i < NI; ++i) x[i] = i < na ? in[base + i * stride] : P::zero();
    if (part == 0) {
      line_out<P, NI, 4, EPI>(A, na, 0, x, base, stride, out, dinv, io, fin);
    } else if (N7) {
      line_out<P, NI, 3, EPI>(A, na, 4, x, base, stride, out, dinv, io, fin);
    } else if (na > 4) {
      line_out<P, NI, 4, EPI>(A, na, 4, x, base, stride, out, dinv, io, fin);
      if (na > 8) line_out<P, NI, 1, EPI>(A, na, 8, x, base, stride, out, dinv, io, fin);
    }
  }
}

// K_II^{-1} of t (destroyed); the last step as EPI says, into t for EPI 2
template <class P, int N7, int EPI, class Fin>
__device__ __forceinline__ void fdm_lines(const typename P::V* Vs, const int* n, typename P::V* t, typename P::V* u,
                                          const void* dinv, int64_t io, Fin fin) {
  auto none = [](int, typename P::V) {};
  contract1<P, N7, 0>(Vs, 0, n, t, u, dinv, io, none);
  __syncthreads();
  contract1<P, N7, 0>(Vs + 2 * VMAT, 1, n, u, t, dinv, io, none);
  __syncthreads();
  contract1<P, N7, 1>(Vs + 4 * VMAT, 2, n, t, u, dinv, io, none);
  __syncthreads();
  contract1<P, N7, 0>(Vs + VMAT, 0, n, u, t, dinv, io, none);
  __syncthreads();
  contract1<P, N7, 0>(Vs + 3 * VMAT, 1, n, t, u, dinv, io, none);
  __syncthreads();
  contract1<P, N7, EPI>(Vs + 5 * VMAT, 2, n, u, t, dinv, io, fin);
}

// rows of slices [b, e) times v (compact local vector: interface, then interior); emit(out, value)
template <class P, class Emit>
__device__ __forceinline__ void apply_rows(const LocalRows& R, int b, int e, int nb_base, const typename P::V* coef,
                                           const typename P::V* v, Emit emit) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int sl = b + warp; sl < e; sl += nw) {
    const int off = R.sl_off[sl] + lane;
    const int cnt = R.sl_cnt[sl * 32 + lane], o = R.sl_out[sl * 32 + lane];
    const typename P::V* c = coef + off;
    const int16_t* nb = R.nb + nb_base + off;
    typename P::Acc acc[3];
#pragma unroll
    for (int u = 0; u < 3; ++u) P::init(acc[u]);
    // nine entries' loads before their products (a face row has 18)
    for (int q0 = 0; q0 < cnt; q0 += 9) {
      typename P::V cv[9];
      int ni[9];
#pragma unroll
      for (int u = 0; u < 9; ++u)
        if (q0 + u < cnt) {
          cv[u] = c[(q0 + u) * 32];
          ni[u] = nb[(q0 + u) * 32];
        }
#pragma unroll
      for (int u = 0; u < 9; ++u)
        if (q0 + u < cnt) P::fma(acc[u % 3], cv[u], v[ni[u]]);
    }
    if (o >= 0) emit(o, P::add(P::add(P::get(acc[0]), P::get(acc[1])), P::get(acc[2])));
  }
}

constexpr int LBS = 128;  // threads of the single-vector kernel: 98 line halves, four slices of rows. 416 (all
                          // slices of a pass at once) took 47 us instead of 26 on 512 subdomains

// One vector. 12.9 KB of shared memory per 8^3 subdomain (a compact vector and one interior buffer 8.6 KB, the
// staged bases 4.3 KB) and 72 registers a thread (95 in the df64 recovery): registers let seven (five) CTAs on an SM,
// whose phases overlap; the rows' coefficients stream from HBM (about 77 KB per 8^3 subdomain). Bound by
// latency, of instruction fetches first of all (the unrolled products), then of the coefficients.
template <class P, int MODE>
__global__ void __launch_bounds__(LBS) k_local_apply(DevMesh m, const double* __restrict__ xg,
                                                     const double* __restrict__ f, double* __restrict__ out) {
  using V = typename P::V;
  const LocalRows& R = m.rows;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  V* Vs = reinterpret_cast<V*>(smem_raw);  // [6][VMAT]
  V* v = Vs + 6 * VMAT;                     // [nG + nI] interface values, then interior values
  __shared__ int n[3];
  const int s = blockIdx.x;
  const int64_t io = m.ioff[s], go = m.goff[s];
  const int nG = (int)(m.goff[s + 1] - go), nI = (int)(m.ioff[s + 1] - io);
  V* t = v + nG;
  V* u = t + nI;  // [nI]
  const int* tr = R.trange + 5 * R.type[s];
  const V* coef = static_cast<const V*>(R.coef) + R.coff[s];
  if (threadIdx.x < 3) n[threadIdx.x] = m.fdm_n[3 * s + threadIdx.x];
  if (MODE != ELEM_CONDENSE)
    for (int j = threadIdx.x; j < nG; j += LBS) v[j] = P::from_d(xg[m.gmap[go + j]]);
  else
    for (int j = threadIdx.x; j < nG; j += LBS) v[j] = P::zero();
  for (int j = threadIdx.x; j < nI; j += LBS) t[j] = MODE == ELEM_SCHUR ? P::zero() : P::from_d(f[R.ifree[io + j]]);
  stage_bases<P>(m, s, Vs);
  __syncthreads();
  if (MODE == ELEM_SCHUR) {
    apply_rows<P>(R, tr[0], tr[1], tr[4], coef, v, [&](int o, V y) { v[o] = y; });
    __syncthreads();
  } else if (MODE == ELEM_RECOVER) {
    apply_rows<P>(R, tr[0], tr[1], tr[4], coef, v,
                  [&](int o, V y) { v[o] = P::from_d(f[R.ifree[io + o - nG]] - P::to_d(y)); });
    __syncthreads();
  }
  const bool n7 = n[0] == 7 && n[1] == 7 && n[2] == 7;
  if (MODE == ELEM_RECOVER) {
    auto fin = [&](int idx, V y) { out[R.ifree[io + idx]] = P::to_d(y); };
    if (n7)
      fdm_lines<P, 1, 3>(Vs, n, t, u, m.fdm_Dinv, io, fin);
    else
      fdm_lines<P, 0, 3>(Vs, n, t, u, m.fdm_Dinv, io, fin);
    // interface values: each interface dof written by its first copy's subdomain
    for (int j = threadIdx.x; j < nG; j += LBS) {
      const int g = m.gmap[go + j];
      if (m.gidx[m.gptr[g]] == (int)(go + j)) out[m.gamma_free[g]] = xg[g];
    }
    return;
  }
  auto none = [](int, V) {};
  if (n7)
    fdm_lines<P, 1, 2>(Vs, n, t, u, m.fdm_Dinv, io, none);
  else
    fdm_lines<P, 0, 2>(Vs, n, t, u, m.fdm_Dinv, io, none);
  __syncthreads();
  apply_rows<P>(R, tr[2], tr[3], tr[4], coef, v, [&](int o, V y) { out[go + o] = P::to_d(y); });
}

template <class P, int MODE>
static void local_go(const DevMesh& m, const double* xg, const double* f, double* out,
                     cudaStream_t s) {
  const size_t smem = sizeof(typename P::V) * ((size_t)6 * VMAT + m.rows.max_loc + m.max_nint);
  max_smem(k_local_apply<P, MODE>, smem);
  k_local_apply<P, MODE><<<m.S, LBS, smem, s>>>(m, xg, f, out);
}

void launch_local_apply(const DevMesh& m, int mode, const double* xg, const double* f, double* out,
                        cudaStream_t s) {
  const bool df = m.schur_prec == DD_PREC_DF64;
  if (mode == ELEM_SCHUR)
    df ? local_go<PolDF, ELEM_SCHUR>(m, xg, f, out, s) : local_go<PolF64, ELEM_SCHUR>(m, xg, f, out, s);
  else if (mode == ELEM_CONDENSE)
    df ? local_go<PolDF, ELEM_CONDENSE>(m, xg, f, out, s) : local_go<PolF64, ELEM_CONDENSE>(m, xg, f, out, s);
  else
    df ? local_go<PolDF, ELEM_RECOVER>(m, xg, f, out, s) : local_go<PolF64, ELEM_RECOVER>(m, xg, f, out, s);
  DD_CHECK_LAUNCH();
}

// ---------------------------------------------------------------------------
// dense local solver: the same rows around a product with the boundary block of K_II^{-1}
// ---------------------------------------------------------------------------
// INTERIOR: t_B = K_BG x_G; else y = K_GG x_G - K_GB s_B
template <class P, bool INTERIOR>
__global__ void __launch_bounds__(LBS) k_rows(DevMesh m, const double* __restrict__ xg, const double* __restrict__ sB,
                                              double* __restrict__ out) {
  using V = typename P::V;
  const LocalRows& R = m.rows;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  V* v = reinterpret_cast<V*>(smem_raw);  // [nG + nB]
  const int s = blockIdx.x;
  const int64_t go = m.goff[s], bo = R.boff[s];
  const int nG = (int)(m.goff[s + 1] - go), nB = (int)(R.boff[s + 1] - bo);
  const int* tr = R.trange + 5 * R.type[s];
  const V* coef = static_cast<const V*>(R.coef) + R.coff[s];
  for (int j = threadIdx.x; j < nG; j += LBS) v[j] = P::from_d(xg[m.gmap[go + j]]);
  if (!INTERIOR)
    for (int j = threadIdx.x; j < nB; j += LBS) v[nG + j] = P::from_d(-sB[bo + j]);
  __syncthreads();
  if (INTERIOR)
    apply_rows<P>(R, tr[0], tr[1], tr[4], coef, v, [&](int o, V y) { out[bo + o - nG] = P::to_d(y); });
  else
    apply_rows<P>(R, tr[2], tr[3], tr[4], coef, v, [&](int o, V y) { out[go + o] = P::to_d(y); });
}

template <bool INTERIOR>
static void rows_go(const DevMesh& m, const double* xg, const double* sB, double* out, cudaStream_t s) {
  const size_t smem = sizeof(double) * (size_t)m.rows.max_loc;  // df64 values have the same size
  if (m.schur_prec == DD_PREC_DF64)
    k_rows<PolDF, INTERIOR><<<m.S, LBS, smem, s>>>(m, xg, sB, out);
  else
    k_rows<PolF64, INTERIOR><<<m.S, LBS, smem, s>>>(m, xg, sB, out);
  DD_CHECK_LAUNCH();
}

void launch_rows_interior(const DevMesh& m, const double* xg, double* tB, cudaStream_t s) {
  rows_go<true>(m, xg, nullptr, tB, s);
}
void launch_rows_interface(const DevMesh& m, const double* xg, const double* sB, double* yloc, cudaStream_t s) {
  rows_go<false>(m, xg, sB, yloc, s);
}

// ---------------------------------------------------------------------------
// RC ensemble members per CTA (members [m0, m0 + RC), lane = member within a line or pair of
// members within a row): the bases and the rows' coefficients serve all of them
// ---------------------------------------------------------------------------
template <class P, int RC, int N7, bool SCALE, bool NEG>
__device__ __forceinline__ void contract_b(const typename P::V* A, int ax, const int* nr, typename P::V* t,
                                           const void* dinv, int64_t io) {
  using V = typename P::V;
  const int n7[3] = {7, 7, 7};
  const int* n = N7 ? n7 : nr;
  const int na = N7 ? 7 : (ax == 0 ? n[0] : (ax == 1 ? n[1] : n[2]));
  const int nl = N7 ? 49 : (ax == 0 ? n[1] * n[2] : (ax == 1 ? n[0] * n[2] : n[0] * n[1]));
  constexpr int NI = N7 ? 7 : 9;
  // a thread owns a line of one member: it reads the line before it writes it, in place
  for (int q = threadIdx.x; q < nl * RC; q += blockDim.x) {
    const int mm = q % RC;
    int base, stride;
    line_geom(ax, n, q / RC, base, stride);
    V* p = t + (size_t)base * RC + mm;
    V x[NI];
#pragma unroll
    for (int i = 0; i < NI; ++i) x[i] = i < na ? p[i * stride * RC] : P::zero();
    auto put = [&](int j, V y) {
      if (j >= na) return;
      if (SCALE) {
        typename P::Acc d;
        P::init(d);
        P::fma(d, y, ld_fdm<P>(dinv, io + base + j * stride));
        y = P::get(d);
      }
      p[j * stride * RC] = NEG ? P::neg(y) : y;
    };
    V o[4];
    line_products<P, NI, 4, false>(A, na, 0, x, o);
#pragma unroll
    for (int j = 0; j < 4; ++j) put(j, o[j]);
    if (N7) {
      line_products<P, NI, 3, false>(A, na, 4, x, o);
#pragma unroll
      for (int j = 0; j < 3; ++j) put(4 + j, o[j]);
    } else if (na > 4) {
      line_products<P, NI, 4, false>(A, na, 4, x, o);
#pragma unroll
      for (int j = 0; j < 4; ++j) put(4 + j, o[j]);
      if (na > 8) {
        line_products<P, NI, 1, false>(A, na, 8, x, o);
        put(8, o[0]);
      }
    }
  }
}

template <class P, int RC, int N7, bool NEG>
__device__ __forceinline__ void fdm_lines_b(const typename P::V* Vs, const int* n, typename P::V* t, const void* dinv,
                                            int64_t io) {
  contract_b<P, RC, N7, false, false>(Vs, 0, n, t, dinv, io);
  __syncthreads();
  contract_b<P, RC, N7, false, false>(Vs + 2 * VMAT, 1, n, t, dinv, io);
  __syncthreads();
  contract_b<P, RC, N7, true, false>(Vs + 4 * VMAT, 2, n, t, dinv, io);
  __syncthreads();
  contract_b<P, RC, N7, false, false>(Vs + VMAT, 0, n, t, dinv, io);
  __syncthreads();
  contract_b<P, RC, N7, false, false>(Vs + 3 * VMAT, 1, n, t, dinv, io);
  __syncthreads();
  contract_b<P, RC, N7, false, NEG>(Vs + 5 * VMAT, 2, n, t, dinv, io);
  __syncthreads();
}

// rows times RC members: lane = row (of 32 / (RC / 2)) x pair of members
template <class P, int RC, class Emit>
__device__ __forceinline__ void apply_rows_b(const LocalRows& R, int b, int e, int nb_base,
                                             const typename P::V* coef, const typename P::V* v, Emit emit) {
  using V = typename P::V;
  constexpr int PAIRS = RC / 2, IPW = 32 / PAIRS, WPS = 32 / IPW;  // rows per warp, warps per slice
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int pr = lane % PAIRS;
  for (int w = warp; w < (e - b) * WPS; w += nw) {
    const int sl = b + w / WPS, it = (w % WPS) * IPW + lane / PAIRS;
    const int off = R.sl_off[sl] + it;
    const int cnt = R.sl_cnt[sl * 32 + it], o = R.sl_out[sl * 32 + it];
    const V* c = coef + off;
    const int16_t* nb = R.nb + nb_base + off;
    typename P::Acc a0[2], a1[2];  // two members, two chains each
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      P::init(a0[u]);
      P::init(a1[u]);
    }
    for (int q0 = 0; q0 < cnt; q0 += 6) {
      V cv[6];
      int ni[6];
#pragma unroll
      for (int u = 0; u < 6; ++u)
        if (q0 + u < cnt) {
          cv[u] = c[(q0 + u) * 32];
          ni[u] = nb[(q0 + u) * 32];
        }
#pragma unroll
      for (int u = 0; u < 6; ++u)
        if (q0 + u < cnt) {
          const Two<V> x = *reinterpret_cast<const Two<V>*>(v + (size_t)ni[u] * RC + 2 * pr);
          P::fma(a0[u & 1], cv[u], x.a);
          P::fma(a1[u & 1], cv[u], x.b);
        }
    }
    P::merge(a0[0], a0[1]);
    P::merge(a1[0], a1[1]);
    if (o >= 0) emit(o, 2 * pr, P::get(a0[0]), P::get(a1[0]));
  }
}

// threads of the ensemble kernel: the 49 lines of RC members
template <int RC>
constexpr int lbt() {
  return (49 * RC + 31) / 32 * 32;
}

template <class P, int MODE, int RC>
__global__ void __launch_bounds__(lbt<RC>(), 16 / RC) k_local_apply_b(DevMesh m, const df64* __restrict__ xg,
                                                          const df64* __restrict__ f, df64* __restrict__ out) {
  using V = typename P::V;
  const LocalRows& R = m.rows;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  V* Vs = reinterpret_cast<V*>(smem_raw);
  V* v = Vs + 6 * VMAT;  // [nG + nI][RC]
  __shared__ int n[3];
  constexpr int LBT = lbt<RC>();
  const int s = blockIdx.x, m0 = blockIdx.y * RC;
  const int64_t io = m.ioff[s], go = m.goff[s];
  const int nG = (int)(m.goff[s + 1] - go), nI = (int)(m.ioff[s + 1] - io);
  V* t = v + (size_t)nG * RC;
  const int* tr = R.trange + 5 * R.type[s];
  const V* coef = static_cast<const V*>(R.coef) + R.coff[s];
  if (threadIdx.x < 3) n[threadIdx.x] = m.fdm_n[3 * s + threadIdx.x];
  for (int q = threadIdx.x; q < nG * RC; q += LBT)
    v[q] = MODE == ELEM_CONDENSE ? P::zero() : P::from_v(xg[(int64_t)m.gmap[go + q / RC] * BW + m0 + q % RC]);
  for (int q = threadIdx.x; q < nI * RC; q += LBT)
    t[q] = MODE == ELEM_SCHUR ? P::zero() : P::from_v(f[(int64_t)R.ifree[io + q / RC] * BW + m0 + q % RC]);
  stage_bases<P>(m, s, Vs);
  __syncthreads();
  if (MODE != ELEM_CONDENSE) {
    apply_rows_b<P, RC>(R, tr[0], tr[1], tr[4], coef, v, [&](int o, int mm, V y0, V y1) {
      V* d = v + (size_t)o * RC + mm;
      if (MODE == ELEM_SCHUR) {
        d[0] = y0;
        d[1] = y1;
      } else {
        d[0] = P::add(d[0], P::neg(y0));
        d[1] = P::add(d[1], P::neg(y1));
      }
    });
    __syncthreads();
  }
  constexpr bool NEG = MODE != ELEM_RECOVER;
  if (n[0] == 7 && n[1] == 7 && n[2] == 7)
    fdm_lines_b<P, RC, 1, NEG>(Vs, n, t, m.fdm_Dinv, io);
  else
    fdm_lines_b<P, RC, 0, NEG>(Vs, n, t, m.fdm_Dinv, io);
  if (MODE == ELEM_RECOVER) {
    for (int q = threadIdx.x; q < nI * RC; q += LBT)
      out[(int64_t)R.ifree[io + q / RC] * BW + m0 + q % RC] = P::to_v(t[q]);
    for (int q = threadIdx.x; q < nG * RC; q += LBT) {
      const int j = q / RC, g = m.gmap[go + j];
      if (m.gidx[m.gptr[g]] == (int)(go + j))
        out[m.gamma_free[g] * BW + m0 + q % RC] = xg[(int64_t)g * BW + m0 + q % RC];
    }
    return;
  }
  apply_rows_b<P, RC>(R, tr[2], tr[3], tr[4], coef, v, [&](int o, int mm, V y0, V y1) {
    df64* d = out + (go + o) * BW + m0 + mm;
    d[0] = P::to_v(y0);
    d[1] = P::to_v(y1);
  });
}

template <class P, int MODE, int RC>
static void local_b_go(const DevMesh& m, int nact, const df64* xg, const df64* f, df64* out,
                       cudaStream_t s) {
  const size_t smem = sizeof(typename P::V) * ((size_t)6 * VMAT + (size_t)m.rows.max_loc * RC);
  max_smem(k_local_apply_b<P, MODE, RC>, smem);
  k_local_apply_b<P, MODE, RC><<<dim3(m.S, (nact + RC - 1) / RC), lbt<RC>(), smem, s>>>(m, xg, f, out);
}
template <class P, int RC>
static void local_b_mode(const DevMesh& m, int mode, int nact, const df64* xg, const df64* f,
                         df64* out, cudaStream_t s) {
  if (mode == ELEM_SCHUR)
    local_b_go<P, ELEM_SCHUR, RC>(m, nact, xg, f, out, s);
  else if (mode == ELEM_CONDENSE)
    local_b_go<P, ELEM_CONDENSE, RC>(m, nact, xg, f, out, s);
  else
    local_b_go<P, ELEM_RECOVER, RC>(m, nact, xg, f, out, s);
}

void launch_local_apply_b(const DevMesh& m, int mode, int rc, int nact, const df64* xg,
                          const df64* f, df64* out, cudaStream_t s) {
  if (m.schur_prec == DD_PREC_DF64) {
    if (rc == 4)
      local_b_mode<PolDF, 4>(m, mode, nact, xg, f, out, s);
    else
      local_b_mode<PolDF, 8>(m, mode, nact, xg, f, out, s);
  } else {
    local_b_mode<PolF64, 8>(m, mode, nact, xg, f, out, s);
  }
  DD_CHECK_LAUNCH();
}

}  // namespace dd

// Coarse tail of an FP32 V-cycle (included by pfc_mixed.cu, inside its anonymous
// namespace): every level of at most kTailMaxN^3 cells in one launch of one
// thread block whose levels all live in shared memory.
//
// What bounds it is the shared-memory rate of one SM (32 words a clock) and
// the latency of a pass, so the levels are stored by colour: a component's
// colour-0 cells in the order of the colour-split layout, then its colour-1
// cells, n^3/2 each, without gaps.  A pass over one colour then reads and
// writes consecutive words (stored in natural order, half of its wavefronts
// were bank conflicts), a thread's positions and their neighbours are the same
// indices for both colours and are worked out once per call, and r, q of a
// thread's cells stay in registers over the sweeps of a call.  Measured (ncu):
// V(2,2) on 16^3 with four coarsest sweeps on 8^3 36.4 -> 19.6 us, 9.2 of them at
// the shared-memory rate (19.1 k wavefronts), the SM issuing 57 % of the time; 16^3
// alone with two sweeps 16.4 -> 9.6 (warm caches).

extern __shared__ float tsm[];

// A level in shared memory: component f of d, r, t, colour c, at element
// x + (2 f + c) cs of tsm; q likewise.  cs = n^3 / 2 + 16: the pad puts the two
// colours of a row in different banks for the prolongation, which reads both.
// Offsets, not pointers: a call that takes a pointer loses that it is shared
// memory.
struct TLev {
  int d, r, q, t;
  int hc, cs;                            // cells of a colour, distance of the colours
};

__host__ __device__ constexpr int tail_floats(int n) { return 10 * (n * n * n + 32); }

__device__ __forceinline__ TLev tlev(const TailParams& P, int l) {
  const int n = P.L[l].n;
  TLev S;
  S.hc = n * n * n >> 1;
  S.cs = S.hc + 16;
  S.d = P.off[l];
  S.r = S.d + 6 * S.cs;
  S.q = S.d + 12 * S.cs;
  S.t = S.d + 14 * S.cs;
  return S;
}

// x / d for x d < 2^16 from recip = 65536 / d + 1 (worked out on the host): a
// division by a run-time number takes about 25 instructions, in phases that
// have 100.
__device__ __forceinline__ int small_div(int x, int recip) {
  return (x * recip) >> 16;
}

// Position `pos` = p + half (j + n k) of both colours: the positions of its y
// and z neighbours and of the x neighbours below it and above it (PAIR: above
// position p + 1), all of the other colour, and the parity sg = (j + k) & 1: a
// cell of colour c lies at i = 2p + (sg ^ c), so its x neighbours are position p
// and the one above if sg ^ c, else the one below.
template <bool PAIR>
struct TPos {
  int c, ym, yp, zm, zp, xl, xr;
  bool sg, on;
  __device__ __forceinline__ TPos(const TailParams& P, int l, int pos) {
    constexpr int w = PAIR ? 2 : 1;
    const int n = P.L[l].n, half = n >> 1, hp = half * n;
    const int r = small_div(pos, P.rhalf[l]), p = pos - r * half;
    const int k = small_div(r, P.rn[l]), j = r - k * n;
    on = k < n;
    c = pos;
    ym = pos + (j == 0 ? hp - half : -half);
    yp = pos + (j + 1 == n ? half - hp : half);
    zm = pos + (k == 0 ? hp * (n - 1) : -hp);
    zp = pos + (k + 1 == n ? -hp * (n - 1) : hp);
    xl = pos + (p == 0 ? half - 1 : -1);
    xr = pos + (p + w == half ? w - half : w);
    sg = (j + k) & 1;
  }
};

// One value, or two of adjacent positions.
template <bool PAIR>
struct TVal;
template <>
struct TVal<false> {
  using T = float;
  static __device__ __forceinline__ T ld(int at) { return tsm[at]; }
  static __device__ __forceinline__ void st(int at, T v) { tsm[at] = v; }
  static __device__ __forceinline__ T all(float v) { return v; }
  static __device__ __forceinline__ float top(T a) { return fabsf(a); }
  static __device__ __forceinline__ T diff(T a, T b) { return a - b; }
  static __device__ __forceinline__ T step(float w, T x, T old) { return fmaf(w, x - old, old); }
  // neighbour sum of the colour-c cell from the other colour's values at o
  static __device__ __forceinline__ T sum(const TPos<false>& P, int o, bool sg) {
    const float* const v = tsm + o;
    return ((v[P.c] + v[sg ? P.xr : P.xl]) + (v[P.ym] + v[P.yp])) + (v[P.zm] + v[P.zp]);
  }
  static __device__ __forceinline__ void solve(const LvlF& L, const T (&s)[3], const T (&rq)[4],
                                               T (&x)[3]) {
    lin_point(L, s[0], s[1], s[2], rq[3], rq[0], rq[1], rq[2], x[0], x[1], x[2]);
  }
};
template <>
struct TVal<true> {
  using T = float2;
  static __device__ __forceinline__ T ld(int at) { return *reinterpret_cast<const T*>(tsm + at); }
  static __device__ __forceinline__ void st(int at, T v) { *reinterpret_cast<T*>(tsm + at) = v; }
  static __device__ __forceinline__ T all(float v) { return f2_all(v); }
  static __device__ __forceinline__ float top(T a) { return fmaxf(fabsf(a.x), fabsf(a.y)); }
  static __device__ __forceinline__ T diff(T a, T b) { return f2_sub(a, b); }
  static __device__ __forceinline__ T step(float w, T x, T old) {
    return f2_fma(f2_all(w), f2_sub(x, old), old);
  }
  static __device__ __forceinline__ T sum(const TPos<true>& P, int o, bool sg) {
    return nbsum2(ld(o + P.c), tsm[o + (sg ? P.xr : P.xl)], sg, ld(o + P.ym), ld(o + P.yp),
                  ld(o + P.zm), ld(o + P.zp));
  }
  static __device__ __forceinline__ void solve(const LvlF& L, const T (&s)[3], const T (&rq)[4],
                                               T (&x)[3]) {
    lin_point2(L, s[0], s[1], s[2], rq[3], rq[0], rq[1], rq[2], x[0], x[1], x[2]);
  }
};

// `sweeps` sweeps of SLOTS positions (PAIR: of position pairs) a thread.  zero:
// d = 0 on entry (not read).  Coarsest: stop once the largest change is <= 1e-6
// of the largest value, tested every fourth sweep (the outer FP64 loop absorbs
// the rest).
template <bool PAIR, int SLOTS>
__device__ __forceinline__ void tail_sweeps(const TailParams& P, int l, const TLev S, int sweeps,
                                            bool zero, bool coarsest, float (*red)[32],
                                            int* done) {
  const LvlF L = P.L[l];
  const int kind = P.kind[l];
  const float w = P.w;
  using V = TVal<PAIR>;
  using T = typename V::T;
  const int cs = S.cs, step = PAIR ? 2 : 1;
  const TPos<PAIR> pos[2] = {TPos<PAIR>(P, l, threadIdx.x * step),
                             TPos<PAIR>(P, l, (threadIdx.x + blockDim.x) * step)};
  T rq[SLOTS][2][4];
#pragma unroll
  for (int s = 0; s < SLOTS; ++s)
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int f = 0; f < 4; ++f)
        rq[s][c][f] = pos[s].on ? V::ld((f < 3 ? S.r + 2 * f * cs : S.q) + c * cs + pos[s].c)
                                : V::all(0.f);
  int d = S.d, o = S.t;                  // Jacobi: d -> o, then exchanged
  for (int sweep = 0; sweep < sweeps; ++sweep) {
    const bool fresh = zero && sweep == 0;
    const bool test = coarsest && (sweep & 3) == 3 && sweep + 1 < sweeps;
    float change = 0.f, size = 0.f;
    if (kind == PFC_SWEEP_JACOBI) {
#pragma unroll
      for (int s = 0; s < SLOTS; ++s) {
        if (!pos[s].on) continue;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          T sum[3], old[3], x[3];
#pragma unroll
          for (int f = 0; f < 3; ++f) {
            sum[f] = old[f] = V::all(0.f);
            if (!fresh) {
              sum[f] = V::sum(pos[s], d + (2 * f + 1 - c) * cs, pos[s].sg != (c != 0));
              old[f] = V::ld(d + (2 * f + c) * cs + pos[s].c);
            }
          }
          V::solve(L, sum, rq[s][c], x);
#pragma unroll
          for (int f = 0; f < 3; ++f) {
            const T v = V::step(w, x[f], old[f]);
            V::st(o + (2 * f + c) * cs + pos[s].c, v);
            if (test) {
              change = fmaxf(change, V::top(V::diff(v, old[f])));
              size = fmaxf(size, V::top(v));
            }
          }
        }
      }
      __syncthreads();
      const int x = d;
      d = o;
      o = x;
    } else {
#pragma unroll
      for (int c = 0; c < 2; ++c) {
#pragma unroll
        for (int s = 0; s < SLOTS; ++s) {
          if (!pos[s].on) continue;
          T sum[3], x[3];
#pragma unroll
          for (int f = 0; f < 3; ++f)
            sum[f] = fresh && c == 0
                         ? V::all(0.f)
                         : V::sum(pos[s], d + (2 * f + 1 - c) * cs, pos[s].sg != (c != 0));
          V::solve(L, sum, rq[s][c], x);
#pragma unroll
          for (int f = 0; f < 3; ++f) {
            const int at = d + (2 * f + c) * cs + pos[s].c;
            if (test) {
              const T old = fresh ? V::all(0.f) : V::ld(at);
              change = fmaxf(change, V::top(V::diff(x[f], old)));
              size = fmaxf(size, V::top(x[f]));
            }
            V::st(at, x[f]);
          }
        }
        __syncthreads();
      }
    }
    if (!test) continue;
    for (int b = 16; b > 0; b >>= 1) {
      change = fmaxf(change, __shfl_down_sync(0xffffffffu, change, b));
      size = fmaxf(size, __shfl_down_sync(0xffffffffu, size, b));
    }
    if ((threadIdx.x & 31) == 0) {
      red[0][threadIdx.x >> 5] = change;
      red[1][threadIdx.x >> 5] = size;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      float cmax = 0.f, z = 0.f;
      for (int v = 0; v < (int)((blockDim.x + 31) >> 5); ++v) {
        cmax = fmaxf(cmax, red[0][v]);
        z = fmaxf(z, red[1][v]);
      }
      *done = (cmax <= 1e-6f * z);
    }
    __syncthreads();
    if (*done) break;
  }
  if (d != S.d) {                        // an odd number of Jacobi sweeps
#pragma unroll
    for (int s = 0; s < SLOTS; ++s)
      if (pos[s].on)
#pragma unroll
        for (int f = 0; f < 6; ++f) V::st(S.d + f * cs + pos[s].c, V::ld(S.t + f * cs + pos[s].c));
    __syncthreads();
  }
}

// The transfers put two threads on a coarse cell (I, J, K), one per child row jj
// in y, so that the block's warps are busy and consecutive threads touch
// consecutive rows of the fine level (without bank conflicts).
struct TCoarse {
  int t, jj, I, J, K;
  bool on;
  // rnc: small_div's reciprocal of nc
  __device__ __forceinline__ TCoarse(int nc, int rnc) {
    int r = small_div(threadIdx.x, rnc);     // 2 nc^3 <= blockDim (tail_threads)
    I = threadIdx.x - r * nc;
    jj = r & 1;
    r >>= 1;
    K = small_div(r, rnc);
    J = r - K * nc;
    on = K < nc;
    t = I + nc * r;
  }
  // position of (I, J, K) in a level of nc^3 cells stored by colour, and its colour
  __device__ __forceinline__ int at(int nc) const { return (nc >> 1) * (J + nc * K) + (I >> 1); }
  __device__ __forceinline__ int colour() const { return (I + J + K) & 1; }
};

// rho = r - J d of the fine level averaged onto the coarse level's r (the block
// sums of k_lin_residual_restrict32), and q with it; the second row's share
// passes through the fine level's scratch t.  dzero: d = 0.
__device__ __forceinline__ void tail_restrict(const TailParams& P, int l, const TLev F,
                                              const TLev C, bool dzero) {
  const LvlF L = P.L[l];
  const int n = L.n, half = n >> 1, nc = half, cs = F.cs, hp = half * n, cells = nc * nc * nc;
  const TCoarse c(nc, P.rhalf[l]);
  float a[4] = {0.f, 0.f, 0.f, 0.f};     // rows, q
  if (c.on) {
    // position I of both colours in row j of the two child planes
    const int j = 2 * c.J + c.jj, k = 2 * c.K, base = c.I + half * (j + n * k);
    const int row[2] = {base, base + hp};
#pragma unroll
    for (int f = 0; f < 3; ++f)
#pragma unroll
      for (int q = 0; q < 2; ++q)
        a[f] += tsm[F.r + 2 * f * cs + row[q]] + tsm[F.r + (2 * f + 1) * cs + row[q]];
    float q2[2][2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      q2[q][0] = tsm[F.q + row[q]];
      q2[q][1] = tsm[F.q + cs + row[q]];
      a[3] += q2[q][0] + q2[q][1];
    }
    if (!dzero) {
      const int Im = c.I == 0 ? nc - 1 : -1, Ip = c.I + 1 == nc ? 1 - nc : 1;
      // the row beside this one and the planes below and above, outside the block
      const int dy = c.jj ? (j + 1 == n ? half - hp : half) : (j == 0 ? hp - half : -half);
      const int zm = base + (k == 0 ? hp * (n - 1) : -hp);
      const int zp = base + (k + 2 == n ? hp * (2 - n) : 2 * hp);
      float in[3], out[3], qp = 0.f;
#pragma unroll
      for (int f = 0; f < 3; ++f) {
        const float* const v0 = tsm + F.d + 2 * f * cs;
        const float* const v1 = v0 + cs;
        float si = 0.f, so = (v0[zm] + v1[zm]) + (v0[zp] + v1[zp]);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const bool par = (q + c.jj) & 1;               // (j + k) & 1 of the row
          const float x0 = v0[row[q]], x1 = v1[row[q]];
          si += x0 + x1;
          if (f == 0) qp = fmaf(q2[q][0], x0, fmaf(q2[q][1], x1, qp));
          // (2I - 1, j, k) and (2I + 2, j, k)
          so += v0[row[q] + Im + (par ? 0 : cs)] + v0[row[q] + Ip + (par ? cs : 0)];
          so += v0[row[q] + dy] + v1[row[q] + dy];
        }
        in[f] = si;
        out[f] = so;
      }
      a[0] = fmaf(L.tg, fmaf(-3.f, in[1], out[1]), a[0] - in[0]);
      a[1] = fmaf(L.g, fmaf(-3.f, in[2], out[2]), a[1] - in[1]) + qp;
      a[2] = fmaf(L.gh, fmaf(-3.f, in[0], out[0]), a[2] - in[2]);
    }
    if (c.jj)
#pragma unroll
      for (int f = 0; f < 4; ++f) tsm[F.t + f * cells + c.t] = a[f];
  }
  __syncthreads();
  if (c.on && !c.jj) {
    const int o = c.at(nc) + c.colour() * C.cs;
#pragma unroll
    for (int f = 0; f < 4; ++f)
      tsm[(f < 3 ? C.r + 2 * f * C.cs : C.q) + o] = 0.125f * (a[f] + tsm[F.t + f * cells + c.t]);
  }
  __syncthreads();
}

// d_F += P d_C (assign: d_F = P d_C): one-dimensional passes z, y, x with
// weights 3 and 1 as k_prolong_add32.
__device__ __forceinline__ void tail_prolong(const TailParams& P, int l, const TLev C,
                                             const TLev F, bool assign) {
  const int n = P.L[l].n, half = n >> 1, nc = half, hn = nc >> 1;
  const TCoarse c(nc, P.rhalf[l]);
  if (c.on) {
    const int xs[3] = {c.I == 0 ? nc - 1 : c.I - 1, c.I, c.I + 1 == nc ? 0 : c.I + 1};
    // rows J and the one on the child's side, planes K - 1, K, K + 1
    const int ys[2] = {c.J, c.jj ? (c.J + 1 == nc ? 0 : c.J + 1) : (c.J == 0 ? nc - 1 : c.J - 1)};
    const int zs[3] = {c.K == 0 ? nc - 1 : c.K - 1, c.K, c.K + 1 == nc ? 0 : c.K + 1};
    // columns x - 1, x, x + 1 of a row whose J + K is even, and odd
    int ox[2][3];
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      ox[0][x] = (xs[x] & 1) * C.cs + (xs[x] >> 1);
      ox[1][x] = (1 - (xs[x] & 1)) * C.cs + (xs[x] >> 1);
    }
    const int base = c.I + half * (2 * c.J + c.jj + n * 2 * c.K);
#pragma unroll
    for (int f = 0; f < 3; ++f) {
      const float* const e = tsm + C.d + 2 * f * C.cs;
      float v[3][2][3];
#pragma unroll
      for (int z = 0; z < 3; ++z)
#pragma unroll
        for (int y = 0; y < 2; ++y)
#pragma unroll
          for (int x = 0; x < 3; ++x)
            v[z][y][x] = e[hn * (ys[y] + nc * zs[z]) + (((ys[y] + zs[z]) & 1) ? ox[1][x] : ox[0][x])];
#pragma unroll
      for (int kk = 0; kk < 2; ++kk) {
        float y[3];
#pragma unroll
        for (int x = 0; x < 3; ++x)
          y[x] = fmaf(3.f, fmaf(3.f, v[1][0][x], v[2 * kk][0][x]),
                      fmaf(3.f, v[1][1][x], v[2 * kk][1][x]));
        // child a (i = 2I + a) has colour a ^ par
        const int row = base + kk * half * n, par = (c.jj + kk) & 1;
        float* const a0 = tsm + F.d + (2 * f + par) * F.cs + row;
        float* const a1 = tsm + F.d + (2 * f + 1 - par) * F.cs + row;
        const float v0 = fmaf(3.f, y[1], y[0]), v1 = fmaf(3.f, y[1], y[2]);
        *a0 = assign ? (1.f / 64.f) * v0 : fmaf(1.f / 64.f, v0, *a0);
        *a1 = assign ? (1.f / 64.f) * v1 : fmaf(1.f / 64.f, v1, *a1);
      }
    }
  }
  __syncthreads();
}

// One V-cycle over the tail's levels; the top level's r, q (and d unless it
// starts from zero) come from global memory, the lower levels' r and q are
// averaged here, the top level's d goes back at the end.
__global__ void __launch_bounds__(kTailThreads) k_lin_tail32(TailParams P) {
  pdl_wait();
  __shared__ float red[2][32];
  __shared__ int done;
  const bool zero_top = P.zero_init != 0;
  const int n0 = P.L[0].n, half = n0 >> 1, cells = n0 * n0 * n0;
  const size_t off = (size_t)blockIdx.x * cells;   // one block per member
  const TLev S0 = tlev(P, 0);
  // position pos of colour c is element (pos / half) n + c half + pos % half of
  // the colour-split layout in global memory; all of a thread's loads come
  // before its stores
  {
    float v[2][7][2];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const int pos = threadIdx.x + s * blockDim.x, row = small_div(pos, P.rhalf[0]);
      const size_t g = off + row * n0 + pos - row * half;
      if (pos >= S0.hc) break;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
#pragma unroll
        for (int f = 0; f < 3; ++f) {
          v[s][f][c] = __ldg(P.gr[f] + g + c * half);
          if (!zero_top) v[s][4 + f][c] = P.gd[f][g + c * half];
        }
        v[s][3][c] = __ldg(P.gq + g + c * half);
      }
    }
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const int pos = threadIdx.x + s * blockDim.x;
      if (pos >= S0.hc) break;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
#pragma unroll
        for (int f = 0; f < 3; ++f) {
          tsm[S0.r + (2 * f + c) * S0.cs + pos] = v[s][f][c];
          if (!zero_top) tsm[S0.d + (2 * f + c) * S0.cs + pos] = v[s][4 + f][c];
        }
        tsm[S0.q + c * S0.cs + pos] = v[s][3][c];
      }
    }
  }
  __syncthreads();
  const int last = P.nlev - 1;
  unsigned dzero = 0;                    // levels whose d is still zero on the way up
  // down to the coarsest level and up again, in one loop: each of the phases is
  // in the code once, which an SM that runs it a few times has to fetch
  for (int s = 0; s <= 2 * last; ++s) {
    const int l = s <= last ? s : 2 * last - s;
    const bool down = s < last, coarsest = s == last;
    const TLev S = tlev(P, l);
    if (s > last) tail_prolong(P, l, tlev(P, l + 1), S, (dzero >> l) & 1u);
    const int nu = down ? P.nu1 : P.nu2;
    const int jf = P.kind[l] == PFC_SWEEP_JACOBI ? (l == 0 ? P.jfactor_top : P.jfactor) : 1;
    const int sweeps = coarsest ? P.coarse_sweeps : nu * jf;
    const bool zero = coarsest || (down && (l > 0 || zero_top));
    if (sweeps > 0) {
      if (P.L[l].n % 4 == 0)             // at most 1024 pairs
        tail_sweeps<true, 1>(P, l, S, sweeps, zero, coarsest, red, &done);
      else                               // n = 14: 1372 positions
        tail_sweeps<false, 2>(P, l, S, sweeps, zero, coarsest, red, &done);
    } else if (zero) {
      dzero |= 1u << l;
    }
    if (down) tail_restrict(P, l, S, tlev(P, l + 1), (dzero >> l) & 1u);
  }
  for (int pos = threadIdx.x; pos < S0.hc; pos += blockDim.x) {
    const int row = small_div(pos, P.rhalf[0]), g = row * n0 + pos - row * half;
#pragma unroll
    for (int f = 0; f < 3; ++f)
#pragma unroll
      for (int c = 0; c < 2; ++c) P.gd[f][off + g + c * half] = tsm[S0.d + (2 * f + c) * S0.cs + pos];
  }
}

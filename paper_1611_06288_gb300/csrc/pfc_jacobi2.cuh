// Two damped collective Jacobi sweeps of the FP32 correction solve in one pass
// over memory (included by pfc_mixed.cu, inside its anonymous namespace).
//
// On levels that L2 does not hold a sweep runs at the copy bandwidth, 40 B a
// cell.  Here the second sweep is formed from the first one's values before they
// leave the SM, so d, r and q are read and the result is written once for both.
// Two sweeps, us, two launches of k_lin_jacobi32m / one of this: 256^3 204 /
// 161, 192^3 99 / 68, 160^3 61 / 43, 132^3 33 / 30, 6 x 128^3 158 / 117, 3 x
// 96^3 36 / 28, 8 x 80^3 59 / 49, 42 x 64^3 139 / 110, 39 x 48^3 61.6 / 53.8, 60
// x 40^3 60 / 49.  What bounds it: the latency that 16 warps an SM (126 registers a
// thread) leave; no unit is full at 256^3 (ncu: issue 48 %, L1 / shared-memory pipe
// 47 % with 128 wavefronts a warp and plane, DRAM 53 %).
//
// A block owns whole rows (so that a row's neighbours are in the block, every
// access of a warp is aligned, and a plane of the tile is one range of memory)
// and marches upwards in z over `zc` planes, one plane k of the first sweep and
// plane k - 1 of the second per iteration.  A thread holds two positions of a row,
// both colours, as in the marching single sweep, and the first and last row of
// threads form the halo of the first sweep and write nothing.  The first sweep
// reads d as the single sweep does; its values go to shared memory, double
// buffered (one barrier a plane), for the second one's neighbours in x and y,
// and stay in registers for those in z.  r and q are loaded again for the second
// sweep, from L1 or L2: kept, their 16 registers would cost a quarter of the
// warps.  Tiles of part of a row (22 of 64 columns) needed 192 wavefronts: 184 us
// at 256^3.  Source planes through shared memory as well (cp.async): 205 us.
//
// Every value is formed with the operations and order of k_lin_jacobi32m: the
// result equals two launches of it bit for bit.

// CM: thread columns (n / 4) at most; RM: rows of threads at most.
template <int CM, int RM>
struct J2 {
  static constexpr int kThreads = CM > 32 ? 512 : 256, kPerSM = 512 / kThreads;
  static constexpr int W = 2 * CM, R = 2 * W, P = RM * R;   // half-row, row, a component's plane
  static constexpr size_t kSmem = (size_t)2 * 3 * P * sizeof(float);
};
constexpr int kJ2MinN = 40, kJ2MaxN = 256;
// A level takes the pairs where its fields (d, t, r, q: 40 B a cell) are more than
// L2 keeps between sweeps: 84 MB (128^3) took 21.2 against 19.4 us, 92 MB (132^3)
// 29.8 against 33.1; and from rows of ten threads on: 80 x 32^3 41 against 35.
constexpr int64_t kJ2MinBytes = 86 << 20;

// ZERO: d = 0 on entry (nothing is read from d).  AHEAD: planes that are fetched
// into L2 before they are used (0: none).  A variant that added its result to the
// state u, as k_lin_jacobi32m does, took 326 us at 256^3 against 105 and 219 for
// the two sweeps alone, and 241 against 217 at 42 x 64^3.
template <int CM, int RM, bool ZERO, int AHEAD>
__global__ void __launch_bounds__(J2<CM, RM>::kThreads, J2<CM, RM>::kPerSM) k_lin_jacobi2x32(
    LvlF L, float w, int rows, int zc, const float* __restrict__ d1,
    const float* __restrict__ d2, const float* __restrict__ d3, float* __restrict__ t1,
    float* __restrict__ t2, float* __restrict__ t3, const float* __restrict__ r1,
    const float* __restrict__ r2, const float* __restrict__ r3, const float* __restrict__ q) {
  constexpr int W = J2<CM, RM>::W, R = J2<CM, RM>::R, P = J2<CM, RM>::P;
  pdl_wait();
  extern __shared__ float j2s[];
  const int n = L.n, half = n >> 1, nn = n * n, cols = n >> 2;
  const int cy = threadIdx.x / cols, cx = threadIdx.x - cy * cols, p = 2 * cx;
  const bool on = cy < rows;
  int zb = blockIdx.z;
  const int m = member_of(zb, (n + zc - 1) / zc);
  const int k0 = zb * zc, k1 = min(n, k0 + zc);
  const int j0 = blockIdx.y * (rows - 2) - 1;               // row of the first row of threads
  const int j = (j0 + cy + n) % n;
  const bool own = on && cy >= 1 && cy < rows - 1 && j0 + cy < n;
  const size_t moff = (size_t)m * nn * n;
  // offsets in a plane of the source (without the colour's half-row) and of v
  const int c = j * n + p;
  const int ym = (j == 0 ? n - 1 : j - 1) * n + p, yp = (j + 1 == n ? 0 : j + 1) * n + p;
  const int xl = j * n + (p == 0 ? half - 1 : p - 1), xr = j * n + (p + 2 >= half ? 0 : p + 2);
  const int sc = cy * R + p;
  const int sl = p == 0 ? sc + half - 1 : sc - 1, sr = p + 2 >= half ? sc - p : sc + 2;
  const float* const d[3] = {d1 + moff, d2 + moff, d3 + moff};
  const float* const rq[4] = {r1 + moff, r2 + moff, r3 + moff, q + moff};
  float* const t[3] = {t1 + moff, t2 + moff, t3 + moff};

  // one array's range of a plane of the tile per thread (the part inside the
  // plane's ends, 16-byte granular as n is a multiple of 4)
  const int ja = max(0, j0), jb = min(n, j0 + rows);
  const float* range = nullptr;
  if (AHEAD > 0 && threadIdx.x < (ZERO ? 4 : 7)) {
    const int a = threadIdx.x;
    range = (a == 0   ? r1
             : a == 1 ? r2
             : a == 2 ? r3
             : a == 3 ? q
             : a == 4 ? d1
             : a == 5 ? d2
                      : d3) +
            moff + (size_t)ja * n;
  }
  auto fetch = [&](int k) {                                 // planes up to k1 + 1 are used
    if (AHEAD > 0 && range && k <= k1 + 1)
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(
                       range + (size_t)(k >= n ? k - n : k) * nn),
                   "r"((unsigned)((jb - ja) * n * sizeof(float)))
                   : "memory");
  };

  const float2 ww = f2_all(w), z2 = f2_all(0.f);
  float2 am[3][2], ac[3][2], vm[3][2], vc[3][2];            // d and v: plane below, plane
  const int ka = k0 == 0 ? n - 1 : k0 - 1, kb = ka == 0 ? n - 1 : ka - 1;
#pragma unroll
  for (int f = 0; f < 3; ++f)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      vm[f][h] = vc[f][h] = z2;
      am[f][h] = ZERO ? z2 : ldg2(d[f] + (size_t)kb * nn + h * half + c);
      ac[f][h] = ZERO ? z2 : ldg2(d[f] + (size_t)ka * nn + h * half + c);
    }
  float* vb = j2s;                                          // v of plane k, of plane k - 1
  float* vp = j2s + 3 * P;
  int kw = ka, kl = 0;                                      // planes k and k - 1, wrapped
#pragma unroll 1
  for (int k = k0 - 1; k <= k1; ++k) {
    const int kn = kw + 1 == n ? 0 : kw + 1;
    const size_t g = (size_t)kw * nn, gp = (size_t)kn * nn, gl = (size_t)kl * nn;
    const bool sg = (j + kw) & 1;                           // of colour 0; colour 1 has the other
    fetch(k + AHEAD);
    // first sweep, plane k
    float2 v[3][2], ap[3][2];
    {
      float2 s[4][2], sum[3][2];
#pragma unroll
      for (int f = 0; f < 4; ++f)
#pragma unroll
        for (int h = 0; h < 2; ++h) s[f][h] = ldg2(rq[f] + g + h * half + c);
#pragma unroll
      for (int f = 0; f < 3; ++f) {
#pragma unroll
        for (int h = 0; h < 2; ++h) ap[f][h] = ZERO ? z2 : ldg2(d[f] + gp + h * half + c);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const bool o1 = sg != (h != 0);
          const float* const o = d[f] + g + (1 - h) * half;
          sum[f][h] = ZERO ? z2
                           : nbsum2(ac[f][1 - h], __ldg(o + (o1 ? xr : xl)), o1, ldg2(o + ym),
                                    ldg2(o + yp), am[f][1 - h], ap[f][1 - h]);
        }
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float2 x[3];
        lin_point2(L, sum[0][h], sum[1][h], sum[2][h], s[3][h], s[0][h], s[1][h], s[2][h], x[0],
                   x[1], x[2]);
#pragma unroll
        for (int f = 0; f < 3; ++f) {
          v[f][h] = f2_fma(ww, f2_sub(x[f], ac[f][h]), ac[f][h]);
          if (on) *reinterpret_cast<float2*>(vb + f * P + h * W + sc) = v[f][h];
        }
      }
    }
    // second sweep, plane k - 1
    if (own && k > k0) {
      float2 s[4][2], sum[3][2];
#pragma unroll
      for (int f = 0; f < 4; ++f)
#pragma unroll
        for (int h = 0; h < 2; ++h) s[f][h] = ldg2(rq[f] + gl + h * half + c);
#pragma unroll
      for (int f = 0; f < 3; ++f)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const bool o1 = sg == (h != 0);                   // the offsets of plane k - 1
          const float* const o = vp + f * P + (1 - h) * W;
          sum[f][h] = nbsum2(vc[f][1 - h], o[o1 ? sr : sl], o1,
                             *reinterpret_cast<const float2*>(o + sc - R),
                             *reinterpret_cast<const float2*>(o + sc + R), vm[f][1 - h],
                             v[f][1 - h]);
        }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float2 x[3];
        lin_point2(L, sum[0][h], sum[1][h], sum[2][h], s[3][h], s[0][h], s[1][h], s[2][h], x[0],
                   x[1], x[2]);
#pragma unroll
        for (int f = 0; f < 3; ++f)
          *reinterpret_cast<float2*>(t[f] + gl + h * half + c) =
              f2_fma(ww, f2_sub(x[f], vc[f][h]), vc[f][h]);
      }
    }
#pragma unroll
    for (int f = 0; f < 3; ++f)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        am[f][h] = ac[f][h];
        ac[f][h] = ap[f][h];
        vm[f][h] = vc[f][h];
        vc[f][h] = v[f][h];
      }
    float* const x = vb;
    vb = vp;
    vp = x;
    kl = kw;
    kw = kn;
    __syncthreads();            // v of plane k is there, that of plane k - 1 has been read
  }
}

// Rows of threads and planes of a block: as many rows as its threads hold, evenly
// split, and the chunks of planes with the fewest waves of resident blocks times
// the planes of a block (two more than it owns).
struct J2Tile {
  int rows, zc;
  dim3 grid;
};

template <class T>
J2Tile jacobi2_tile(int n, int members, int rows_max) {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
    sms = 152;
  const int cols = n / 4;
  int rows = T::kThreads / cols;
  if (rows > rows_max) rows = rows_max;
  const int tiles = (n + rows - 3) / (rows - 2), slots = sms * T::kPerSM;
  J2Tile b;
  b.rows = (n + tiles - 1) / tiles + 2;
  b.zc = n;
  int64_t best = INT64_MAX;
  for (int chunks = 1; chunks <= n && (int64_t)chunks * members <= 65535; ++chunks) {
    const int zc = (n + chunks - 1) / chunks;
    if ((n + zc - 1) / zc != chunks) continue;              // the split of a smaller count
    const int64_t blocks = (int64_t)tiles * chunks * members;
    const int64_t cost = (blocks + slots - 1) / slots * (zc + 2);
    if (cost < best) {
      best = cost;
      b.zc = zc;
    }
  }
  b.grid = dim3(1, tiles, (n + b.zc - 1) / b.zc * members);
  return b;
}

// Two sweeps d -> t.
template <int CM, int RM, bool ZERO, int AHEAD>
cudaError_t launch_jacobi2_on(const LvlF& L, float w, float* const* d, float* const* t,
                              float* const* r, const float* q, cudaStream_t st, bool pdl, int nb) {
  using T = J2<CM, RM>;
  const J2Tile b = jacobi2_tile<T>(L.n, nb, RM);
  const auto k = k_lin_jacobi2x32<CM, RM, ZERO, AHEAD>;
  const cudaError_t e =
      cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)T::kSmem);
  if (e != cudaSuccess) return e;
  return launch_k(pdl, k, b.grid, dim3((L.n / 4 * b.rows + 31) / 32 * 32), T::kSmem, st, L, w,
                  b.rows, b.zc, d[0], d[1], d[2], t[0], t[1], t[2], r[0], r[1],
                  r[2], q);
}

template <bool ZERO>
cudaError_t launch_jacobi2(const LvlF& L, float w, float* const* d, float* const* t,
                           float* const* r, const float* q, cudaStream_t st, bool pdl, int nb) {
  return L.n <= 64   ? launch_jacobi2_on<16, 24, ZERO, 0>(L, w, d, t, r, q, st, pdl, nb)
         : L.n <= 96 ? launch_jacobi2_on<32, 16, ZERO, 0>(L, w, d, t, r, q, st, pdl, nb)
                     : launch_jacobi2_on<64, 16, ZERO, 2>(L, w, d, t, r, q, st, pdl, nb);
}

// Whether a level's sweeps go in pairs: whole rows in a block, fields larger than
// L2 holds, and 16-byte boundaries for the fetches ahead.
bool jacobi2_pays(int n, int nb, float* const* d, float* const* t, float* const* r,
                  const float* q) {
  if (n % 4 != 0 || n < kJ2MinN || n > kJ2MaxN || (int64_t)40 * n * n * n * nb <= kJ2MinBytes)
    return false;
  uintptr_t bits = (uintptr_t)q;
  for (int f = 0; f < 3; ++f) bits |= (uintptr_t)d[f] | (uintptr_t)t[f] | (uintptr_t)r[f];
  return bits % 16 == 0;
}

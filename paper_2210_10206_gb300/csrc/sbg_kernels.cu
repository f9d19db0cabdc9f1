// Preprocessing, kernel generation, 3PCF Gram, FP32 SIMT 4PCF contraction and
// FP64 finalisation kernels.
#include <algorithm>

#include "sbg_kernels.cuh"
#include "sbg_tcgen05.cuh"

namespace sbg {

// ------------------------------------------------------------------ reduce --
__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ void block_add_d(double v, double* dst) {
  __shared__ double part[32];
  v = warp_sum_d(v);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) part[w] = v;
  __syncthreads();
  if (w == 0) {
    v = lane < (int)(blockDim.x >> 5) ? part[lane] : 0.0;
    v = warp_sum_d(v);
    if (lane == 0) atomicAdd(dst, v);
  }
}

// field f = blockIdx.y of a slab: its n values start at f * n; acc[2f] collects
// the sum and acc[2f + 1] N_gal
__global__ void sum_kernel(const void* in, int is_f64, long long n, double* acc) {
  const long long f0 = (long long)blockIdx.y * n;
  double s = 0.0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    s += is_f64 ? reinterpret_cast<const double*>(in)[f0 + i] : (double)reinterpret_cast<const float*>(in)[f0 + i];
  block_add_d(s, acc + 2 * blockIdx.y);
}

__global__ void convert_kernel(const void* in, int is_f64, long long n, const double* acc, int subtract,
                               float* out, double* ngal) {
  const long long f0 = (long long)blockIdx.y * n;
  const double mean = subtract ? acc[2 * blockIdx.y] / (double)n : 0.0;
  double s = 0.0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    double v = is_f64 ? reinterpret_cast<const double*>(in)[f0 + i] : (double)reinterpret_cast<const float*>(in)[f0 + i];
    v -= mean;
    out[f0 + i] = (float)v;
    s += v + 1.0;
  }
  block_add_d(s, ngal + 2 * blockIdx.y);
}

static int grid_for(long long n, int threads) {
  long long b = (n + threads - 1) / threads;
  const long long cap = (long long)device_sms() * 16;
  if (b > cap) b = cap;
  return (int)(b < 1 ? 1 : b);
}

// CTAs per field of a slab of nfld fields: the single-field grid, shared out
static dim3 grid_fields(long long n, int nfld) {
  long long b = grid_for(n, 256);
  if (nfld > 1) b = std::max<long long>(1, std::min<long long>(b, ((long long)device_sms() * 16 + nfld - 1) / nfld));
  return dim3((unsigned)b, (unsigned)nfld);
}

cudaError_t launch_sum(const void* in, int is_f64, long long n, double* acc, cudaStream_t st, int nfld) {
  if (nfld < 1 || nfld > 65535) return cudaErrorInvalidValue;
  sum_kernel<<<grid_fields(n, nfld), 256, 0, st>>>(in, is_f64, n, acc);
  return cudaGetLastError();
}

cudaError_t launch_convert(const void* in, int is_f64, long long n, const double* acc, int subtract, float* out,
                           cudaStream_t st, int nfld) {
  if (nfld < 1 || nfld > 65535) return cudaErrorInvalidValue;
  convert_kernel<<<grid_fields(n, nfld), 256, 0, st>>>(in, is_f64, n, acc, subtract, out,
                                                        const_cast<double*>(acc) + 1);
  return cudaGetLastError();
}

// ---------------------------------------------------------- kernel generation --
__device__ __forceinline__ int min_image(int i, int n) { return i < n - i ? i : i - n; }

__device__ __forceinline__ int find_bin(double r2, const double* e2, int nb) {
  if (!(r2 > e2[0]) || r2 > e2[nb]) return -1;
  int b = 0;
  while (b < nb - 1 && r2 > e2[b + 1]) ++b;
  return b;
}

// conj(Y_lm) * Theta_b on the minimum-image offset grid (Algorithm 1); Y_lm from the
// reduced associated Legendre recurrence times ((x + i y)/r)^m, in FP64.
__global__ void kgen3d_kernel(int n, int l, int m, double norm, const double* __restrict__ e2, int nb, double scale,
                              float2* __restrict__ out) {
  const long long ng = (long long)n * n * n;
  const long long cell = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (cell >= ng) return;
  const int ix = (int)(cell % n), iy = (int)((cell / n) % n), iz = (int)(cell / ((long long)n * n));
  const int x = min_image(ix, n), y = min_image(iy, n), z = min_image(iz, n);
  const double r2 = (double)x * x + (double)y * y + (double)z * z;
  const int b = find_bin(r2, e2, nb);
  if (b < 0) return;
  const double r = sqrt(r2);
  const double t = z / r;
  // reduced associated Legendre (-1)^m d^m P_l/dt^m
  double pmm = (m & 1) ? -1.0 : 1.0;
  for (int k = 1; k < 2 * m; k += 2) pmm *= k;
  double p = pmm;
  if (l > m) {
    double a = pmm, bb = (2 * m + 1) * t * pmm;
    for (int ll = m + 2; ll <= l; ++ll) {
      double c = ((2 * ll - 1) * t * bb - (ll + m - 1) * a) / (ll - m);
      a = bb;
      bb = c;
    }
    p = bb;
  }
  double ur = x / r, ui = y / r, er = 1.0, ei = 0.0;
  for (int k = 0; k < m; ++k) {
    const double tr = er * ur - ei * ui;
    ei = er * ui + ei * ur;
    er = tr;
  }
  const double s = norm * p * scale;
  out[(long long)b * ng + cell] = make_float2((float)(s * er), (float)(-s * ei));
}

// conj(((x + i y)/rho)^m) * Theta_b (Algorithm 2) for m = m0 + blockIdx.y, every
// bin's array written in full (zeros outside the bin)
__global__ void kgen2d_kernel(int n, int m0, const double* __restrict__ e2, int nb, double scale,
                              float2* __restrict__ out) {
  const long long ng = (long long)n * n;
  const long long cell = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (cell >= ng) return;
  const int m = m0 + blockIdx.y;
  out += (long long)blockIdx.y * nb * ng;
  const int x = min_image((int)(cell % n), n), y = min_image((int)(cell / n), n);
  const double r2 = (double)x * x + (double)y * y;
  const int b = find_bin(r2, e2, nb);
  float2 v = make_float2(0.f, 0.f);
  if (b >= 0) {
    const double r = sqrt(r2);
    double ur = x / r, ui = y / r, er = 1.0, ei = 0.0;
    for (int k = 0; k < m; ++k) {
      const double tr = er * ur - ei * ui;
      ei = er * ui + ei * ur;
      er = tr;
    }
    v = make_float2((float)(er * scale), (float)(-ei * scale));
  }
  for (int k = 0; k < nb; ++k) out[(long long)k * ng + cell] = k == b ? v : make_float2(0.f, 0.f);
}

cudaError_t launch_kgen3d(int n, int l, int m, double norm_lm, const double* e2_dev, int nb, double scale,
                          float2* out, cudaStream_t st) {
  const long long ng = (long long)n * n * n;
  kgen3d_kernel<<<(unsigned)((ng + 255) / 256), 256, 0, st>>>(n, l, m, norm_lm, e2_dev, nb, scale, out);
  return cudaGetLastError();
}

cudaError_t launch_kgen2d(int n, int m0, int nm, const double* e2_dev, int nb, double scale, float2* out,
                          cudaStream_t st) {
  const long long ng = (long long)n * n;
  if (nm < 1 || nm > 65535) return cudaErrorInvalidValue;
  kgen2d_kernel<<<dim3((unsigned)((ng + 255) / 256), (unsigned)nm), 256, 0, st>>>(n, m0, e2_dev, nb, scale, out);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ gram3 --
// S[b1][b2] += sum_x delta(x) a_b1(x) conj(a_b2(x)) for b1 <= b2 (Algorithm 5's
// delta-weighted products of the coefficients, Eq. zeta3 of Sec. 2.2).  One CTA
// sweeps a contiguous x-range in chunks of 128 points, staged in shared memory
// by cp.async through a ring of kGramStages chunks (three in flight while one
// is summed).  The bins (at most 20) form blocks of 4; warp w owns block pair
// w (I <= J; at most 15) and its lanes take every 32nd point, so each lane
// holds a 4 x 4 tile of pair sums (16 complex, FP32 with packed f32x2 FMAs: 8
// operand loads per 16 products).  Every kGramFlush chunks a warp reduce-scatter hands
// lane k the warp's total of tile element k, which it adds to an FP64
// register; at the end each lane adds its element to S (FP64 atomics).
constexpr int kGramChunk = 128;
constexpr int kGramMaxNb = 20;
constexpr int kGramFlush = 4;   // chunks (16 points per lane) between FP64 flushes
constexpr int kGramStages = 4;  // ring of staged chunks

__device__ __forceinline__ void gram_cp(void* dst, const void* src, bool ok, int bytes) {
  // bytes 4 / 8 / 16; a copy outside the range reads nothing and writes zeros
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  const int n = ok ? bytes : 0;
  if (bytes == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(n) : "memory");
  else if (bytes == 8)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d), "l"(src), "r"(n) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(n) : "memory");
}

__global__ void __launch_bounds__(512, 2) gram3_kernel(const float2* __restrict__ a, long long ng, int nb,
                                                    const float* __restrict__ delta, double* __restrict__ S,
                                                    int nsingle, int single0, long long s_stride) {
  // field f = blockIdx.y of a slab: its arrays follow field f - 1's (group
  // buffer) or its points do (blocked store); its delta and S likewise.  Group
  // blockIdx.z: the next nb arrays or singles, and the next S block
  const long long fx = (long long)blockIdx.y * ng;
  if (!nsingle) a += ((long long)blockIdx.y * gridDim.z + blockIdx.z) * nb * ng;
  single0 += blockIdx.z * nb;
  delta += fx;
  S += (long long)blockIdx.y * s_stride + (long long)blockIdx.z * nb * nb * 2;
  const int nbb = (nb + 3) / 4, nrow = 4 * nbb;
  // stage: nrow rows of kGramChunk (re, im), then kGramChunk deltas; rows nb ..
  // of the last block stay zero
  extern __shared__ __align__(16) uint8_t gsm[];
  const int stage_bytes = nrow * kGramChunk * 8 + kGramChunk * 4;
  auto srow = [&](int st, int b) { return reinterpret_cast<float2*>(gsm + st * stage_bytes) + b * kGramChunk; };
  auto sdel = [&](int st) { return reinterpret_cast<float*>(gsm + st * stage_bytes + nrow * kGramChunk * 8); };
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // x-ranges of whole chunks: x0 and x1 are multiples of 4 (ng is), so the
  // 16-byte copies below never straddle x1
  const long long per = ((ng + gridDim.x - 1) / gridDim.x + kGramChunk - 1) / kGramChunk * kGramChunk;
  const long long x0 = blockIdx.x * per, x1 = min(ng, x0 + per);
  const int nch = x0 < x1 ? (int)((x1 - x0 + kGramChunk - 1) / kGramChunk) : 0;
  for (int i = threadIdx.x; i < kGramStages * (nrow - nb) * kGramChunk; i += blockDim.x) {
    const int st = i / ((nrow - nb) * kGramChunk), r = i % ((nrow - nb) * kGramChunk);
    srow(st, nb + r / kGramChunk)[r % kGramChunk] = make_float2(0.f, 0.f);
  }
  // this warp's block pair (none for warps past the last one)
  int bI = -1, bJ = -1;
  for (int i = 0, q = warp; i < nbb && q >= 0; ++i) {
    if (q < nbb - i) {
      bI = i;
      bJ = i + q;
    }
    q -= nbb - i;
  }
  // copies of chunk c into stage c % kGramStages, one commit group per chunk
  auto issue = [&](int c) {
    if (c < nch) {
      const int st = c % kGramStages;
      const long long xc = x0 + (long long)c * kGramChunk;
      if (nsingle) {
        // blocked store: per 32-point block 32 Re then 32 Im floats of a single
        for (int i = threadIdx.x; i < nb * kGramChunk; i += blockDim.x) {
          const int b = i / kGramChunk, xx = i % kGramChunk;
          const long long x = xc + xx;
          const bool ok = x < x1;
          const float* f = reinterpret_cast<const float*>(a) + blocked_re(fx + (ok ? x : x0), single0 + b, nsingle);
          float2* dst = srow(st, b) + xx;
          gram_cp(&dst->x, f, ok, 4);
          gram_cp(&dst->y, f + 32, ok, 4);
        }
      } else {
        // group buffer: bins of ng complex, two points per 16-byte copy
        for (int i = threadIdx.x; i < nb * kGramChunk / 2; i += blockDim.x) {
          const int b = i / (kGramChunk / 2), xx = 2 * (i % (kGramChunk / 2));
          const long long x = xc + xx;  // even, and x1 is a multiple of 4
          const bool ok = x < x1;
          gram_cp(srow(st, b) + xx, a + (long long)b * ng + (ok ? x : x0), ok, 16);
        }
      }
      for (int i = threadIdx.x; i < kGramChunk / 4; i += blockDim.x) {
        const long long x = xc + 4 * i;
        const bool ok = x < x1;
        gram_cp(sdel(st) + 4 * i, delta + (ok ? x : x0), ok, 16);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  uint64_t acc[16];
  double dacc = 0.0;
#pragma unroll
  for (int e = 0; e < 16; ++e) acc[e] = 0ull;
  // lane k of the warp gets the warp's total of element k of the 32 floats
  auto flush = [&]() {
    float v[32];
#pragma unroll
    for (int e = 0; e < 16; ++e) {
      upk(acc[e], v[2 * e], v[2 * e + 1]);
      acc[e] = 0ull;
    }
#pragma unroll
    for (int lv = 0; lv < 5; ++lv) {
      const int o = 16 >> lv;
      const bool up = (lane & o) != 0;
#pragma unroll
      for (int e = 0; e < o; ++e) {
        const float send = up ? v[e] : v[e + o];
        const float keep = up ? v[e + o] : v[e];
        v[e] = keep + __shfl_xor_sync(0xffffffffu, send, o);
      }
    }
    dacc += (double)v[0];
  };
  __syncthreads();  // zero rows written
#pragma unroll
  for (int c = 0; c < kGramStages - 1; ++c) issue(c);
  int nflush = 0;
  for (int c = 0; c < nch; ++c) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kGramStages - 2) : "memory");
    __syncthreads();  // chunk c landed for every thread; chunk c - 1 has been summed
    issue(c + kGramStages - 1);
    const int st = c % kGramStages;
    const float* sd = sdel(st);
    if (bI >= 0) {
      const float2* s1 = srow(st, 4 * bI);
      const float2* s2 = srow(st, 4 * bJ);
#pragma unroll 2
      for (int m = 0; m < kGramChunk / 32; ++m) {
        const int xx = lane + 32 * m;
        const float d = sd[xx];
        const uint64_t dd = pk(d, d);
        uint64_t w[4], wr[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float2 u = s1[i * kGramChunk + xx];
          w[i] = mul2(pk(u.x, u.y), dd);    // delta u
          wr[i] = mul2(pk(u.y, -u.x), dd);  // delta (Im u, -Re u)
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float2 v = s2[j * kGramChunk + xx];
          const uint64_t vr = pk(v.x, v.x), vi = pk(v.y, v.y);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            // (Re, Im) of delta u conj(v) = w Re v + (Im w, -Re w) Im v
            acc[4 * i + j] = fma2(w[i], vr, acc[4 * i + j]);
            acc[4 * i + j] = fma2(wr[i], vi, acc[4 * i + j]);
          }
        }
      }
    }
    if (++nflush == kGramFlush) {
      flush();
      nflush = 0;
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  if (nflush) flush();
  if (bI >= 0) {
    // lane = 2 (4 i + j) + component
    const int e = lane >> 1, c = lane & 1, i = e >> 2, j = e & 3;
    const int b1 = 4 * bI + i, b2 = 4 * bJ + j;
    if (b1 <= b2 && b2 < nb) atomicAdd(&S[((long long)b1 * nb + b2) * 2 + c], dacc);
  }
}

cudaError_t launch_gram3(const float2* a, long long ng, int nb, const float* delta, double* S, int nsingle,
                         int single0, cudaStream_t st, int nfld, long long s_stride, int ngrp) {
  if (nb < 1 || nb > kGramMaxNb || nfld < 1 || nfld > 65535 || ngrp < 1 || ngrp > 65535) return cudaErrorInvalidValue;
  // 16-byte copies of the group buffer and of delta
  if (!nsingle && (((uintptr_t)a & 15) || (ng & 1))) return cudaErrorInvalidValue;
  if (((uintptr_t)delta & 15) || (ng & 3)) return cudaErrorInvalidValue;
  const int nbb = (nb + 3) / 4, nbp = nbb * (nbb + 1) / 2;
  const int threads = std::max(32 * nbp, 128);  // a warp per block pair, at least 4 to stage
  const int smem = kGramStages * (4 * nbb * kGramChunk * 8 + kGramChunk * 4);
  // the attribute is set once per device: to the largest stage ring
  constexpr int kMaxSmem = kGramStages * (4 * ((kGramMaxNb + 3) / 4) * kGramChunk * 8 + kGramChunk * 4);
  cudaError_t e = ensure_smem_attr<gram3_kernel>(kMaxSmem);
  if (e != cudaSuccess) return e;
  // chunks per CTA: about 4 on small grids; on large ones as many CTAs as fit
  long long blocks = (ng + 4 * kGramChunk - 1) / (4 * kGramChunk);
  int per_sm = 1;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, gram3_kernel, threads, smem)) != cudaSuccess) return e;
  const long long cap = std::max<long long>(1, ((long long)device_sms() * std::max(per_sm, 1) + nfld - 1) / nfld);
  if (blocks > cap) blocks = cap;
  gram3_kernel<<<dim3((unsigned)blocks, nfld, ngrp), threads, smem, st>>>(a, ng, nb, delta, S, nsingle, single0, s_stride);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ simt4 --
// T[r][c] = sum_x delta(x) f1_r(x) f2_r(x) a_c(x): the pair-by-single contraction
// of the 4PCF (Eq. mu of Sec. 2.3, Eq. proj_4pcf_coeff) as an FP32 SIMT GEMM over
// x with the pair operand formed on chip.
//
// Bound: the FMA pipe (2 FMAs per entry and point, 4 for complex T) and, in narrow
// tiles, the shared-memory pipe.  Each thread holds 8 rows x 8 or 4 columns, so a
// point costs it 8 or 6 16-byte shared-memory loads for 128 or 64 FMAs (complex T:
// 128; 4 x 4 in narrow tiles).  The FMAs are packed (f32x2, two pipe cycles each),
// which leaves about half of the issue slots to the loads and to forming the
// operands.  A packed FMA multiplies two rows by two columns; with the column pair
// once straight and once swapped in registers it serves the four entries of a 2 x 2
// block, and no operand has to be duplicated.  Per chunk of 8 points (complex T 16)
// the tile's row singles, its columns and delta are copied with cp.async while the
// previous chunk is accumulated, then formed in shared memory as [x][row] and
// [x][column] arrays.  Three to seven CTAs per SM overlap one's forming with
// another's FMAs.  The output takes about half of a 3D block's entries (the l3 of
// one parity), so a tile has few columns (a few l3 of every bin) and up to 256 rows.
// Accumulation: FP32 over a span (at most 512 points), then one FP64 reduction
// into T (red.add, fire and forget; T is laid out [accumulator][thread], so a
// warp's 32 values are contiguous): no FP64 add, whose rate is 1/75 of the FMA
// rate here, occupies the SM.
// Measured: 256^3, lmax 4, 10 bins: 686 -> 176 ms per field (268 with every column
// of a block for each of its rows); 128^3, lmax 3, 8 bins 20.1 -> 5.4 ms (8.0); 1024^2,
// mmax 5, 20 bins 41.4 -> 14.9 ms; 37 slices of 256^2, mmax 5, 5 bins 1.93 -> 1.72 ms
// with 4 x 4 for complex T; against the earlier 4 x 4 entries per thread with
// two 256-thread CTAs per SM, whose strided float4 loads conflicted in the banks.
// In tiles of 8 x 4 the shared-memory pipe is 81% busy, the FMA pipe 56%, issue 56%
// (8 x 8: 54%, 62%, 48%; 128^3, lmax 4, 10 bins).
constexpr int kSpanX = 512;     // points per FP32 span
constexpr int simt_threads(int rt) { return rt == 4 ? 256 : 128; }
constexpr int simt_x(bool cplx) { return cplx ? 16 : 8; }  // points per chunk
// most rows of a tile and most columns (complex T: 2D, one column per bin)
constexpr int simt_rows(bool cplx) { return cplx ? 192 : 256; }
constexpr int simt_cols(int ct, bool cplx) { return cplx ? 20 : ct == 4 ? 24 : 64; }
// floats per raw row: Re, Im of a chunk's points, pad (an odd number of 16-byte units: no bank conflicts)
constexpr int simt_raw(int x) { return 2 * x + 4; }

__device__ __forceinline__ void simt_cp16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ uint64_t swap2(uint64_t v) {
  float a, b;
  upk(v, a, b);
  return pk(b, a);
}
__device__ __forceinline__ uint64_t neg2(uint64_t v) { return v ^ 0x8000000080000000ull; }
// sign bits of both halves where b & 1
__device__ __forceinline__ uint64_t sign2(int b) {
  const uint32_t m = (uint32_t)b << 31;
  return (uint64_t)m << 32 | m;
}
__device__ __forceinline__ void red_add(double* p, float v) {
  asm volatile("red.global.add.f64 [%0], %1;" ::"l"(p), "d"((double)v) : "memory");
}

// Spans of one column class: x-split k covers the points [k per, (k + 1) per) and
// consists of nsp spans of kSpanX points (the last one shorter or empty).
struct SimtSpans {
  int nsplit, nsp;   // x-splits, spans per x-split
  long long per;     // points per x-split
  int unit;          // spans per CTA
};
struct SimtArgs {
  const float* astore;
  const float* delta;
  const Tile4* tiles;
  const Row4* rows;
  const int *cols, *uniq;
  double* T;
  long long ng, t_field_stride;
  int nsingle, imag;
  int spf[3];        // x-splits per field of a slab (0: one field)
  SimtSpans sp[3];
};

// Row and column group of a tile's thread.  A 16-byte shared load of a warp takes
// two cycles if lanes l and l ^ 1 read one address throughout, or l and l ^ 2,
// and four otherwise, however few addresses there are (measured: lane / 2, lane %
// 2 and lane / 4 2.1 cycles, lane / 5 and lane % 4 4.0).  So four lanes take two row
// groups by two column groups: the row operand is shared by l and l ^ 2, the
// column operand by l and l ^ 1.  What an odd count leaves over comes last.
__host__ __device__ __forceinline__ void simt_position(int t, int nrg, int ncg, int& rg, int& cg) {
  const int pc = ncg >> 1, quads = (nrg >> 1) * pc;
  if (t < 4 * quads) {
    const int q = t >> 2, rp = q / pc;
    rg = 2 * rp + (t & 1);
    cg = 2 * (q - rp * pc) + (t >> 1 & 1);
    return;
  }
  t -= 4 * quads;
  if (ncg & 1) {  // the last column group
    if (t < nrg) {
      rg = t;
      cg = ncg - 1;
      return;
    }
    t -= nrg;
  }
  rg = nrg - 1;  // the last row group
  cg = t;
}
// its inverse
inline int simt_thread(int rg, int cg, int nrg, int ncg) {
  const int pc = ncg >> 1, quads = (nrg >> 1) * pc;
  if (rg < (nrg & ~1) && cg < (ncg & ~1)) return 4 * ((rg >> 1) * pc + (cg >> 1)) + (rg & 1) + 2 * (cg & 1);
  if (cg >= (ncg & ~1)) return 4 * quads + rg;
  return 4 * quads + (ncg & 1 ? nrg : 0) + cg;
}

template <int RT, int CT, bool CPLX>
__global__ void __launch_bounds__(simt_threads(RT), CPLX ? 3 : CT == 8 ? 4 : 7) simt4_kernel(const SimtArgs p) {
  const Tile4 tl = p.tiles[blockIdx.x];
  const SimtSpans sp = p.sp[tl.cls];
  const int spf = p.spf[tl.cls];
  const int s0 = blockIdx.y * sp.unit, s1 = min(s0 + sp.unit, sp.nsplit * sp.nsp);
  extern __shared__ float4 smem4[];
  // row strides of the formed operands (compile-time: the accumulation's loads
  // and the forming's stores take immediate offsets)
  constexpr int kX = simt_x(CPLX), kRawF = simt_raw(kX), kP = kX / 2;  // kP: 16-byte pieces of a raw row
  constexpr int TRS = simt_rows(CPLX), TCS = simt_cols(CT, CPLX);
  const int nrg = tl.nrg, ncg = tl.ncg;
  const int TR = RT * nrg, TC = CT * ncg;
  float* Px = reinterpret_cast<float*>(smem4);   // [kX][TRS]
  float* Py = Px + kX * TRS;                     // real T: -Im P, complex T: Im P
  float* Cx = Py + kX * TRS;                     // [kX][TCS]
  float* Cy = Cx + kX * TCS;
  int2* meta = reinterpret_cast<int2*>(Cy + kX * TCS);      // [TRS], see below
  float* raw = reinterpret_cast<float*>(meta + TRS);        // [nuniq + ncols][kRawF], then delta [kX]
  float* rdel = raw + (tl.nuniq + tl.ncols) * kRawF;
  int* sidx = reinterpret_cast<int*>(rdel + kX);  // store index of each raw row
  const int tid = threadIdx.x, nt = blockDim.x;
  int rg, cg;
  simt_position(tid, nrg, ncg, rg, cg);
  const bool active = tid < nrg * ncg;
  const int nraw = tl.nuniq + tl.ncols;

  // the chunk's part (kX Re, kX Im) of the 32-point block of each single: thread
  // t copies piece t % kP of the raw rows t / kP, + nt / kP, ...
  const int sch = tid % kP;
  float* const sdst = raw + (tid / kP) * kRawF + sch * 4;
  const float* const ssrc = p.astore + (sch % (kP / 2)) * 4 + (sch / (kP / 2)) * 32;
  auto stage = [&](long long xc) {
    const float* base = ssrc + (xc >> 5) * (long long)p.nsingle * 64 + (xc & 31);
    float* dst = sdst;
    for (int row = tid / kP; row < nraw; row += nt / kP, dst += (nt / kP) * kRawF)
      simt_cp16(dst, base + (long long)sidx[row] * 64);
    if (tid < kX / 4) simt_cp16(rdel + tid * 4, p.delta + xc + tid * 4);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  // The staged chunk's operands, 8 points of a row or column per item.  meta
  // holds a row's raw offsets of its two singles and the sign bits of their
  // conjugations (the row's own sign is left to the couplings).  Rows and columns
  // past the tile's repeat its last ones and are never written out.
  auto form = [&]() {
    for (int i = tid; i < kX / 8 * TR; i += nt) {
      const int h = i >= TR ? 8 : 0, r = i >= TR ? i - TR : i;
      const int2 m = meta[r];
      const float* u1 = raw + (m.x & 0xffff) + h;
      const float* u2 = raw + (m.x >> 16) + h;
      const uint64_t s1 = sign2(m.y & 1), s2 = sign2(m.y >> 1);
      float* o = Px + h * TRS + r;
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const ulonglong2 ar = *(const ulonglong2*)(u1 + 4 * q), ai = *(const ulonglong2*)(u1 + kX + 4 * q);
        const ulonglong2 br = *(const ulonglong2*)(u2 + 4 * q), bi = *(const ulonglong2*)(u2 + kX + 4 * q);
        const ulonglong2 d = *(const ulonglong2*)(rdel + h + 4 * q);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const uint64_t a_r = e ? ar.y : ar.x, a_i = (e ? ai.y : ai.x) ^ s1, b_r = e ? br.y : br.x;
          const uint64_t b_i = (e ? bi.y : bi.x) ^ s2, dd = e ? d.y : d.x;
          const uint64_t pr = mul2(fma2(a_r, b_r, mul2(neg2(a_i), b_i)), dd);
          uint64_t pi = mul2(fma2(a_i, b_r, mul2(a_r, b_i)), dd);
          if (!CPLX) pi = neg2(pi);
          float v0, v1;
          upk(pr, v0, v1);
          o[(4 * q + 2 * e) * TRS] = v0;
          o[(4 * q + 2 * e + 1) * TRS] = v1;
          upk(pi, v0, v1);
          o[(kX + 4 * q + 2 * e) * TRS] = v0;  // Py
          o[(kX + 4 * q + 2 * e + 1) * TRS] = v1;
        }
      }
    }
    // columns: the last threads first, whose row items are the fewest
    for (int i = nt - 1 - tid; i < kX / 8 * TC; i += nt) {
      const int h = i >= TC ? 8 : 0, c = i >= TC ? i - TC : i;
      const float* a = raw + (tl.nuniq + min(c, tl.ncols - 1)) * kRawF + h;
      float* o = Cx + h * TCS + c;
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const float4 re = *(const float4*)(a + 4 * q), im = *(const float4*)(a + kX + 4 * q);
        const float vr[4] = {re.x, re.y, re.z, re.w}, vi[4] = {im.x, im.y, im.z, im.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          // imag: the column is (Im a, -Re a), so that the real sum gives Im(P a)
          o[(4 * q + e) * TCS] = p.imag ? vi[e] : vr[e];
          o[(kX + 4 * q + e) * TCS] = p.imag ? -vr[e] : vi[e];  // Cy
        }
      }
    }
  };

  // accumulators: [component][row pair][column pair][straight, swapped]; entry
  // (row 2 i + e, column 2 j + (e ^ w)) is lane e of acc[.][i][j][w]
  constexpr int NC = CPLX ? 2 : 1, NI = RT / 2, NJ = CT / 2;
  uint64_t acc[NC][NI][NJ][2];
  auto zero = [&]() {
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
      for (int i = 0; i < NI; ++i)
#pragma unroll
        for (int j = 0; j < NJ; ++j) acc[c][i][j][0] = acc[c][i][j][1] = 0ull;
  };
  auto accumulate = [&]() {
    const float* px = Px + rg * 4;
    const float* py = Py + rg * 4;
    const float* cx = Cx + cg * 4;
    const float* cy = Cy + cg * 4;
#pragma unroll 16
    for (int x = 0; x < kX; ++x) {
      uint64_t X[NI], Y[NI];
#pragma unroll
      for (int h = 0; h < RT / 4; ++h) {  // rows 4 rg .. + 3 of each section of 4 nrg rows
        const ulonglong2 vx = *(const ulonglong2*)(px + x * TRS + h * 4 * nrg);
        const ulonglong2 vy = *(const ulonglong2*)(py + x * TRS + h * 4 * nrg);
        X[2 * h] = vx.x; X[2 * h + 1] = vx.y;
        Y[2 * h] = vy.x; Y[2 * h + 1] = vy.y;
      }
#pragma unroll
      for (int h = 0; h < CT / 4; ++h) {
        const ulonglong2 vx = *(const ulonglong2*)(cx + x * TCS + h * 4 * ncg);
        const ulonglong2 vy = *(const ulonglong2*)(cy + x * TCS + h * 4 * ncg);
        const uint64_t u[2][2] = {{vx.x, swap2(vx.x)}, {vx.y, swap2(vx.y)}};
        const uint64_t v[2][2] = {{vy.x, swap2(vy.x)}, {vy.y, swap2(vy.y)}};
#pragma unroll
        for (int jj = 0; jj < 2; ++jj)
#pragma unroll
          for (int w = 0; w < 2; ++w) {
            const int j = 2 * h + jj;
#pragma unroll
            for (int i = 0; i < NI; ++i) {
              if constexpr (CPLX) {
                // Re += Px Cx - Py Cy, Im += Px Cy + Py Cx
                acc[0][i][j][w] = fma2(X[i], u[jj][w], fma2(Y[i], neg2(v[jj][w]), acc[0][i][j][w]));
                acc[NC - 1][i][j][w] = fma2(X[i], v[jj][w], fma2(Y[i], u[jj][w], acc[NC - 1][i][j][w]));
              } else {
                acc[0][i][j][w] = fma2(X[i], u[jj][w], fma2(Y[i], v[jj][w], acc[0][i][j][w]));
              }
            }
          }
      }
    }
  };
  // the span's sums to T, and back to zero
  auto flush = [&](int q) {
    double* t = p.T + (spf ? (long long)(q / sp.nsp / spf) * p.t_field_stride : 0LL);
#pragma unroll
    for (int i = 0; i < NI; ++i)
#pragma unroll
      for (int j = 0; j < NJ; ++j)
#pragma unroll
        for (int w = 0; w < 2; ++w)
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const int ri = 2 * i + e, cj = 2 * j + (e ^ w);
            const int r = (ri >> 2) * 4 * nrg + rg * 4 + (ri & 3);
            const int c = (cj >> 2) * 4 * ncg + cg * 4 + (cj & 3);
            if (r >= tl.nrows || c >= tl.ncols) continue;
            const long long k = tl.tout + (long long)((i * NJ + j) * 2 + w) * 2 * (nrg * ncg) + e * (nrg * ncg) + tid;
#pragma unroll
            for (int m = 0; m < NC; ++m) {
              float lo, hi;
              upk(acc[m][i][j][w], lo, hi);
              red_add(t + k * NC + m, e ? hi : lo);
            }
          }
    zero();
  };

  // the CTA's spans in turn; span q starts at x0 and has nc chunks (an empty one none)
  int q = s0, nc = 0;
  long long x0 = 0;
  auto next_span = [&]() {  // the first span from q on that holds points
    for (; q < s1; ++q) {
      const int k = q / sp.nsp;
      x0 = k * sp.per + (long long)(q - k * sp.nsp) * kSpanX;
      const long long left = min((k + 1) * sp.per, p.ng) - x0;
      nc = (int)min(left, (long long)kSpanX) / kX;
      if (left > 0) return true;
    }
    return false;
  };
  if (!next_span()) return;
  for (int i = tid; i < nraw; i += nt) sidx[i] = i < tl.nuniq ? p.uniq[tl.uniq0 + i] : p.cols[tl.col0 + i - tl.nuniq];
  for (int i = tid; i < TR; i += nt) {
    const Row4 rw = p.rows[tl.row0 + min(i, tl.nrows - 1)];
    meta[i] = make_int2(rw.u1 * kRawF | (rw.u2 * kRawF) << 16, rw.flags & 3);
  }
  __syncthreads();
  zero();
  stage(x0);
  for (int c = 0;;) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();  // the chunk has landed; the previous one's operands have been read
    form();
    __syncthreads();  // the operands are formed and the raw chunk has been read
    const int qd = q;
    const bool done = ++c == nc;  // the span ends with this chunk
    bool more = true;
    if (done) {
      ++q;
      c = 0;
      more = next_span();
    }
    if (more) stage(x0 + c * kX);
    if (active) {
      accumulate();
      if (done) flush(qd);
    }
    if (!more) break;
  }
}

namespace {
// shared memory of a tile
size_t simt_smem(int ct, bool cplx, int nuniq, int ncols) {
  const int x = simt_x(cplx), trs = simt_rows(cplx), tcs = simt_cols(ct, cplx);
  return ((size_t)(nuniq + ncols) * (simt_raw(x) + 1) + x + 2 * x * ((size_t)trs + tcs)) * 4 + (size_t)trs * 8;
}
constexpr int kSimtSmemMax = 75 * 1024;
}  // namespace

template <int RT, int CT, bool CPLX>
static cudaError_t simt4_t(SimtArgs a, const SimtPlan& pl, int k, int nsm, cudaStream_t st) {
  const size_t smem = pl.smem[k];
  const int threads = (pl.threads[k] + 31) / 32 * 32;
  if (smem > kSimtSmemMax || threads < 32 || threads > simt_threads(RT)) return cudaErrorInvalidValue;
  cudaError_t e = ensure_smem_attr<simt4_kernel<RT, CT, CPLX>>(kSimtSmemMax);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, simt4_kernel<RT, CT, CPLX>, threads, smem)) !=
      cudaSuccess)
    return e;
  // spans per CTA: about 8 CTAs per resident slot, so that the last wave costs
  // little; at least one span, at most 64
  const long long slots = (long long)nsm * std::max(per_sm, 1);
  int rows = 1;
  for (int c = 0; c < 3; ++c) {
    SimtSpans& sp = a.sp[c];
    const long long spans = (long long)sp.nsplit * sp.nsp;
    sp.unit = (int)std::max<long long>(1, std::min<long long>(64, spans * pl.ntiles[k] / (8 * slots)));
    sp.unit = (int)std::max<long long>(sp.unit, (spans + 65534) / 65535);
    if (pl.uses[k][c]) rows = std::max<int>(rows, (int)((spans + sp.unit - 1) / sp.unit));
  }
  a.tiles += pl.first[k];
  simt4_kernel<RT, CT, CPLX><<<dim3((unsigned)pl.ntiles[k], (unsigned)rows), threads, smem, st>>>(a);
  return cudaGetLastError();
}

SimtGeometry simt_geometry(int complex_t, int ncols) {
  SimtGeometry g;
  // Up to 24 columns (most 3D tiles: one or two l3 of each bin), 8 x 4 entries per
  // thread: 72 registers, so that seven CTAs of tiles of at most 256 rows fit an
  // SM, against four of 8 x 8 (or 16 x 4, which the next line lists), and their
  // warps are fuller.  128^3, ms: 8 bins, lmax 3 5.4 (6.5), 10 bins, lmax 4 22.0
  // (23.0), 5 bins, lmax 4 5.0 (5.5 with five CTAs).  Wider tiles are FMA bound
  // and take 8 x 8 (20 bins, lmax 2, tiles of 40 columns; with 8 x 4 up to 16
  // columns only 16.9 against 15.6, up to 32 15.6 but 22.5 for 10 bins).
  g.cplx = complex_t != 0;
  g.ct = g.cplx || ncols <= 24 ? 4 : 8;
  // Complex T: 4 x 4 entries per thread (80 registers instead of 160) where a tile
  // of 8 x 4 leaves most of its 128 threads idle or its SM short of warps.  512^2,
  // mmax 5, ms: 4 bins 0.26 -> 0.20, 8 0.47 -> 0.46, 12 1.00 both, 16 2.03 -> 1.98,
  // but 20 3.69 -> 4.04 (half as many FMAs per operand load).
  // The CTAs per SM cost spills: 4 x 4 complex 92 bytes at 80 registers, 8 x 4 36 at 72,
  // 8 x 8 8 at 128.  With two CTAs instead of three (118 registers, none spilt) the
  // complex tiles of 10 columns gain (256^2, 10 bins 0.240 -> 0.215 ms, 37 slices, 5
  // bins 1.72 -> 1.58) and those of 13 and 16 lose (512^2 1.43 -> 1.54, 1.98 -> 2.16);
  // with six instead of seven (80 registers, 20 bytes) 8 x 4 is 1% slower.
  g.rt = g.cplx && ncols <= 16 ? 4 : 8;
  g.launch = g.cplx ? g.rt == 8 : g.ct == 8;
  g.ncg = (ncols + g.ct - 1) / g.ct;
  // the most row groups that fill their warps well; max_uniq singles and
  // simt_rows() rows keep a tile's shared memory within the resident CTAs' share of an SM's
  const int most = std::min(simt_threads(g.rt) / g.ncg, simt_rows(g.cplx) / g.rt);
  auto fill = [&](int n) { return n * g.ncg / (double)((n * g.ncg + 31) / 32 * 32); };
  double best = 0.0;
  for (int n = (most + 1) / 2; n <= most; ++n) best = std::max(best, fill(n));
  int n = most;
  while (fill(n) < best - 0.06) --n;
  g.max_rows = g.rt * n;
  g.max_uniq = complex_t ? 96 : 128;
  return g;
}

long long simt_entry(const Tile4& t, const SimtGeometry& g, int r, int c) {
  const int pr = r % (4 * t.nrg), pc = c % (4 * t.ncg);  // within the section
  const int ri = r / (4 * t.nrg) * 4 + pr % 4, cj = c / (4 * t.ncg) * 4 + pc % 4;
  const int i = ri / 2, e = ri & 1, j = cj / 2, w = (cj & 1) ^ e;
  return t.tout + ((long long)((i * (g.ct / 2) + j) * 2 + w) * 2 + e) * (t.nrg * t.ncg) + simt_thread(pr / 4, pc / 4, t.nrg, t.ncg);
}

size_t simt_tile_smem(const Tile4& t, const SimtGeometry& g) {
  return simt_smem(g.ct, g.cplx, t.nuniq, t.ncols);
}

cudaError_t launch_simt4(const float2* astore, long long ng, const float* delta, const Tile4* tiles,
                         const SimtPlan& plan, const Row4* rows, const int* cols, const int* uniq, int complex_out,
                         int nsingle, double* T, int nsm, cudaStream_t st, int* launches, int nfld,
                         long long t_field_stride) {
  if (ng % 32 || complex_out < 0 || complex_out > 2 || nfld < 1 || (ng / nfld) % 32) return cudaErrorInvalidValue;
  SimtArgs a{};
  a.astore = (const float*)astore;
  a.delta = delta;
  a.tiles = tiles;
  a.rows = rows;
  a.cols = cols;
  a.uniq = uniq;
  a.T = T;
  a.ng = ng;
  a.nsingle = nsingle;
  a.imag = complex_out == 2 ? 1 : 0;  // real T holding Im(P a)
  a.t_field_stride = t_field_stride;
  // The x-splits of a column class: one field, as many as fill 2 .. 8 waves of
  // the units (span_tiles x split) best on 2 (complex T: 1) units per SM; a slab,
  // per field a power of two by the same measure.  They set where the FP32
  // spans begin, hence the rounding of every result, and nothing else: the
  // spans are dealt to CTAs in simt4_t, however many fit there.
  const long long slots = (long long)nsm * (complex_out == 1 ? 1 : 2), chunks = ng / 32;
  int spf[3] = {0, 0, 0};
  for (int c = 0; c < 3; ++c) {
    const long long nt = plan.span_tiles[c];
    long long ns = 1;
    double best = -1.0;
    if (nt && nfld > 1) {
      const long long fchunks = chunks / nfld;
      spf[c] = 1;
      for (long long k = 1; k <= fchunks && k <= 64; k *= 2) {
        const long long units = nt * nfld * k;
        if (units > 65535LL * nt) break;
        const double fill = (double)units / (double)(slots * ((units + slots - 1) / slots));
        if (fill > best + 1e-3) {
          best = fill;
          spf[c] = (int)k;
        }
        if (units >= 4 * slots) break;
      }
      ns = (long long)nfld * spf[c];
    } else if (nt) {
      for (int w = 2; w <= 8; ++w) {
        const long long n = std::max<long long>(1, std::min<long long>(chunks, slots * w / nt));
        const long long units = n * nt;
        const double fill = (double)units / (double)(slots * ((units + slots - 1) / slots));
        if (fill > best + 1e-3) {
          best = fill;
          ns = n;
        }
      }
    }
    SimtSpans& sp = a.sp[c];
    sp.nsplit = (int)ns;
    sp.per = (chunks + ns - 1) / ns * 32;
    sp.nsp = (int)((sp.per + kSpanX - 1) / kSpanX);
    sp.unit = 1;
    a.spf[c] = spf[c];
  }
  *launches = 0;
  for (int k = 0; k < 2; ++k) {
    if (!plan.ntiles[k]) continue;
    cudaError_t e;
    if (complex_out == 1) e = k == 0 ? simt4_t<4, 4, true>(a, plan, k, nsm, st) : simt4_t<8, 4, true>(a, plan, k, nsm, st);
    else e = k == 0 ? simt4_t<8, 4, false>(a, plan, k, nsm, st) : simt4_t<8, 8, false>(a, plan, k, nsm, st);
    if (e != cudaSuccess) return e;
    ++*launches;
  }
  return cudaSuccess;
}

// ------------------------------------------------------------- finalisation --
__global__ void couple_kernel(const double* __restrict__ T, int complex_t, const int* __restrict__ ptr,
                              const int* __restrict__ idx, const double* __restrict__ coef, int nout,
                              double* __restrict__ zeta, long long t_stride) {
  const int o = blockIdx.x * blockDim.x + threadIdx.x;
  if (o >= nout) return;
  // field blockIdx.y of a slab: its T and zeta follow the previous field's
  T += (long long)blockIdx.y * t_stride * (complex_t ? 2 : 1);
  zeta += (long long)blockIdx.y * nout * (complex_t ? 2 : 1);
  double re = 0.0, im = 0.0;
  for (int e = ptr[o]; e < ptr[o + 1]; ++e) {
    int i = idx[e];
    const bool cj = i < 0;
    if (cj) i = -i - 1;
    const double c = coef ? coef[e] : 1.0;
    if (complex_t) {
      re += c * T[2LL * i];
      im += c * (cj ? -T[2LL * i + 1] : T[2LL * i + 1]);
    } else {
      re += c * T[i];
    }
  }
  if (complex_t) {
    zeta[2LL * o] = re;
    zeta[2LL * o + 1] = im;
  } else {
    zeta[o] = re;
  }
}

cudaError_t launch_couple(const double* T, int complex_t, const int* ptr, const int* idx, const double* coef, int nout,
                          double* zeta, cudaStream_t st, int nfld, long long t_stride) {
  if (nout <= 0) return cudaSuccess;
  if (nfld < 1 || nfld > 65535) return cudaErrorInvalidValue;
  couple_kernel<<<dim3((nout + 255) / 256, nfld), 256, 0, st>>>(T, complex_t, ptr, idx, coef, nout, zeta, t_stride);
  return cudaGetLastError();
}

__global__ void finish3_kernel(const double* __restrict__ S, int full, int lmax, int nb, double* __restrict__ zeta,
                               long long s_stride) {
  const int nl = lmax + 1;
  const int o = blockIdx.x * blockDim.x + threadIdx.x;
  if (o >= nl * nb * nb) return;
  // field blockIdx.y of a slab
  S += (long long)blockIdx.y * s_stride;
  zeta += (long long)blockIdx.y * nl * nb * nb * (full ? 1 : 2);
  const int l = o / (nb * nb), b1 = (o / nb) % nb, b2 = o % nb;
  // S stored for b1 <= b2; S[b2][b1] = conj(S[b1][b2])
  const int lo = min(b1, b2), hi = max(b1, b2);
  const double cj = (b1 <= b2) ? 1.0 : -1.0;
  if (full) {
    double s = 0.0;
    for (int m = 0; m <= l; ++m) {
      const long long pi = (long long)l * (l + 1) / 2 + m;
      const double re = S[((pi * nb + lo) * nb + hi) * 2];
      s += (m == 0 ? 1.0 : 2.0) * re;
    }
    zeta[o] = ((l & 1) ? -1.0 : 1.0) / sqrt(2.0 * l + 1.0) * s;
  } else {
    const long long pi = l;
    zeta[2LL * o] = S[((pi * nb + lo) * nb + hi) * 2];
    zeta[2LL * o + 1] = cj * S[((pi * nb + lo) * nb + hi) * 2 + 1];
  }
}

cudaError_t launch_finish3(const double* S, int full, int lmax, int nb, double* zeta, cudaStream_t st, int nfld,
                           long long s_stride) {
  if (nfld < 1 || nfld > 65535) return cudaErrorInvalidValue;
  const int n = (lmax + 1) * nb * nb;
  finish3_kernel<<<dim3((n + 255) / 256, nfld), 256, 0, st>>>(S, full, lmax, nb, zeta, s_stride);
  return cudaGetLastError();
}

__global__ void normalize_kernel(double* zeta, long long nouter, int nb, int order, int ncomp, const double* acc,
                                 double ng, const double* vbin) {
  const long long per = (order == 4 ? (long long)nb * nb * nb : (long long)nb * nb);
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= nouter * per) return;
  // field blockIdx.y of a slab: its outputs and N_gal
  zeta += (long long)blockIdx.y * nouter * per * ncomp;
  const double ngal = acc[2 * blockIdx.y + 1];
  const double nbar = ngal / ng;
  const long long w = i % per;
  double norm = ngal;
  if (order == 4) {
    norm *= nbar * vbin[w / (nb * nb)] * nbar * vbin[(w / nb) % nb] * nbar * vbin[w % nb];
  } else {
    norm *= nbar * vbin[w / nb] * nbar * vbin[w % nb];
  }
  for (int c = 0; c < ncomp; ++c) zeta[i * ncomp + c] /= norm;
}

cudaError_t launch_normalize(double* zeta, long long nouter, int nb, int order, int ncomp, const double* acc, double ng,
                             const double* vbin_dev, cudaStream_t st, int nfld) {
  const long long per = (order == 4 ? (long long)nb * nb * nb : (long long)nb * nb);
  const long long n = nouter * per;
  if (n <= 0) return cudaSuccess;
  if (nfld < 1 || nfld > 65535) return cudaErrorInvalidValue;
  normalize_kernel<<<dim3((unsigned)((n + 255) / 256), nfld), 256, 0, st>>>(zeta, nouter, nb, order, ncomp, acc, ng,
                                                                            vbin_dev);
  return cudaGetLastError();
}

}  // namespace sbg

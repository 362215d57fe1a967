// Sparse MPO action with its input rows staged in shared memory (the general kernels are in
// kernels.cu).
//
// A stage multiplies, for every batch index, the short sparse rows of an MPO core (8 nonzeros on
// average, the longest 89 to 165 at L = 16; 18 and 211 in the folded hand-over core) with dense
// rows of a tensor: out[r][v] = sum_e val[e] in[row(e)][v].  Each input
// row is used by as many output rows, and gathering it from L2 every time is what bounded
// the general kernels: 7.5 TB/s of gathers for 2.1 to 2.5 TB/s of tensor traffic.  Here a
// block takes a narrow slice of the vector index (32 to 128 bytes a row) of ALL input rows of
// one batch index into shared memory (72 to 114 KB at bond dimensions of 342 to 562, so
// that two or three blocks share an SM and one's copies overlap another's sums) and then
// forms every output row of the slice from there.  L lanes with 16 bytes each serve an
// output row, 32 / L rows a warp.  The rows are sorted by their number of nonzeros (the rows
// of a warp then have the same length) and the nonzeros of 16 consecutive rows are
// interleaved, so that a warp reads the indices of its rows with one memory request; row by
// row they took 32 / L requests each, more than the sums themselves.  Sums run over the
// nonzeros in their stored order, as in the general kernels: the results are the same bits.
// Measured at D = 256 on the L = 16 chemistry MPO (bond 5; ms, general kernel first):
// BF16 S2 0.78 -> 0.58, S3 1.01 -> 0.76; FP32 pairs S2 + S3 6.34 -> 5.42; bond 7, split
// products, S3 (three planes in and out) 4.82 -> 3.68.
#include <algorithm>

#include "kernels.cuh"
#include "sparse.cuh"

namespace a2 {
namespace {

constexpr size_t kStTwo = 112 * 1024;    // shared memory of a block when two share an SM

struct StArgs {
  SparseRows<float> sp;
  SparseGeom g;
  const void* in;
  long long in_plane;      // planes / pairs: distance of the parts
  void* out;
  long long out_plane;
  int lsh;                 // log2 of the lanes per row
};

template <int IN> struct StIn;
template <> struct StIn<ST_BF16> { using T = __nv_bfloat16; static constexpr int NV = 8; };
template <> struct StIn<ST_PLANES> { using T = __nv_bfloat16; static constexpr int NV = 4; };
template <> struct StIn<ST_DF> { using T = float; static constexpr int NV = 4; };

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                   (unsigned)__cvta_generic_to_shared(dst)),
               "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
}

__device__ __forceinline__ void split3f(float x, __nv_bfloat16& h, __nv_bfloat16& m,
                                        __nv_bfloat16& l) {
  h = __float2bfloat16_rn(x);
  const float r1 = x - __bfloat162float(h);
  m = __float2bfloat16_rn(r1);
  l = __float2bfloat16_rn(r1 - __bfloat162float(m));
}

// Double-float multiply-add (Dekker's exact product via FMA, Knuth's two-sum; the
// product of the two low parts, below 2^-48 of the result, is dropped).
__device__ __forceinline__ void df_fma(float& ah, float& al, float wh, float wl, float xh,
                                       float xl) {
  const float p = __fmul_rn(wh, xh);
  const float pe = __fmaf_rn(wh, xh, -p);
  const float q = __fmaf_rn(wh, xl, __fmaf_rn(wl, xh, pe));
  const float s = __fadd_rn(ah, p);
  const float bp = __fsub_rn(s, ah);
  const float err = __fadd_rn(__fsub_rn(ah, __fsub_rn(s, bp)), __fsub_rn(p, bp));
  ah = s;
  al = __fadd_rn(al, __fadd_rn(err, q));
}

// OUT: ST_BF16, ST_PLANES (three BF16 planes), ST_DF (FP32 pair), ST_F64 (sum of the pair).
// ADD: added to the output (BF16).  VEC: every row segment is 16-byte (8-byte for planes) aligned
// and whole; otherwise element by element (not for planes).
template <int IN, int OUT, bool ADD, bool VEC, int NT>
__global__ void __launch_bounds__(NT, 1024 / NT) sparse_staged_kernel(StArgs a) {
  using TI = typename StIn<IN>::T;
  constexpr int NV = StIn<IN>::NV;
  constexpr bool kPair = IN == ST_DF;
  extern __shared__ __align__(16) unsigned char st_smem[];
  const SparseGeom& g = a.g;
  const int L = 1 << a.lsh, rows = a.sp.in_rows, nt = a.sp.in_t;
  const int b1 = blockIdx.z / g.B2, b2 = blockIdx.z % g.B2;
  const long long ib = (long long)b1 * g.in_b1 + (long long)b2 * g.in_b2;
  const int vbase = blockIdx.y * (L * NV);
  const int nvec = min(L * NV, g.veclen - vbase);      // elements of this slice
  const TI* in = reinterpret_cast<const TI*>(a.in) + ib + vbase;
  uint4* sh = reinterpret_cast<uint4*>(st_smem);       // [row][lane] (hi parts)
  uint4* sl = sh + (size_t)rows * L;                   // low parts (pairs)
  // ---- stage the slice of every input row
  if constexpr (VEC) {
    for (int it = threadIdx.x; it < rows * L; it += NT) {
      const int row = it >> a.lsh, l = it & (L - 1);
      if (l * NV >= nvec) continue;
      const TI* src = in + (long long)(row / nt) * g.in_sw + (long long)(row % nt) * g.in_st + l * NV;
      if constexpr (IN == ST_PLANES) {
        float x[4];
        const uint2 p0 = __ldg(reinterpret_cast<const uint2*>(src));
        const uint2 p1 = __ldg(reinterpret_cast<const uint2*>(src + a.in_plane));
        const uint2 p2 = __ldg(reinterpret_cast<const uint2*>(src + 2 * a.in_plane));
        const __nv_bfloat16* q0 = reinterpret_cast<const __nv_bfloat16*>(&p0);
        const __nv_bfloat16* q1 = reinterpret_cast<const __nv_bfloat16*>(&p1);
        const __nv_bfloat16* q2 = reinterpret_cast<const __nv_bfloat16*>(&p2);
#pragma unroll
        for (int i = 0; i < 4; ++i)
          x[i] = __bfloat162float(q0[i]) + (__bfloat162float(q1[i]) + __bfloat162float(q2[i]));
        *reinterpret_cast<float4*>(sh + it) = make_float4(x[0], x[1], x[2], x[3]);
      } else {
        cp_async16(sh + it, src);
        if constexpr (kPair) cp_async16(sl + it, src + a.in_plane);
      }
    }
    if constexpr (IN != ST_PLANES) cp_async_wait();
  } else {
    TI* eh = reinterpret_cast<TI*>(sh);
    TI* el = reinterpret_cast<TI*>(sl);
    const int wsh = a.lsh + (NV == 8 ? 3 : 2);         // log2 of the slice's width
    for (int it = threadIdx.x; it < rows << wsh; it += NT) {
      const int row = it >> wsh, v = it & ((1 << wsh) - 1);
      if (v >= nvec) continue;
      const TI* src = in + (long long)(row / nt) * g.in_sw + (long long)(row % nt) * g.in_st + v;
      eh[it] = __ldg(src);
      if constexpr (kPair) el[it] = __ldg(src + a.in_plane);
    }
  }
  __syncthreads();
  // ---- output rows: a warp takes 32 / L consecutive rows at a time, L lanes each
  const int lane = threadIdx.x & (L - 1), sub = (threadIdx.x & 31) >> a.lsh;
  const int csh = 5 - a.lsh;                           // log2 of the rows per warp
  const int nunits = (a.sp.nrows + (1 << csh) - 1) >> csh;
  const int v = lane * NV;
  if (v >= nvec) return;
  const long long ob = (long long)b1 * g.out_b1 + (long long)b2 * g.out_b2 + vbase + v;
  for (int un = blockIdx.x + gridDim.x * (threadIdx.x >> 5); un < nunits;
       un += gridDim.x * (NT / 32)) {
    const int r = (un << csh) + sub;
    if (r >= a.sp.nrows) continue;
    const int4 meta = __ldg(a.sp.sell_row + r);        // length, first entry, output (w, s)
    const int2* __restrict__ pk = a.sp.sell + meta.y;
    const float* __restrict__ wlo = a.sp.sell_lo + meta.y;
    float acc[NV], acl[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) acc[i] = acl[i] = 0.f;
    auto one = [&](const int2& k, float wl) {
      const float w = __int_as_float(k.y);
      const uint4 raw = sh[(k.x << a.lsh) + lane];
      if constexpr (IN == ST_BF16) {
        const unsigned u[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          acc[2 * i] = fmaf(w, __uint_as_float(u[i] << 16), acc[2 * i]);
          acc[2 * i + 1] = fmaf(w, __uint_as_float(u[i] & 0xffff0000u), acc[2 * i + 1]);
        }
      } else {
        const float x[4] = {__uint_as_float(raw.x), __uint_as_float(raw.y),
                            __uint_as_float(raw.z), __uint_as_float(raw.w)};
        if constexpr (kPair) {
          const uint4 rl = sl[(k.x << a.lsh) + lane];
          const float y[4] = {__uint_as_float(rl.x), __uint_as_float(rl.y),
                              __uint_as_float(rl.z), __uint_as_float(rl.w)};
#pragma unroll
          for (int i = 0; i < 4; ++i) df_fma(acc[i], acl[i], w, wl, x[i], y[i]);
        } else {
#pragma unroll
          for (int i = 0; i < 4; ++i) acc[i] = fmaf(w, x[i], acc[i]);
        }
      }
    };
    int e = 0;
    for (; e + 4 <= meta.x; e += 4) {   // four index loads in flight (loading further ahead
                                        // costs more instructions than it gains)
      int2 k[4];
      float wl[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        k[u] = __ldg(pk + (e + u) * kSellRows);
        wl[u] = kPair ? __ldg(wlo + (e + u) * kSellRows) : 0.f;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) one(k[u], wl[u]);
    }
    for (; e < meta.x; ++e)
      one(__ldg(pk + e * kSellRows), kPair ? __ldg(wlo + e * kSellRows) : 0.f);
    const long long o = ob + (long long)meta.z * g.out_sw + (long long)meta.w * g.out_ss;
    const int nst = VEC ? NV : min(NV, nvec - v);
    if constexpr (OUT == ST_BF16) {
      __nv_bfloat16* p = reinterpret_cast<__nv_bfloat16*>(a.out) + o;
      __align__(16) __nv_bfloat16 t[NV];
      if constexpr (ADD) {
#pragma unroll
        for (int i = 0; i < NV; ++i)
          if (VEC || i < nst) acc[i] += __bfloat162float(p[i]);
      }
#pragma unroll
      for (int i = 0; i < NV; ++i) t[i] = __float2bfloat16_rn(acc[i]);
      if constexpr (VEC) {
        *reinterpret_cast<uint4*>(p) = *reinterpret_cast<const uint4*>(t);
      } else {
#pragma unroll
        for (int i = 0; i < NV; ++i)
          if (i < nst) p[i] = t[i];
      }
    } else if constexpr (OUT == ST_PLANES) {
      __nv_bfloat16* p = reinterpret_cast<__nv_bfloat16*>(a.out) + o;
      __align__(8) __nv_bfloat16 h[NV], m[NV], l3[NV];
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        split3f(acc[i], h[i], m[i], l3[i]);
      }
      *reinterpret_cast<uint2*>(p) = *reinterpret_cast<const uint2*>(h);
      *reinterpret_cast<uint2*>(p + a.out_plane) = *reinterpret_cast<const uint2*>(m);
      *reinterpret_cast<uint2*>(p + 2 * a.out_plane) = *reinterpret_cast<const uint2*>(l3);
    } else if constexpr (OUT == ST_DF) {
      float* p = reinterpret_cast<float*>(a.out) + o;
      float h[NV], lo[NV];
#pragma unroll
      for (int i = 0; i < NV; ++i) {   // renormalise: |lo| <= ulp(hi) / 2
        const float s = __fadd_rn(acc[i], acl[i]);
        h[i] = s;
        lo[i] = __fsub_rn(acl[i], __fsub_rn(s, acc[i]));
      }
      if constexpr (VEC) {
        *reinterpret_cast<float4*>(p) = make_float4(h[0], h[1], h[2], h[3]);
        *reinterpret_cast<float4*>(p + a.out_plane) = make_float4(lo[0], lo[1], lo[2], lo[3]);
      } else {
#pragma unroll
        for (int i = 0; i < NV; ++i)
          if (i < nst) {
            p[i] = h[i];
            p[a.out_plane + i] = lo[i];
          }
      }
    } else {
      double* p = reinterpret_cast<double*>(a.out) + o;
      if constexpr (VEC) {
        *reinterpret_cast<double2*>(p) = make_double2((double)acc[0] + (double)acl[0],
                                                      (double)acc[1] + (double)acl[1]);
        *reinterpret_cast<double2*>(p + 2) = make_double2((double)acc[2] + (double)acl[2],
                                                          (double)acc[3] + (double)acl[3]);
      } else {
#pragma unroll
        for (int i = 0; i < NV; ++i)
          if (i < nst) p[i] = (double)acc[i] + (double)acl[i];
      }
    }
  }
}

template <int IN, int OUT, bool ADD, bool VEC, int NT>
void st_launch(const StArgs& a, dim3 grid, size_t smem, cudaStream_t s) {
  static PerDevice<bool> set;
  set.at(current_device(), [] {
    A2_CUDA(cudaFuncSetAttribute(sparse_staged_kernel<IN, OUT, ADD, VEC, NT>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024));
    return true;
  });
  sparse_staged_kernel<IN, OUT, ADD, VEC, NT><<<grid, NT, smem, s>>>(a);
  A2_CHECK_LAUNCH();
}

template <int IN, int OUT, bool ADD>
void st_launch_vec(const StArgs& a, bool vec, dim3 grid, size_t smem, cudaStream_t s) {
  const bool one = smem > kStTwo;        // one block on an SM: twice the threads
  if (vec) {
    if (one) st_launch<IN, OUT, ADD, true, 1024>(a, grid, smem, s);
    else st_launch<IN, OUT, ADD, true, 512>(a, grid, smem, s);
  } else if constexpr (IN != ST_PLANES) {
    if (one) st_launch<IN, OUT, ADD, false, 1024>(a, grid, smem, s);
    else st_launch<IN, OUT, ADD, false, 512>(a, grid, smem, s);
  }
}

}  // namespace

// Taken when a staged row is used at least twice on average and there are enough of them
// for the staging to matter (Heisenberg's 10 rows stay with the general kernels: the same
// time, no copies); the widest slice that leaves room for two blocks on an SM, but at least
// 64 bytes a row where one block's shared memory holds that (narrower rows conflict in the
// banks: bond 7's S3 3.68 ms, with 32 bytes 4.04).  Pairs go down to 16 + 16 bytes instead:
// they are bound by arithmetic and want the second block (bond 7, D = 128: S2 + S3 5.35 ms
// against 5.78 with one).  FP32 inputs stay with the general kernels, which gather them at 10 TB/s and
// were as fast or faster (bond 5: S2 1.10 ms both, S3 1.53 against 1.71; bond 7: S2 1.92
// against 2.33).  BF16 rows that are not whole 16-byte vectors are copied element by element,
// which pays with long rows only (16 nonzeros or more on average; S3 at Dl, Dr = 40, 98: 0.100 ms
// against 0.152; short ones 107, 234: 0.254 against 0.196; 41, 44: 0.054 against 0.029); under 128
// blocks the general kernels, with one warp a row, spread better (S2 at 45, 26, 90 blocks: 13.6 us
// against 10.1).
bool sparse_staged(const SparseRows<float>& sp, const SparseGeom& g, int in_kind, const void* in,
                   long long in_plane, int out_kind, void* out, long long out_plane,
                   cudaStream_t s) {
  if (!sp.sell || sp.in_rows < 64 || sp.nnz_total < 2LL * sp.in_rows) return false;
  const int nv = in_kind == ST_BF16 ? 8 : 4;
  const size_t unit = (size_t)sp.in_rows * 16 * (in_kind == ST_DF ? 2 : 1);   // one lane
  int lmax = 0;
  while (lmax < 3 && (1 << lmax) * nv < g.veclen) ++lmax;
  const int lgood = std::min(lmax, in_kind == ST_DF ? 0 : 2);
  int lsh = lmax;
  while (lsh > lgood && (unit << lsh) > kStTwo) --lsh;
  while (lsh > 0 && (unit << lsh) > 220 * 1024) --lsh;
  if ((unit << lsh) > 220 * 1024) return false;
  const int nt = (unit << lsh) > kStTwo ? 1024 : 512;
  const long long chunks = cdiv(g.veclen, nv << lsh), batch = (long long)g.B1 * g.B2;
  if (chunks >= 65536 || batch >= 65536) return false;
  // too few slices for the SMs: the rows are shared out as well
  const long long blocks = chunks * batch;
  int parts = 1;
  if (blocks < 304) parts = (int)std::min<long long>((304 + blocks - 1) / blocks,
                                                     cdiv(sp.nrows, nt >> lsh));
  // aligned: 16 bytes of input per lane (8 of each plane), whole vectors in and out
  const int isz = in_kind == ST_DF ? 4 : 2;
  const int osz = out_kind == ST_F64 ? 8 : out_kind == ST_DF ? 4 : 2;
  auto al = [&](long long x) { return x % nv == 0; };
  const bool vec = al(g.veclen) && al(g.in_sw) && al(g.in_st) && al(g.in_b1) && al(g.in_b2) &&
                   al(in_plane) && al(g.out_sw) && al(g.out_ss) && al(g.out_b1) &&
                   al(g.out_b2) && al(out_plane) &&
                   reinterpret_cast<uintptr_t>(in) % (isz * nv) == 0 &&
                   reinterpret_cast<uintptr_t>(out) % std::min(16, osz * nv) == 0;
  if (in_kind == ST_BF16 && (blocks < 128 || (!vec && sp.nnz_total < 16LL * sp.nrows)))
    return false;
  if (in_kind == ST_PLANES && !vec) return false;   // (its callers' rows are padded)
  StArgs a;
  a.sp = sp;
  a.g = g;
  a.in = in;
  a.in_plane = in_plane;
  a.out = out;
  a.out_plane = out_plane;
  a.lsh = lsh;
  const dim3 grid(parts, (unsigned)chunks, (unsigned)batch);
  const size_t smem = unit << lsh;
  if (in_kind == ST_BF16 && out_kind == ST_BF16) {
    if (g.accumulate) st_launch_vec<ST_BF16, ST_BF16, true>(a, vec, grid, smem, s);
    else st_launch_vec<ST_BF16, ST_BF16, false>(a, vec, grid, smem, s);
  } else if (in_kind == ST_PLANES && out_kind == ST_PLANES) {
    st_launch_vec<ST_PLANES, ST_PLANES, false>(a, vec, grid, smem, s);
  } else if (in_kind == ST_DF && out_kind == ST_DF) {
    st_launch_vec<ST_DF, ST_DF, false>(a, vec, grid, smem, s);
  } else if (in_kind == ST_DF && out_kind == ST_F64) {
    st_launch_vec<ST_DF, ST_F64, false>(a, vec, grid, smem, s);
  } else {
    return false;
  }
  return true;
}

}  // namespace a2

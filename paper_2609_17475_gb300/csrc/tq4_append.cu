// TQ4 encode on append (Sec. 3.1 Eq. 4; App. A.1 Table 3).
//
// The index decision z_j = #{k : u_j > T_k}, u = H_d S x, T_k =
// fp64(fp64(sqrt(d) rho) t_k), is made exactly: a fp32 Hadamard butterfly
// decides every element whose value lies farther than a margin from every
// threshold (it is within 2^-17 rho of the exact value: 8 levels of rounding,
// each at most 2^-24 of a partial sum bounded by sum|x| <= sqrt(d) rho); the
// few closer ones are summed again in fp64, which is exact for bf16 inputs
// whose magnitudes span less than 2^37.  rho is the fp32 rounding of the
// square root of the fp64 sum of squares, from a certified double-float sum.
//
// The work is bound by issue slots, so the layout cuts instructions: 8 lanes
// hold a vector (32 elements each at D = 256), which leaves 3 of the
// butterfly's 8 levels to shuffles and does the rest, like the sum of squares,
// on packed fp32 pairs; and an index takes one table lookup and one
// comparison: a cell of an eighth of rho holds at most one threshold, so the
// table gives the cell's threshold and the count below it.  2,048 rows of
// 24/4/256 (16,384 vectors): 20.1 us with one warp per vector (a 4-level
// threshold search, 890 instructions a vector), 11.9 us now (310).
#include <cstring>

#include "decode_frag.cuh"
#include "tq4_encode.cuh"

namespace jfkv {

struct Tq4AppendArgs {
  uint8_t* pool;
  int64_t num_pages;
  int64_t page_bytes;
  int64_t codes_region;
  int64_t norm_region;
  int32_t P, log2P;   // P is a power of two
  int32_t Hkv;
  const int32_t* page_table;
  int32_t pt_stride;
  int32_t num_requests;
  const int32_t* row_req;
  const int32_t* row_pos;
  const uint16_t* k;
  const uint16_t* v;
  int32_t n_rows;
  int32_t* err;
};

// One vector of the call: its source, K or V, head and destination slot.
struct AppendSlot {
  const uint16_t* src;
  int kind;
  uint8_t* page;   // page record, or null (reported)
  int64_t vrow;    // head * P + slot
};

template <int D>
__device__ __forceinline__ AppendSlot append_slot(const Tq4AppendArgs& a, int64_t vec, bool report) {
  // 64-bit division is ~100 instructions, and few calls need it
  int64_t row;
  int rem;
  if (vec <= 0x7FFFFFFF) {
    const uint32_t q = (uint32_t)vec / (uint32_t)(2 * a.Hkv);
    row = q;
    rem = (int)((uint32_t)vec - q * (uint32_t)(2 * a.Hkv));
  } else {
    row = vec / (2 * a.Hkv);
    rem = (int)(vec % (2 * a.Hkv));
  }
  AppendSlot s;
  s.kind = rem >= a.Hkv ? 1 : 0;
  const int head = rem - s.kind * a.Hkv;
  s.src = (s.kind ? a.v : a.k) + (row * a.Hkv + head) * D;
  s.page = nullptr;
  s.vrow = 0;
  const int32_t req = a.row_req[row];
  const int32_t pos = a.row_pos[row];
  if (req < 0 || req >= a.num_requests || pos < 0 || (pos >> a.log2P) >= a.pt_stride) {
    if (report) flag_error(a.err, JF_DEV_ERR_POSITION);
    return s;
  }
  const int32_t page = a.page_table[(int64_t)req * a.pt_stride + (pos >> a.log2P)];
  if (page < 0 || page >= a.num_pages) {
    if (report) flag_error(a.err, JF_DEV_ERR_PAGE_ID);
    return s;
  }
  s.page = a.pool + (int64_t)page * a.page_bytes;
  s.vrow = (int64_t)head * a.P + (pos & (a.P - 1));
  return s;
}

// One warp per vector: codebooks whose thresholds the lookup table cannot
// hold, and single vectors whose norm is outside the fast path's range.
template <int D>
__device__ __noinline__ void append_one(const Tq4AppendArgs& a, const Tq4Params& prm, int64_t vec,
                                        int lane) {
  const AppendSlot s = append_slot<D>(a, vec, lane == 0);
  float rho;
  const uint32_t word = tq4_encode<D>(s.src, s.kind, prm, lane, rho);
  if (s.page)
    tq4_store<D>(s.page, a.codes_region, a.norm_region, s.kind, s.vrow, lane, word, rho);
}

template <int D>
__global__ void __launch_bounds__(256)
tq4_append_general_kernel(const __grid_constant__ Tq4AppendArgs a, const __grid_constant__ Tq4Params prm) {
  const int64_t vec = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  if (vec >= (int64_t)a.n_rows * a.Hkv * 2) return;   // whole warps
  append_one<D>(a, prm, vec, threadIdx.x & 31);
}

// Threshold table.  Cell i covers u / rho in [(i - 32.5) / 8, (i - 31.5) / 8]
// (the outer two run on); its word is the float threshold (in units of rho)
// that lies in it or within 1/64 cell of it, rounded to a multiple of 16 ulps,
// with the number of thresholds below the cell in the low 4 bits (a huge
// threshold where there is none).  A threshold at or next to zero is taken as
// 2^-40, well inside the margin below: the count's place among the bits of a
// zero would make them those of a NaN.  False if a cell would need two.
constexpr int TQ_CELLS = 65;
struct Tq4Lut {
  uint32_t w[TQ_CELLS];
};

static bool tq4_make_lut(const Tq4Params& p, Tq4Lut* lut) {
  if (p.exact_all || !(p.tq[0] > -3.9f) || !(p.tq[14] < 3.9f)) return false;
  uint32_t below = 0;   // thresholds below the cell (both ascend)
  for (int i = 0; i < TQ_CELLS; ++i) {
    const float lo = i == 0 ? -1e9f : (i - 32.5f - 1.f / 64) / 8;
    const float hi = i == TQ_CELLS - 1 ? 1e9f : (i - 31.5f + 1.f / 64) / 8;
    while (below < 15 && p.tq[below] < lo) ++below;
    float thr = 1e30f;
    if (below < 15 && p.tq[below] <= hi) {
      thr = p.tq[below];
      if (below < 14 && p.tq[below + 1] <= hi) return false;
    }
    if (std::fabs(thr) < 0x1p-40f) thr = 0x1p-40f;
    uint32_t b;
    std::memcpy(&b, &thr, 4);
    lut->w[i] = ((b - below + 8) & ~15u) | below;
  }
  return true;
}

__device__ __forceinline__ f2 shfl_xor2(f2 x, int m) {
  f2 r;
  r.v = __shfl_xor_sync(0xffffffffu, x.v, m);
  return r;
}

// (s, e) += b on a packed pair of double-float accumulators (Knuth's TwoSum)
__device__ __forceinline__ void two_sum_acc2(f2& s, f2& e, f2 b) {
  const f2 t = add2(s, b);
  const f2 bb = sub2(t, s);
  e = add2(e, add2(sub2(s, sub2(t, bb)), sub2(b, bb)));
  s = t;
}

// Lane l (of the 8 of a vector) holds element 64 k + 8 l + e in x[8 k + e]:
// 16-byte loads of 128 contiguous bytes per vector, and one 32-bit word of
// indices for each k.  Packed as pairs (x[i], x[i + N/2]).
template <int D>
__global__ void __launch_bounds__(128)
tq4_append_kernel(const __grid_constant__ Tq4AppendArgs a, const __grid_constant__ Tq4Params prm,
                  const __grid_constant__ Tq4Lut tab) {
  constexpr int N = D / 8;     // elements per lane
  constexpr int K = N / 8;     // 8-element runs per lane
  constexpr int NP = N / 2;    // packed pairs
  __shared__ uint32_t lut[TQ_CELLS];
  if (threadIdx.x < TQ_CELLS) lut[threadIdx.x] = tab.w[threadIdx.x];
  const int lane = threadIdx.x & 31, l = lane & 7;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t total = (int64_t)a.n_rows * a.Hkv * 2;
  __syncthreads();
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  if (warp * 4 >= total) return;   // whole warps
  const int64_t vec = warp * 4 + (lane >> 3);
  const bool live = vec < total;
  const AppendSlot slot = append_slot<D>(a, live ? vec : total - 1, live && l == 0);

  uint4 raw[K];
#pragma unroll
  for (int k = 0; k < K; ++k) raw[k] = *reinterpret_cast<const uint4*>(slot.src + 64 * k + 8 * l);

  // x with the signs of S
  f2 v[NP];
  {
    float x[N];
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const uint32_t sw = (slot.kind ? prm.sv : prm.sk)[2 * k + (l >> 2)] >> (8 * (l & 3));
      const uint32_t w[4] = {raw[k].x, raw[k].y, raw[k].z, raw[k].w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint32_t s = w[i] ^ (((sw << (15 - 2 * i)) & 0x8000u) |
                                   ((sw << (30 - 2 * i)) & 0x80000000u));
        x[8 * k + 2 * i] = bf16lo_to_f32(s);
        x[8 * k + 2 * i + 1] = bf16hi_to_f32(s);
      }
    }
#pragma unroll
    for (int i = 0; i < NP; ++i) v[i] = mk2(x[i], x[i + NP]);
  }

  // rho (see tq4_encode): certified double-float sum of the exact squares
  float rho;
  {
    f2 s2 = mk2(0.f, 0.f), e2 = s2;
#pragma unroll
    for (int i = 0; i < NP; ++i) two_sum_acc2(s2, e2, mul2(v[i], v[i]));
    float sh, sl, bh, bl;
    un2(s2, sh, bh);
    un2(e2, sl, bl);
    two_sum_acc(sh, sl, bh);
    sl = __fadd_rn(sl, bl);
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
      bh = __shfl_xor_sync(0xffffffffu, sh, o);
      bl = __shfl_xor_sync(0xffffffffu, sl, o);
      two_sum_acc(sh, sl, bh);
      sl = __fadd_rn(sl, bl);
    }
    bool sure;
    rho = rho_from_sum(sh, sl, sure);
    if (__any_sync(0xffffffffu, !sure)) {
      double s = 0.0;
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        float x0, x1;
        un2(v[i], x0, x1);
        s += (double)x0 * (double)x0;
        s += (double)x1 * (double)x1;
      }
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (!sure) rho = __double2float_rn(sqrt(s));
    }
  }

  // u = H S x: levels on the elements of a lane (packed, then across the
  // pair), then across lanes (lower lane: u + o; upper lane: o - u)
#pragma unroll
  for (int h = 1; h < NP; h <<= 1)
#pragma unroll
    for (int i = 0; i < NP; ++i)
      if (!(i & h)) {
        const f2 p = v[i], q = v[i + h];
        v[i] = add2(p, q);
        v[i + h] = sub2(p, q);
      }
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    float p, q;
    un2(v[i], p, q);
    v[i] = mk2(p + q, p - q);
  }
#pragma unroll
  for (int m = 1; m < 8; m <<= 1) {
    const float sg = (l & m) ? -1.f : 1.f;
    const f2 sg2 = mk2(sg, sg);
#pragma unroll
    for (int i = 0; i < NP; ++i) v[i] = fma2(v[i], sg2, shfl_xor2(v[i], m));
  }

  // indices.  The table's thresholds are within 2^-18 rho (of at most 4 rho)
  // of the contract's, so with the butterfly's 2^-17 rho an element farther
  // than 2^-16 rho from its cell's threshold is decided.
  const bool in_range = rho >= 1e-30f && rho <= 1e36f;
  const float inv8 = __fdividef(0.125f, in_range ? rho : 1.f);
  const uint32_t lut0 = smem_u32(lut) - (0x4B400000u << 2);
  auto diff = [&](float u, uint32_t& w) -> float {
    float c;
    asm("fma.rn.sat.f32 %0, %1, %2, 0f3F000000;\n" : "=f"(c) : "f"(u), "f"(inv8));
    c = __fmaf_rn(c, 64.f, 12582912.f);
    asm("ld.shared.b32 %0, [%1];\n" : "=r"(w) : "r"(lut0 + (__float_as_uint(c) << 2)));
    return __fmaf_rn(-rho, __uint_as_float(w), u);
  };
  float closest = INFINITY;
  uint32_t word[K];
#pragma unroll
  for (int k = 0; k < K; ++k) word[k] = 0;
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    float u[2];
    un2(v[i], u[0], u[1]);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int idx = i + h * NP;
      uint32_t w;
      const float d = diff(u[h], w);
      closest = fminf(closest, fabsf(d));
      word[idx >> 3] += (w & 15u) << (4 * (idx & 7));
      if (d > 0.f) word[idx >> 3] += 1u << (4 * (idx & 7));
    }
  }
  const float M = rho * 0x1p-16f;
  const bool near = live && in_range && !(closest > M);

  if (__any_sync(0xffffffffu, near)) {
    // Elements within the margin (one vector in ~40): each group of 8 lanes
    // sums one of its own again, u_j = sum_i (-1)^popc(i & j) s_i x_i, and
    // compares with the contract's products for the two bracketing thresholds.
    // The sum is a double-float one, within 2^-38 rho; only when that does
    // not decide either is it taken in fp64 (70 fp64 instructions, 16 cycles
    // of the SM each).
    uint32_t todo = 0;
    if (near) {
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        float u[2];
        un2(v[i], u[0], u[1]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t w;
          if (!(fabsf(diff(u[h], w)) > M)) todo |= 1u << (i + h * NP);
        }
      }
    }
    const double r = (double)rho * sqrt((double)D);
    for (;;) {
      const uint32_t have = __ballot_sync(0xffffffffu, todo != 0);
      if (have == 0) break;
      const uint32_t mine = (have >> (lane & 24)) & 0xFFu;
      const int owner = mine ? (lane & 24) + __ffs(mine) - 1 : lane;
      const uint32_t bits = __shfl_sync(0xffffffffu, todo, owner);
      const int idx = mine ? __ffs(bits) - 1 : 0;
      const int j = 64 * (idx >> 3) + 8 * (owner & 7) + (idx & 7);
      const uint32_t jl = (uint32_t)__popc((8 * l) & j);
      f2 s2 = mk2(0.f, 0.f), e2 = s2;
#pragma unroll 1
      for (int k = 0; k < K; ++k) {
        const uint32_t sw = (slot.kind ? prm.sv : prm.sk)[2 * k + (l >> 2)] >> (8 * (l & 3));
        const uint32_t jk = jl + (uint32_t)__popc((64 * k) & j);
        const uint4 q = *reinterpret_cast<const uint4*>(slot.src + 64 * k + 8 * l);
        const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const uint32_t p0 = jk + (uint32_t)__popc((2 * i) & j) + (sw >> (2 * i));
          const uint32_t p1 = jk + (uint32_t)__popc((2 * i + 1) & j) + (sw >> (2 * i + 1));
          const uint32_t t = w[i] ^ ((p0 & 1u) << 15) ^ ((p1 & 1u) << 31);
          two_sum_acc2(s2, e2, mk2(bf16lo_to_f32(t), bf16hi_to_f32(t)));
        }
      }
      double s;
      {
        float sh, sl, bh, bl;
        un2(s2, sh, bh);
        un2(e2, sl, bl);
        two_sum_acc(sh, sl, bh);
        sl = __fadd_rn(sl, bl);
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) {
          bh = __shfl_xor_sync(0xffffffffu, sh, o);
          bl = __shfl_xor_sync(0xffffffffu, sl, o);
          two_sum_acc(sh, sl, bh);
          sl = __fadd_rn(sl, bl);
        }
        s = (double)sh + (double)sl;
      }
      // the owner's bracketing thresholds
      uint32_t wd = 0;
#pragma unroll
      for (int k = 0; k < K; ++k)
        if ((idx >> 3) == k) wd = word[k];
      const int sft = 4 * (idx & 7);
      const int zf = (wd >> sft) & 15;
      const int k0 = max(zf - 1, 0), k1 = min(zf + 1, 15);
      bool open = false;
      if (mine && lane == owner)
        for (int k = k0; k < k1; ++k)
          open = open || !(fabs(s - r * (double)prm.t[k]) > (double)(rho * 0x1p-36f));
      if (__any_sync(0xffffffffu, open)) {
        double x = 0.0;
#pragma unroll 1
        for (int i = 0; i < N; ++i) {
          const int at = 64 * (i >> 3) + 8 * l + (i & 7);
          const uint32_t flip = (((slot.kind ? prm.sv : prm.sk)[at >> 5] >> (at & 31)) ^
                                 (uint32_t)__popc(at & j)) & 1u;
          x += (double)__uint_as_float(((uint32_t)slot.src[at] << 16) ^ (flip << 31));
        }
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        s = x;
      }
      if (mine && lane == owner) {
        int z = k0;
        for (int k = k0; k < k1; ++k) z += (s > r * (double)prm.t[k]) ? 1 : 0;
        wd = (wd & ~(15u << sft)) | ((uint32_t)z << sft);
#pragma unroll
        for (int k = 0; k < K; ++k)
          if ((idx >> 3) == k) word[k] = wd;
        todo &= todo - 1;
      }
    }
  }

  if (live && in_range && slot.page) {
    uint32_t* dst = reinterpret_cast<uint32_t*>(slot.page + slot.kind * a.codes_region +
                                                slot.vrow * (D / 2));
#pragma unroll
    for (int k = 0; k < K; ++k) dst[8 * k + l] = word[k];
    if (l == 0) {
      const __half h = __float2half_rn(fminf(rho, 65504.f));
      *reinterpret_cast<uint16_t*>(slot.page + 2 * a.codes_region + slot.kind * a.norm_region +
                                   slot.vrow * 2) = __half_as_ushort(h);
    }
  }
  // norms outside the fast path's range (a zero vector among them)
  uint32_t rest = __ballot_sync(0xffffffffu, live && !in_range && l == 0);
  while (rest) {
    const int g = __ffs(rest) - 1;
    rest &= rest - 1;
    append_one<D>(a, prm, warp * 4 + (g >> 3), lane);
  }
}

int launch_tq4_append(const Geom& g, const jf_kv_pool& pool, const Tq4Params& prm,
                      const int32_t* page_table, int32_t pt_stride, int32_t num_requests,
                      const int32_t* row_req, const int32_t* row_pos, const void* k,
                      const void* v, int32_t n_rows, int32_t* err, cudaStream_t stream) {
  Tq4AppendArgs a;
  a.pool = static_cast<uint8_t*>(pool.base);
  a.num_pages = g.num_pages;
  a.page_bytes = g.page_bytes;
  a.codes_region = g.codes_region;
  a.norm_region = g.sb_region;
  a.P = g.P;
  a.log2P = __builtin_ctz((unsigned)g.P);
  a.Hkv = g.Hkv;
  a.page_table = page_table;
  a.pt_stride = pt_stride;
  a.num_requests = num_requests;
  a.row_req = row_req;
  a.row_pos = row_pos;
  a.k = static_cast<const uint16_t*>(k);
  a.v = static_cast<const uint16_t*>(v);
  a.n_rows = n_rows;
  a.err = err;
  // the table holds any codebook with thresholds more than 1/8 + 1/256 rho
  // apart (the Lloyd-Max ones are 0.25 or more apart); a closer one goes
  // through the kernel that takes a warp per vector
  Tq4Lut lut;
  const bool fast = tq4_make_lut(prm, &lut);
  const int64_t vectors = (int64_t)n_rows * g.Hkv * 2;
  const int64_t blocks = fast ? (vectors + 15) / 16 : (vectors + 7) / 8;
  if ((vectors + 7) / 8 > 0x7FFFFFFF) return JF_ERR_INVALID_ARG;
  cudaLaunchAttribute pdl[1];
  pdl[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  pdl[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)blocks);
  cfg.blockDim = dim3(fast ? 128 : 256);
  cfg.stream = stream;
  cfg.attrs = pdl;
  cfg.numAttrs = 1;
  cudaError_t e;
  if (fast)
    e = (g.D == 256) ? cudaLaunchKernelEx(&cfg, tq4_append_kernel<256>, a, prm, lut)
                     : cudaLaunchKernelEx(&cfg, tq4_append_kernel<128>, a, prm, lut);
  else
    e = (g.D == 256) ? cudaLaunchKernelEx(&cfg, tq4_append_general_kernel<256>, a, prm)
                     : cudaLaunchKernelEx(&cfg, tq4_append_general_kernel<128>, a, prm);
  return e == cudaSuccess ? JF_OK : JF_ERR_CUDA;
}

}  // namespace jfkv

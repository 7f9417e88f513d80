// razer_pack_layout, razer_dequant, razer_decode_act: layout shuffle and exact decode kernels.
#include "razer_common.cuh"
#include "razer_decode.cuh"
#include "razer_ptx.cuh"

namespace razer {

// pack_kernel and dequant_kernel work on spans: one strip (16 rows) x SPAN_CHUNKS chunks, whose pieces are contiguous in the
// packed buffer.  Both are bound by DRAM once every global access is contiguous: the row-major side is walked along K
// (a warp covers 32 neighbouring blocks of one row), the packed side in 16-byte vectors, and shared memory holds the span in
// between in the packed order.  Measured on B200 at 11008 x 4096: pack 26.7 -> 16.5 us, dequant to bf16 360.8 -> 26.7 us,
// to FP32 258.9 -> 54.9 us (a thread per block straight from the packed order wrote two bytes at a time).  Then 32-byte stores, and the
// nibble order by two selects and a byte permute instead of a nibble at a time (with the launch): pack 21.5 -> 19.5, bf16 30.7 ->
// 27.5, FP32 59.3 -> 38.9.
constexpr int SPAN_CHUNKS = 16;
constexpr int SPAN_BLOCKS = SPAN_CHUNKS * CHUNK_BLOCKS;              // 16-element blocks of one row of a span
constexpr int SPAN_BYTES = SPAN_CHUNKS * PIECE_BYTES;
constexpr int SPAN_THREADS = 256;
constexpr int FEW_CHUNKS = 4;

// Reads the interchange-format blocks (8 code bytes + 1 scale byte), canonicalises them and writes them at their packed
// positions.
// `sub` = 16-element groups per scale block (block size / 16): the packed form always carries one scale byte per 16
// elements, so a larger block's byte is repeated for each of its groups and the kernels need not know the block size.
// CHUNKS per span: SPAN_CHUNKS, or few where the tensor makes few spans.
template <int CHUNKS>
__global__ void __launch_bounds__(SPAN_THREADS) pack_kernel(const uint8_t* __restrict__ codes, const uint8_t* __restrict__ scales,
                                                            uint8_t* __restrict__ packed, Geometry g, int remap_code, int sub) {
  constexpr int BLOCKS = CHUNKS * CHUNK_BLOCKS;         // 16-element blocks of one row of a span
  __shared__ __align__(16) uint8_t span[CHUNKS * PIECE_BYTES];
  const int spans = (g.k_chunks + CHUNKS - 1) / CHUNKS;
  const int strip = (int)(blockIdx.x / (unsigned)spans), c0 = (int)(blockIdx.x % (unsigned)spans) * CHUNKS;
  const int n_chunks = min(CHUNKS, g.k_chunks - c0);
  // bit 3 of each nibble of nz is set iff the nibble's magnitude (low three bits) is non-zero
  auto canon = [&](uint32_t w, bool negate) -> uint32_t {
    const uint32_t m = w & 0x77777777u;
    const uint32_t nz = ((m + 0x77777777u) & 0x88888888u);
    if (remap_code == 0x8) w ^= (~nz) & 0x88888888u;  // packed form: special value 0x0, true zero 0x8
    if (negate) w ^= nz;                              // flip the sign of non-zero codes
    return w;
  };
  const int k16 = g.K / 16, ks = k16 / sub;
#pragma unroll
  for (int i = 0; i < STRIP_ROWS * BLOCKS / SPAN_THREADS; ++i) {
    const int b = (int)threadIdx.x + i * SPAN_THREADS, r = b / BLOCKS, kb_in = b % BLOCKS;
    const int n = strip * STRIP_ROWS + r, kb = c0 * CHUNK_BLOCKS + kb_in;
    uint32_t w0 = 0, w1 = 0, sb = 0;
    if (n < g.N && kb < k16) {
      const uint2 c = *reinterpret_cast<const uint2*>(codes + ((size_t)n * k16 + kb) * 8);
      w0 = c.x;
      w1 = c.y;
      sb = scales[(size_t)n * ks + (sub == 1 ? kb : kb / sub)];
    }
    const uint32_t scode = sb & 0x3Fu;
    const bool negate = (sb & 0x80u) != 0;              // negative special value: store the block negated
    uint32_t out_sb = 0;
    if (scode != 0) {
      out_sb = (negate ? PACKED_NEGATE : 0u) | ((sb & 0x40u) ? PACKED_SELECT : 0u) | scode;
      w0 = to_packed_order(canon(w0, negate));
      w1 = to_packed_order(canon(w1, negate));
    } else {
      w0 = w1 = 0x88888888u;                            // zero block: sixteen true zeros
    }
    uint8_t* piece = span + (kb_in / CHUNK_BLOCKS) * PIECE_BYTES;
    *reinterpret_cast<uint2*>(piece + piece_code_offset(kb_in % CHUNK_BLOCKS, r)) = make_uint2(w0, w1);
    piece[piece_scale_offset(kb_in % CHUNK_BLOCKS, r)] = (uint8_t)out_sb;
  }
  __syncthreads();
  uint4* dst = reinterpret_cast<uint4*>(packed + ((size_t)strip * g.k_chunks + c0) * PIECE_BYTES);
  for (int i = threadIdx.x; i < n_chunks * (PIECE_BYTES / 16); i += SPAN_THREADS) dst[i] = reinterpret_cast<const uint4*>(span)[i];
}

// Two nibbles of each 16-bit half of `w` at once: pair p of a word (elements 2p, 2p + 1), D1 = block_scale * element as
// exact bf16, zeros as +0 whatever the stored sign (the fused multiply-add with +0).  razer_decode.cuh describes the bits.
__device__ __forceinline__ void decode_pairs(uint32_t w, uint32_t ss2, uint32_t svp, uint32_t (&out)[4]) {
  constexpr uint32_t NEG = 0xC500C500u;                 // (-2048, -2048) as bf16x2
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const uint32_t n = (w >> (4 * p)) & 0x000F000Fu;
    const uint32_t u = and_or(n * ((1u << 6) + (1u << 12)), 0x81C081C0u, fma_relu_bf16x2(n, NEG, svp));
    out[p] = as_u32(__hfma2(as_bf162(u), as_bf162(ss2), as_bf162(0u)));
  }
}

template <bool FP32_OUT>
__global__ void __launch_bounds__(SPAN_THREADS) dequant_kernel(const uint8_t* __restrict__ packed, void* __restrict__ out, Geometry g,
                                                               DecodeParams p) {
  __shared__ __align__(16) uint8_t span[SPAN_BYTES];
  const int spans = (g.k_chunks + SPAN_CHUNKS - 1) / SPAN_CHUNKS;
  const int strip = (int)(blockIdx.x / (unsigned)spans), c0 = (int)(blockIdx.x % (unsigned)spans) * SPAN_CHUNKS;
  const int n_chunks = min(SPAN_CHUNKS, g.k_chunks - c0);
  const uint4* src = reinterpret_cast<const uint4*>(packed + ((size_t)strip * g.k_chunks + c0) * PIECE_BYTES);
  for (int i = threadIdx.x; i < n_chunks * (PIECE_BYTES / 16); i += SPAN_THREADS) reinterpret_cast<uint4*>(span)[i] = src[i];
  __syncthreads();
  const int k16 = g.K / 16;
#pragma unroll
  for (int i = 0; i < STRIP_ROWS * SPAN_BLOCKS / SPAN_THREADS; ++i) {
    const int b = (int)threadIdx.x + i * SPAN_THREADS, r = b / SPAN_BLOCKS, kb_in = b % SPAN_BLOCKS;
    const int n = strip * STRIP_ROWS + r, kb = c0 * CHUNK_BLOCKS + kb_in;
    if (n >= g.N || kb >= k16) continue;
    const uint8_t* piece = span + (kb_in / CHUNK_BLOCKS) * PIECE_BYTES;
    const uint2 c = *reinterpret_cast<const uint2*>(piece + piece_code_offset(kb_in % CHUNK_BLOCKS, r));
    const uint32_t sb = piece[piece_scale_offset(kb_in % CHUNK_BLOCKS, r)];
    // scale x 2^126 and special value x 2^-126 have at most four significant bits: exact upper halves of FP32 patterns
    const uint32_t s = (__float_as_uint(scale_value(sb & 0x3Fu) * 8.50705917e37f) >> 16) | ((sb & PACKED_NEGATE) << 9);
    const uint32_t v = __float_as_uint(p.sv_mag[(sb & PACKED_SELECT) ? 1 : 0] * 1.17549435e-38f) >> 16;
    uint32_t d[8];
    decode_pairs(c.x, s | (s << 16), v | (v << 16), *reinterpret_cast<uint32_t(*)[4]>(d));
    decode_pairs(c.y, s | (s << 16), v | (v << 16), *reinterpret_cast<uint32_t(*)[4]>(d + 4));
    const size_t at = ((size_t)n * k16 + kb) * 16;
    if (FP32_OUT) {
      float* o = reinterpret_cast<float*>(out) + at;
      if (reinterpret_cast<uintptr_t>(out) % 16 == 0) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          uint32_t v[8];
#pragma unroll
          for (int j = 0; j < 8; ++j)
            v[j] = __float_as_uint(__fmul_rn(p.tensor_scale, __uint_as_float((j & 1) ? d[4 * q + j / 2] & 0xFFFF0000u : d[4 * q + j / 2] << 16)));
          store32(o + 8 * q, v, aligned32(out));
        }
      } else {
#pragma unroll
        for (int j = 0; j < 16; ++j) o[j] = __fmul_rn(p.tensor_scale, __uint_as_float((j & 1) ? d[j / 2] & 0xFFFF0000u : d[j / 2] << 16));
      }
    } else {
      uint16_t* o = reinterpret_cast<uint16_t*>(out) + at;
      if (reinterpret_cast<uintptr_t>(out) % 16 == 0) {
        store32(o, d, aligned32(out));
      } else {
#pragma unroll
        for (int j = 0; j < 16; ++j) o[j] = (uint16_t)(d[j / 2] >> (16 * (j & 1)));
      }
    }
  }
}

// Activations in the interchange format (E4M3 scale, metadata bit 7 = sign of the special
// value, remapped code 0x8) -> bf16 block_scale * element, exact, zeros as +0.  One thread per block.  Bound by the DRAM
// writes; the element patterns are built two at a time (elements 4 apart share a word's halves) instead of one by one in
// FP32 (2048 x 8192: 22.6 -> 7.8 us).
__global__ void __launch_bounds__(256) decode_act_kernel(const uint8_t* __restrict__ codes, const uint8_t* __restrict__ scales,
                                                         __nv_bfloat16* __restrict__ out, long long n_blocks, float sv_mag) {
  const uint32_t svb = __float_as_uint(sv_mag * 1.17549435e-38f) >> 16;   // sv x 2^-126 as bf16: a multiple of 8
  const bool wide = aligned32(out);
  grid_dep_wait();
  grid_dep_launch();                                      // only now: the matmul behind reads packed weights at once
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n_blocks;
       t += (long long)gridDim.x * blockDim.x) {
    const uint2 c = *reinterpret_cast<const uint2*>(codes + t * 8);
    const uint32_t sb = scales[t];
    // an E4M3 scale reaches 448: x 2^118 here and x 2^8 behind keep every step inside bf16, and exact
    const uint32_t s = __float_as_uint(scale_value(sb & 0x7Fu) * 3.32306999e35f) >> 16;
    const uint32_t ss2 = s | (s << 16);
    const uint32_t sv8 = (svb | ((sb & 0x80u) << 8)) >> 3;             // times a nibble of 8: the signed special value
    uint32_t o[8];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint32_t w = h ? c.y : c.x;
      const uint32_t nz = ((w & 0x77777777u) + 0x77777777u) & 0x88888888u;
      const uint32_t s8 = w & ~nz & 0x88888888u;                       // code 8 = the special value
      const uint32_t wo = w ^ s8;
      uint32_t u[4];                                                   // pair p: elements p (low half) and p + 4
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        const uint32_t n = (wo >> (4 * p)) & 0x000F000Fu;
        const uint32_t v = ((n * ((1u << 6) + (1u << 12))) & 0x81C081C0u) + ((s8 >> (4 * p)) & 0x00080008u) * sv8;
        u[p] = mul_bf16x2(as_u32(__hfma2(as_bf162(v), as_bf162(ss2), as_bf162(0u))), 0x43804380u);
      }
      o[4 * h] = __byte_perm(u[0], u[1], 0x5410);
      o[4 * h + 1] = __byte_perm(u[2], u[3], 0x5410);
      o[4 * h + 2] = __byte_perm(u[0], u[1], 0x7632);
      o[4 * h + 3] = __byte_perm(u[2], u[3], 0x7632);
    }
    store32(out + t * 16, o, wide);
  }
}

static unsigned span_grid(const Geometry& g, int strips, int chunks = SPAN_CHUNKS) {
  return (unsigned)strips * (unsigned)((g.k_chunks + chunks - 1) / chunks);
}

static int grid_for(long long total, int threads) {
  long long b = (total + threads - 1) / threads;
  const long long cap = 148LL * 32;
  return (int)(b < 1 ? 1 : (b > cap ? cap : b));
}

// The matmul kernels are launched with programmatic stream serialization and begin to fetch packed weights
// before the kernel ahead of them in the stream is known to have finished (only activations, workspace and
// outputs wait for it).  An empty, ordinarily launched kernel behind the pack kernel makes that kernel, not
// the one that writes the weights, the matmul's predecessor: it cannot start before the weights are written
// and visible.
__global__ void pack_done_kernel() {}

int launch_pack(const razer_desc* d, const uint8_t* codes, const uint8_t* scales, void* packed,
                cudaStream_t st) {
  const Geometry g = make_geometry(d->N, d->K);
  // Short spans where long ones would leave SMs idle or most of a span's width empty, us against long ones: 256 x 256 2.5, 3.3;
  // 2048 x 1024 3.2, 3.6; 28672 x 256 5.3, 8.4.  Level at 2048 x 2048 (256 long spans) and 28672 x 512, long ones ahead at 1024 x 8192.
  const bool few = span_grid(g, g.strips()) < 2 * 148 || g.k_chunks <= 8;
  auto kern = few ? pack_kernel<FEW_CHUNKS> : pack_kernel<SPAN_CHUNKS>;
  kern<<<span_grid(g, g.strips(), few ? FEW_CHUNKS : SPAN_CHUNKS), SPAN_THREADS, 0, st>>>(codes, scales, (uint8_t*)packed, g, d->remap_code,
                                                                                      d->block / 16);
  count_launches(1);
  RAZER_TRY(check_cuda(cudaGetLastError(), "pack_kernel launch"));
  pack_done_kernel<<<1, 32, 0, st>>>();
  count_launches(1);
  return check_cuda(cudaGetLastError(), "pack_done_kernel launch");
}

int launch_dequant(const razer_desc* d, const void* packed, void* out, int fp32, cudaStream_t st) {
  const Geometry g = make_geometry(d->N, d->K);
  DecodeParams p{{d->sv_mag[0], d->sv_mag[1]}, d->tensor_scale, d->remap_code};
  const unsigned grid = span_grid(g, (g.N + STRIP_ROWS - 1) / STRIP_ROWS);
  auto kern = fp32 ? dequant_kernel<true> : dequant_kernel<false>;
  kern<<<grid, SPAN_THREADS, 0, st>>>((const uint8_t*)packed, out, g, p);
  count_launches(1);
  return check_cuda(cudaGetLastError(), "dequant_kernel launch");
}

// Up to a few hundred KB from pinned host memory, read over the bus, one 16-byte load a thread.  Bound by the bus's round trip;
// it replaces a copy by the copy engine, whose start and hand-over to the next kernel cost more than the transfer.
__global__ void __launch_bounds__(128) copy_from_host_kernel(const uint4* __restrict__ src, uint4* __restrict__ dst, int n) {
  const int i = (int)(blockIdx.x * blockDim.x + threadIdx.x);
  grid_dep_wait();                                        // source and destination may belong to the preceding kernel
  grid_dep_launch();                                      // only now: the matmul behind reads packed weights at once
  if (i < n) {
    uint4 v;                                              // volatile: the host may have changed it since an earlier call
    asm volatile("ld.volatile.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(src + i));
    dst[i] = v;
  }
}

int launch_copy_from_host(const void* src, void* dst, size_t bytes, cudaStream_t st) {
  const int n = (int)(bytes / 16);                                     // K is a multiple of 16 elements
  return launch_dependent("copy_from_host_kernel launch", copy_from_host_kernel, (n + 127) / 128, 128, 0, st, (const uint4*)src, (uint4*)dst, n);
}

int launch_decode_act(const uint8_t* codes, const uint8_t* scales, int M, int K, float sv_mag,
                      void* out, cudaStream_t st) {
  const long long nb = (long long)M * (K / 16);
  // dependent: it starts up while the kernel ahead (usually the quantizer that writes its input) drains
  return launch_dependent("decode_act_kernel launch", decode_act_kernel, grid_for(nb, 256), 256, 0, st, codes, scales, (__nv_bfloat16*)out,
                          nb, sv_mag);
}

}  // namespace razer

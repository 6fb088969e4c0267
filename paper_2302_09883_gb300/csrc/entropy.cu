// Lossless entropy stage over the records of a compressed state: order-0
// byte-wise rANS (range asymmetric numeral systems, J. Duda 2013), in the
// place where the paper's Sec. 2.3.2 applies a general-purpose byte
// compressor to the thresholded coefficients.
//
//   model  one table for the whole state: byte counts c_s over all records,
//          scaled to frequencies f_s summing to M = 2^12 (every occurring
//          byte gets max(1, floor(c_s M / N)), the largest f_s, first such
//          byte, takes up the difference to M); starts = prefix sums;
//   coder  32-bit state in [2^23, 2^31); a byte s is coded by emitting low
//          bytes while x >= 2^19 f_s, then x <- (x div f_s) 2^12 +
//          (x mod f_s) + start_s; a record is coded from its last byte to
//          its first, its stream is the final state (4 bytes, little endian)
//          followed by the emitted bytes in reverse order of emission, so
//          that decoding reads forward.
//   layout u32 npatch, u32 12, u16 freq[256]; per patch u32 record bytes,
//          u32 coded bytes; the streams in patch order.
//
// What bounds it: a record is one serial chain of state updates, so the time
// is (bytes of the longest record) x (latency of one update), and the work
// goes into that latency.  Thread per record (few to a warp, so that all SMs
// have some); coder: a byte's constants come in one 16-byte read that does
// not depend on the state, the division by f_s is a multiplication; decoder:
// a table by state slot, so one shared-memory read per byte; both take their
// input 16 or 4 bytes at a time.  1024 records of 18 KB: coder 4.1 -> 1.0 ms,
// check 7.0 -> 1.6 ms (before: run-time division, byte loads from L2).
// Everything between the record table and the coded size stays on the
// device.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "entropy.cuh"

namespace wcs {
namespace {

constexpr uint32_t SCALE = 12, M = 1u << SCALE, RL = 1u << 23;

// Constants of byte s for the coder.  Division of a 32-bit x by f as a
// multiplication (Granlund and Montgomery 1994, theorem 4.2): with k =
// ceil(log2 f) and m = floor(2^32 (2^k - f) / f) + 1, x div f is
// (hi(m x) + x) >> k, where hi is the high word; the sum fits 32 bits for the
// states x < 2^31, and f = 1 (k = 0, m = 1) is no special case.  The update
// 2^12 (x div f) + (x mod f) + start is x + q (2^12 - f) + start with the
// quotient q.  (That coders multiply instead of dividing is common practice,
// see Giesen's ryg_rans.)
struct __align__(16) CodeSym {
  uint32_t m;
  uint32_t lim;    // 2^19 f: x stays below it
  uint32_t start;
  uint32_t step;   // 2^12 - f | k << 16
};
struct Tables {
  CodeSym enc[256];
  uint32_t dec[M];  // per slot: f - 1 | (slot - start) << 12 | byte << 24
  uint16_t freq[256];
  unsigned long long hist[256];
  unsigned long long coded;       // bytes of all streams
  unsigned long long mismatches;
  unsigned int bad;               // a table or a slot that did not work out
};

// Byte counts: a block per record, each warp its own counts.
constexpr int HW = 8;
__global__ void __launch_bounds__(32 * HW) byte_hist(const unsigned char* arena, const unsigned long long* tab, int npatch,
                                                     unsigned long long* hist) {
  __shared__ unsigned int h[HW][256];
  for (int i = threadIdx.x; i < HW * 256; i += blockDim.x) h[0][i] = 0u;
  __syncthreads();
  unsigned int* mine = h[threadIdx.x >> 5];
  for (int p = blockIdx.x; p < npatch; p += gridDim.x) {
    const unsigned long long ent = tab[p];
    const uint4* r = reinterpret_cast<const uint4*>(arena + (ent >> 24));  // 16-byte multiples at 16-byte offsets
    const int n = int(ent & 0xffffffull) / 16;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      const uint4 v = __ldg(r + i);
      const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (w[k] == 0u) {  // runs of zeros are common: one count for four
          atomicAdd(mine, 4u);
          continue;
        }
#pragma unroll
        for (int b = 0; b < 4; ++b) atomicAdd(mine + ((w[k] >> (8 * b)) & 0xffu), 1u);
      }
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < 256; i += blockDim.x) {
    unsigned int s = 0u;
    for (int w = 0; w < HW; ++w) s += h[w][i];
    if (s) atomicAdd(&hist[i], (unsigned long long)s);
  }
}

// Bytes of a record's slot.  A coded byte costs at most 12 bits, so 24 for 16
// of the record and the state fit, with room for the coder to test its slot
// once per 16 bytes (which emit at most 32).
__host__ __device__ inline unsigned long long slot_bytes(unsigned long long nbytes) { return nbytes / 16 * 24 + 48; }

// Prefix sums (one block of NT threads) of the slots' sizes, where tab is
// given: where each slot starts; else of the stream lengths: where each
// stream goes.  Returns their sum.
template <int NT>
__device__ unsigned long long place(const unsigned long long* tab, const unsigned int* len, int npatch,
                                    unsigned long long* off, Tables* t) {
  __shared__ unsigned long long ws[32], carry;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) carry = 0ull;
  __syncthreads();
  for (int p0 = 0; p0 < npatch; p0 += NT) {
    const int p = p0 + threadIdx.x;
    const unsigned long long v = p < npatch ? (tab ? slot_bytes(tab[p] & 0xffffffull) : len[p]) : 0ull;
    if (p < npatch && v == 0ull) t->bad = 1u;
    unsigned long long s = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long u = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += u;
    }
    if (lane == 31) ws[warp] = s;
    __syncthreads();
    if (warp == 0) {
      unsigned long long q = lane < NT / 32 ? ws[lane] : 0ull;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long u = __shfl_up_sync(0xffffffffu, q, o);
        if (lane >= o) q += u;
      }
      ws[lane] = q;
    }
    __syncthreads();
    const unsigned long long base = carry + (warp ? ws[warp - 1] : 0ull);
    if (p < npatch) off[p] = base + s - v;
    __syncthreads();
    if (threadIdx.x == NT - 1) carry = base + s;
    __syncthreads();
  }
  return carry;
}
__global__ void __launch_bounds__(1024) place_streams(const unsigned int* len, int npatch, unsigned long long* dst_off,
                                                      Tables* t) {
  const unsigned long long sum = place<1024>(nullptr, len, npatch, dst_off, t);
  if (threadIdx.x == 0) t->coded = sum;
}

// Frequencies summing to 2^12 from the byte counts (see the file comment) and
// the coder's and decoder's tables; one block of 256 threads.  A second block
// places the records' slots meanwhile.
__global__ void __launch_bounds__(256) build_tables(Tables* t, const unsigned long long* tab, int npatch,
                                                    unsigned long long* slot_off) {
  if (blockIdx.x == 1) {
    (void)place<256>(tab, nullptr, npatch, slot_off, t);
    return;
  }
  __shared__ uint32_t f[256], ws[8];
  __shared__ unsigned long long wn[8];
  __shared__ uint32_t wb[8];
  const int s = threadIdx.x, lane = s & 31, warp = s >> 5;
  const unsigned long long cnt = t->hist[s];
  unsigned long long N = cnt;
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) N += __shfl_xor_sync(0xffffffffu, N, o);
  if (lane == 0) wn[warp] = N;
  __syncthreads();
  N = 0;
  for (int k = 0; k < 8; ++k) N += wn[k];
  const unsigned long long v = N && cnt ? cnt * M / N : 0ull;
  uint32_t fs = uint32_t(cnt && v < 1 ? 1ull : v);
  // their sum, and the largest (the first such byte): 13 bits of f, then 255 - s
  uint32_t sum = fs, big = (fs << 8) | uint32_t(255 - s);
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) {
    sum += __shfl_xor_sync(0xffffffffu, sum, o);
    const uint32_t u = __shfl_xor_sync(0xffffffffu, big, o);
    big = u > big ? u : big;
  }
  if (lane == 0) {
    ws[warp] = sum;
    wb[warp] = big;
  }
  __syncthreads();
  sum = 0;
  big = 0;
  for (int k = 0; k < 8; ++k) {
    sum += ws[k];
    big = wb[k] > big ? wb[k] : big;
  }
  if (s == 255 - int(big & 0xffu)) {  // (no byte at all: byte 0 gets everything)
    const int fb = int(fs) + int(M) - int(sum);
    if (fb < 1) t->bad = 1u;
    fs = uint32_t(fb < 1 ? 1 : fb);
  }
  f[s] = fs;
  __syncthreads();
  uint32_t cs = 0;
  for (int k = 0; k < s; ++k) cs += f[k];
  if (s == 255 && cs + fs != M) t->bad = 1u;
  t->freq[s] = uint16_t(fs);
  if (fs > 0) {
    uint32_t k = 0;
    while ((1u << k) < fs) ++k;
    CodeSym e;
    e.m = uint32_t((((1ull << k) - fs) << 32) / fs + 1);
    e.lim = ((RL >> SCALE) << 8) * fs;
    e.start = cs;
    e.step = (M - fs) | k << 16;
    t->enc[s] = e;  // (bytes that do not occur have none)
  }
  for (uint32_t k = 0; k < fs && cs + k < M; ++k) t->dec[cs + k] = (fs - 1) | (k << 12) | (uint32_t(s) << 24);
}

// Codes record p (a thread each) into its slot, downwards from the slot's
// end; coded length to len[p].  0 in len[p] signals an overflowing slot
// (cannot happen with the slot sizes used).
__global__ void __launch_bounds__(256) rans_encode_records(const unsigned char* arena, const unsigned long long* tab,
                                                           int npatch, int lanes, const Tables* __restrict__ t,
                                                           const unsigned long long* slot_off, unsigned char* out,
                                                           unsigned int* len) {
  __shared__ CodeSym e[256];
  for (int i = threadIdx.x; i < 256; i += blockDim.x) e[i] = t->enc[i];
  __syncthreads();
  const int lane = threadIdx.x & 31, p = (blockIdx.x * int(blockDim.x >> 5) + int(threadIdx.x >> 5)) * lanes + lane;
  if (lane >= lanes || p >= npatch) return;
  const unsigned long long ent = tab[p];
  const uint4* r = reinterpret_cast<const uint4*>(arena + (ent >> 24));
  const int n16 = int(ent & 0xffffffull) / 16;
  unsigned char* const lo = out + slot_off[p] + 4;
  unsigned char* const end = out + slot_off[p] + slot_bytes(ent & 0xffffffull);
  unsigned char* w = end;
  uint32_t x = RL;
  // four bytes' constants are read before the states of the four before them
  // (the byte stores could alias them as far as the compiler knows, and would
  // put each read on the chain)
  uint4 cur = n16 > 0 ? __ldg(r + n16 - 1) : make_uint4(0, 0, 0, 0);
  CodeSym c[4];
  auto fetch = [&](uint32_t v) {
#pragma unroll
    for (int b = 0; b < 4; ++b) c[b] = e[(v >> (24 - 8 * b)) & 0xffu];
  };
  fetch(cur.w);
  for (int i = n16 - 1; i >= 0; --i) {
    const uint4 nxt = i > 0 ? __ldg(r + i - 1) : cur;
    if (w - 32 < lo) {  // 16 bytes emit at most 32
      len[p] = 0u;
      return;
    }
    const uint32_t q4[4] = {cur.z, cur.y, cur.x, nxt.w};  // the words after the one in c
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      CodeSym now[4];
#pragma unroll
      for (int b = 0; b < 4; ++b) now[b] = c[b];
      fetch(q4[k]);
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const CodeSym s = now[b];
        // x has to come below lim: by one byte, or by two where it is at 2^8 lim
        // or above (f < 16: 2^27 f is past every state otherwise), both known
        // from x at once
        const bool e1 = x >= s.lim, e2 = s.lim < RL && x >= s.lim << 8;
        if (e1) *(w - 1) = (unsigned char)x;
        if (e2) *(w - 2) = (unsigned char)(x >> 8);
        w -= (e1 ? 1 : 0) + (e2 ? 1 : 0);
        x = e2 ? x >> 16 : (e1 ? x >> 8 : x);
        const uint32_t q = (__umulhi(x, s.m) + x) >> (s.step >> 16);
        x = q * (s.step & 0xffffu) + (x + s.start);
      }
    }
    cur = nxt;
  }
  w -= 4;
  for (int k = 0; k < 4; ++k) w[k] = (unsigned char)(x >> (8 * k));
  len[p] = unsigned(end - w);
}

// The layout's head and the streams at their places (block per patch).
__global__ void __launch_bounds__(256) gather_streams(const unsigned char* slots, const unsigned long long* tab,
                                                      const unsigned long long* slot_off, const unsigned int* len,
                                                      const unsigned long long* dst_off, const Tables* t,
                                                      unsigned char* dst, int npatch) {
  const int p = blockIdx.x;
  const size_t head = 8 + 512 + size_t(8) * npatch;
  if (p == 0) {
    if (threadIdx.x == 0) {
      reinterpret_cast<uint32_t*>(dst)[0] = uint32_t(npatch);
      reinterpret_cast<uint32_t*>(dst)[1] = SCALE;
    }
    for (int i = threadIdx.x; i < 256; i += blockDim.x) reinterpret_cast<uint16_t*>(dst + 8)[i] = t->freq[i];
  }
  const unsigned long long ent = tab[p];
  const unsigned int n = len[p];
  if (threadIdx.x < 2)
    reinterpret_cast<uint32_t*>(dst + 520 + size_t(8) * p)[threadIdx.x] = threadIdx.x == 0 ? uint32_t(ent & 0xffffffull) : n;
  const unsigned char* s = slots + slot_off[p] + slot_bytes(ent & 0xffffffull) - n;
  unsigned char* d = dst + head + dst_off[p];
#pragma unroll 4
  for (unsigned int i = threadIdx.x; i < n; i += blockDim.x) d[i] = s[i];
}

// Decodes every stream of the layout (thread per patch) and counts the bytes
// that differ from the records.
__global__ void __launch_bounds__(256) rans_check(const unsigned char* coded, unsigned long long coded_bytes,
                                                  const unsigned long long* dst_off, const unsigned int* len,
                                                  const unsigned char* arena, const unsigned long long* tab, int npatch,
                                                  int lanes, Tables* t) {
  __shared__ uint32_t dec[M];
  for (int i = threadIdx.x; i < int(M); i += blockDim.x) dec[i] = t->dec[i];
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int p = (blockIdx.x * int(blockDim.x >> 5) + warp) * lanes + lane;
  if (lane >= lanes || p >= npatch) return;
  const unsigned int nin = len[p];
  const unsigned long long ent = tab[p];
  const uint4* r = reinterpret_cast<const uint4*>(arena + (ent >> 24));
  const int n16 = int(ent & 0xffffffull) / 16;
  if (nin < 4) {
    atomicAdd(&t->mismatches, (unsigned long long)(16 * n16 + 1));
    return;
  }
  // the coded streams by 4-byte words: w0 holds byte `pos`, w1 the bytes after
  // it, w2 is on its way; words past the stream's end (its successor's, or the
  // padding) are never consumed
  const unsigned long long at = dst_off[p];
  const uint32_t* in = reinterpret_cast<const uint32_t*>(coded);
  const unsigned int nword = (unsigned int)((coded_bytes + 3) / 4 - at / 4);
  in += at / 4;
  unsigned int q = 3;  // next word to read
  auto word = [&](unsigned int k) -> uint32_t { return k < nword ? __ldg(in + k) : 0u; };
  uint32_t w0 = word(0), w1 = word(1), w2 = word(2);
  unsigned int pos = unsigned(at & 3ull);
  const unsigned int first = pos;
  uint32_t x = __funnelshift_r(w0, w1, 8 * pos);
  pos += 4;
  w0 = w1;
  w1 = w2;
  w2 = word(q++);
  unsigned int wrong = 0;
  uint4 cur = n16 > 0 ? __ldg(r) : make_uint4(0, 0, 0, 0);
  for (int i = 0; i < n16; ++i) {
    const uint4 nxt = i + 1 < n16 ? __ldg(r + i + 1) : cur;
    const uint32_t q4[4] = {cur.x, cur.y, cur.z, cur.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      uint32_t got = 0u;
#pragma unroll
      for (int b = 0; b < 32; b += 8) {
        const uint32_t by = __funnelshift_r(w0, w1, 8 * (pos & 3u));  // the next bytes, low first
        const uint32_t d = dec[x & (M - 1)];
        x = ((d & 0xfffu) + 1u) * (x >> SCALE) + ((d >> 12) & 0xfffu);
        got |= (d >> 24) << b;
        // x >= 2^11 after a step: two bytes at most bring it back to 2^23
        const uint32_t x1 = __byte_perm(x, by, 0x2104);  // x << 8 | first byte
        const uint32_t x2 = __byte_perm(x, by, 0x1045);  // x << 16 | first << 8 | second
        const bool one = x < RL, two = x < (RL >> 8);
        x = two ? x2 : (one ? x1 : x);
        const unsigned int np = pos + (two ? 2u : (one ? 1u : 0u));
        if ((pos ^ np) & 4u) {
          w0 = w1;
          w1 = w2;
          w2 = word(q++);
        }
        pos = np;
      }
      const uint32_t diff = got ^ q4[k];
      wrong += (diff & 0xffu ? 1u : 0u) + (diff & 0xff00u ? 1u : 0u) + (diff & 0xff0000u ? 1u : 0u) + (diff >> 24 ? 1u : 0u);
    }
    cur = nxt;
  }
  if (pos - first != nin) ++wrong;  // the stream ends with its record
  if (wrong) atomicAdd(&t->mismatches, (unsigned long long)wrong);
}

}  // namespace

cudaError_t entropy_code_state(const unsigned char* arena, const unsigned long long* tab, int npatch,
                               unsigned long long live, cudaStream_t stream, entropy_sink sink, void* user,
                               long long* nbytes, unsigned long long* mismatches) {
  cudaError_t e;
  unsigned char* work = nullptr;   // tables, places of the slots and streams, lengths, slots
  unsigned char* coded = nullptr;  // the layout
  auto done = [&](cudaError_t r) {
    cudaFree(work);
    cudaFree(coded);
    return r;
  };
  const size_t o_at = (sizeof(Tables) + 255) / 256 * 256, o_dst = o_at + size_t(npatch) * 8, o_len = o_dst + size_t(npatch) * 8;
  const size_t o_slot = (o_len + size_t(npatch) * 4 + 255) / 256 * 256;
  // the slots of all records: 24 bytes for 16, and 48 each
  if ((e = cudaMalloc(&work, o_slot + size_t(live / 16 * 24) + size_t(npatch) * 48)) != cudaSuccess) return done(e);
  Tables* t = reinterpret_cast<Tables*>(work);
  unsigned long long* at = reinterpret_cast<unsigned long long*>(work + o_at);
  unsigned long long* dst = reinterpret_cast<unsigned long long*>(work + o_dst);
  unsigned int* len = reinterpret_cast<unsigned int*>(work + o_len);
  unsigned char* slots = work + o_slot;
  int dev = 0, nsm = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  // records per warp: one while that leaves at most 16 warps per SM.  Each is
  // a chain whose latency, not the issue rate, is the time, and records that
  // share a warp wait for each other's loads (7 to a warp: 0.92 ms and 2.3 ms
  // for the coder and the check, one: 0.95 ms and 1.6 ms)
  const int lanes = std::min(32, std::max(1, (npatch + 16 * nsm - 1) / (16 * nsm)));
  const int nwarp = (npatch + lanes - 1) / lanes, wpb = std::min(8, std::max(1, (nwarp + nsm - 1) / nsm));
  const int nblk = (nwarp + wpb - 1) / wpb;
  const size_t head = 8 + 512 + size_t(8) * npatch;
  if ((e = cudaMemsetAsync(t->hist, 0, sizeof(Tables) - (reinterpret_cast<unsigned char*>(t->hist) - work), stream)) != cudaSuccess)
    return done(e);
  byte_hist<<<std::min(npatch, 8 * nsm), 32 * HW, 0, stream>>>(arena, tab, npatch, t->hist);
  build_tables<<<2, 256, 0, stream>>>(t, tab, npatch, at);
  rans_encode_records<<<nblk, 32 * wpb, 0, stream>>>(arena, tab, npatch, lanes, t, at, slots, len);
  place_streams<<<1, 1024, 0, stream>>>(len, npatch, dst, t);
  struct { unsigned long long coded, mismatches; unsigned int bad; } res;
  const size_t o_res = reinterpret_cast<unsigned char*>(&t->coded) - work;
  if ((e = cudaGetLastError()) != cudaSuccess ||
      (e = cudaMemcpyAsync(&res, work + o_res, sizeof(res), cudaMemcpyDeviceToHost, stream)) != cudaSuccess ||
      (e = cudaStreamSynchronize(stream)) != cudaSuccess)
    return done(e);
  if (res.bad) return done(cudaErrorInvalidValue);
  const size_t total = head + size_t(res.coded);
  if ((e = cudaMalloc(&coded, (total + 7) / 4 * 4)) != cudaSuccess) return done(e);
  gather_streams<<<npatch, 256, 0, stream>>>(slots, tab, at, len, dst, t, coded, npatch);
  rans_check<<<nblk, 32 * wpb, 0, stream>>>(coded + head, res.coded, dst, len, arena, tab, npatch, lanes, t);
  if ((e = cudaGetLastError()) != cudaSuccess) return done(e);
  if ((e = cudaMemcpyAsync(&res, work + o_res, sizeof(res), cudaMemcpyDeviceToHost, stream)) != cudaSuccess ||
      (e = cudaStreamSynchronize(stream)) != cudaSuccess)
    return done(e);
  *mismatches = res.mismatches;
  if (res.mismatches) return done(cudaSuccess);  // the caller's memory stays as it is
  *nbytes = (long long)total;
  void* to = sink ? sink(user, (long long)total) : nullptr;
  if (to && ((e = cudaMemcpyAsync(to, coded, total, cudaMemcpyDeviceToHost, stream)) != cudaSuccess ||
             (e = cudaStreamSynchronize(stream)) != cudaSuccess))
    return done(e);
  return done(cudaSuccess);
}

}  // namespace wcs

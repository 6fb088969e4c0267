// The compressed-patch time step in three dimensions: D3Q19 BGK on cubic
// patches of P cells ((P+1)^3 nodes, folded BL5/3, Sec. 2.1.2 and 3.1.1),
// FP32 arithmetic.
//
// One patch of 19 fields of (P+1)^3 values (2.7 MB at P = 32) does not fit in
// shared memory, so the kernel is persistent (one CTA per SM, three for
// 16-cell patches, patches taken in a stride) and each CTA owns a scratch slot
// in global memory: 19 cubes of (P+3)^3 values, the nodes plus a ghost layer.
// A field's cube is free once its new values are gathered; its export faces
// and its section of the new record go there (a record buffer of its own
// beside the cubes took as much memory again: 921 KB a slot for 16 cells, 6.1 MB
// for 32, now 530 KB and 3.3 MB; six steps of 256^3 45.1 -> 44.7 ms, twelve of
// 176 x 80 x 112 with 16-cell patches 7.75 -> 7.72, 64 such patches alone 345
// us a step before and after).
// Per patch:
//   decode:   for every field, the record section -> shared tile -> inverse
//             tensor lifting (z, y, x lines, one thread per line) -> scratch;
//   scheme:   ghost layer from the neighbours' rings, BGK collision of every
//             node in scratch (thread per node, 19 values in registers);
//   encode:   for every field, the pull-streamed values (the scratch read at
//             x - c_i) -> shared tile -> forward lifting x, y, then z fused
//             with the threshold (a warp holds 32 z-lines; one ballot per
//             node row gives the row's mask word) -> quantise, scans, record
//             section to the field's scratch -> re-decode in the tile -> the
//             six export layers of the field to its scratch;
//   export:   collision of the export layers, the inward populations to the
//             ring (6 faces x 5 populations, 12 edges x 1: D3Q19 has no
//             corner velocities), then one allocation in the arena and the
//             record copied there.
// The record format, mask order and quantisation are those of the 2-D path
// with three axes (rows are (y, z) pairs, z slowest, the shared face x = P
// follows as one bit per row; edge coefficients are those on a face of the
// patch).
#pragma once
#include "common.cuh"

#include <type_traits>

namespace wcs {

// D3Q19 velocity components (0 rest, 1..6 = +x -x +y -y +z -z, then the
// diagonals 7 (+,+,0) 8 (-,-,0) 9 (+,-,0) 10 (-,+,0) 11 (+,0,+) 12 (-,0,-)
// 13 (+,0,-) 14 (-,0,+) 15 (0,+,+) 16 (0,-,-) 17 (0,+,-) 18 (0,-,+)).
__host__ __device__ __forceinline__ constexpr int d3_cx(int i) {
  return (i == 1 || i == 7 || i == 9 || i == 11 || i == 13) ? 1 : ((i == 2 || i == 8 || i == 10 || i == 12 || i == 14) ? -1 : 0);
}
__host__ __device__ __forceinline__ constexpr int d3_cy(int i) {
  return (i == 3 || i == 7 || i == 10 || i == 15 || i == 17) ? 1 : ((i == 4 || i == 8 || i == 9 || i == 16 || i == 18) ? -1 : 0);
}
__host__ __device__ __forceinline__ constexpr int d3_cz(int i) {
  return (i == 5 || i == 11 || i == 14 || i == 15 || i == 18) ? 1 : ((i == 6 || i == 12 || i == 13 || i == 16 || i == 17) ? -1 : 0);
}
__host__ __device__ __forceinline__ constexpr int d3_c(int i, int a) { return a == 0 ? d3_cx(i) : (a == 1 ? d3_cy(i) : d3_cz(i)); }

template <typename T> __device__ __forceinline__ T d3q19_w(int i) {
  return i == 0 ? T(1.0 / 3.0) : (i <= 6 ? T(1.0 / 18.0) : T(1.0 / 36.0));
}

// c_i . u: the axis terms in the order x, y, z, the first one with its sign.
template <typename T> __device__ __forceinline__ T d3q19_cu(int i, T ux, T uy, T uz) {
  const T u[3] = {ux, uy, uz};
  T s = T(0);
  bool first = true;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int c = d3_c(i, a);
    if (c == 0) continue;
    if (first) s = c > 0 ? u[a] : -u[a];
    else s = c > 0 ? s + u[a] : s - u[a];
    first = false;
  }
  return s;
}

template <typename T> __device__ __forceinline__ void d3q19_equilibrium(T rho, T ux, T uy, T uz, T* feq) {
  const T usq = (ux * ux + uy * uy) + uz * uz;
#pragma unroll
  for (int i = 0; i < 19; ++i) {
    const T cu = d3q19_cu<T>(i, ux, uy, uz);
    T t = T(1) + T(3) * cu;
    t = t + (T(4.5) * cu) * cu;
    t = t - T(1.5) * usq;
    feq[i] = (d3q19_w<T>(i) * rho) * t;
  }
}

// In-place BGK collision of one node: rho = f_0 + ... + f_18 left to right,
// j_a over i = 1..18 in order (first non-zero term with its sign).
template <typename T> __device__ __forceinline__ void d3q19_collide(T* f, T omega) {
  T rho = f[0];
#pragma unroll
  for (int i = 1; i < 19; ++i) rho = rho + f[i];
  T u[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    T j = T(0);
    bool first = true;
#pragma unroll
    for (int i = 1; i < 19; ++i) {
      const int c = d3_c(i, a);
      if (c == 0) continue;
      if (first) j = c > 0 ? f[i] : -f[i];
      else j = c > 0 ? j + f[i] : j - f[i];
      first = false;
    }
    u[a] = j / rho;
  }
  T feq[19];
  d3q19_equilibrium<T>(rho, u[0], u[1], u[2], feq);
#pragma unroll
  for (int i = 0; i < 19; ++i) f[i] = f[i] - omega * (f[i] - feq[i]);
}

// The five populations of ring face phi (0: x = 1 layer, c_x = -1; 1: x =
// P-1, c_x = +1; 2: y = 1, c_y = -1; 3: y = P-1, c_y = +1; 4: z = 1, c_z =
// -1; 5: z = P-1, c_z = +1), in increasing population order.
__host__ __device__ __forceinline__ constexpr int d3_face_pop(int phi, int k) {
  return phi == 0 ? (k == 0 ? 2 : k == 1 ? 8 : k == 2 ? 10 : k == 3 ? 12 : 14)
       : phi == 1 ? (k == 0 ? 1 : k == 1 ? 7 : k == 2 ? 9 : k == 3 ? 11 : 13)
       : phi == 2 ? (k == 0 ? 4 : k == 1 ? 8 : k == 2 ? 9 : k == 3 ? 16 : 18)
       : phi == 3 ? (k == 0 ? 3 : k == 1 ? 7 : k == 2 ? 10 : k == 3 ? 15 : 17)
       : phi == 4 ? (k == 0 ? 6 : k == 1 ? 12 : k == 2 ? 13 : k == 3 ? 16 : 17)
                  : (k == 0 ? 5 : k == 1 ? 11 : k == 2 ? 14 : k == 3 ? 15 : 18);
}

__device__ __forceinline__ unsigned int ldg_u32(const unsigned char* p) {
  return __ldg(reinterpret_cast<const unsigned int*>(p));
}

struct Patch3Args {
  int npx, npy, npz;
  long long step;
  const unsigned char* arena_in;
  const unsigned long long* tab_in;  // (offset << 24) | nbytes per patch
  unsigned char* arena_out;
  unsigned long long* tab_out;
  unsigned long long cap_out;
  const float* ring_in;
  float* ring_out;
  Ctl* ctl;
  int cur_out, cur_rst;
  double* pstats;             // npatch * 19 coarse-block sums
  float* coarse_lo;           // hi + lo coarse storage: npatch * 19 * NC lo parts (null: off)
  double* pstats_lo;          //   npatch * 19 sums of them, scaled like pstats
  double* hbuf;               //   per CTA: hbuf_doubles of FP64 work space
  unsigned long long hbuf_doubles;
  const double* band_factor;  // threshold multiplier per band
  double eps, eps_edge;
  const double* eps_patch;    // optional per-patch threshold constant
  float omega;
  float* scratch;             // per CTA: slot_floats floats, 19 cubes
  unsigned long long slot_floats;
  const double* macro[4];     // INIT: rho, ux, uy, uz on the global node grid
  const void* state;          // INIT from a dense state instead (19 planes
                              // [z][y][x]; null: macro fields)
  int state_dtype;            // 0 double, 1 float
  void* dense;                // EXPORT: [field][z][y][x] over the global nodes
  int dense_dtype;            // 0 double, 1 float
  int field_sel;              // EXPORT: one field or -1 for all
  long long G0, G1, G2;       // global nodes per axis (periodic: cells)
  unsigned int flags;         // record flags word
  // learned threshold (FEAT kernels)
  float* feat;                // per patch 42 features of the new state
  float feat_inv_cnt[24];     // per group: 1 / (fields x nodes of the group)
  const float* mlp_wt;        // network in kernel layout (W1, W2 transposed)
  double* eps_next;           // the eps of the next step, per patch
  double eps_lo, eps_hi;      // clamp of the network's eps; non-finite -> eps
};

template <int P, int L, int ST> struct Cfg3 {
  static constexpr int F = 19;
  static constexpr int E = P + 1, E2 = E * E, E3 = E2 * E;
  static constexpr int EG = E + 2, EG2 = EG * EG, EG3 = EG2 * EG;
  // Threads: the line passes have E^2 lines and the z passes E + FG warp
  // tasks, so 18 warps take a 33^3 patch in two full rounds (1024 threads
  // took two as well, the second with 65 lines) with registers to spare; 10
  // warps take a 17^3 patch, and three such CTAs share an SM: with one, two and
  // three a step of 160^3 takes 2289, 1552, 1416 us (slots of 79, 158, 238 MB in
  // all, BF16), of 176 x 80 x 112 (385 patches, FP32) 886, 683, 570 (81, 161, 204
  // MB), of 64^3 (64 patches, one per SM) 327, 338, 345.
  static constexpr int NT = P >= 32 ? 576 : 320, NWARP = NT / 32;
  static constexpr int MINB = P >= 32 ? 1 : 3;
  static constexpr int NC1 = (P >> L) + 1, NC = NC1 * NC1 * NC1;
  static constexpr int WR = (P + 31) / 32;       // mask words per x-row
  static constexpr int NRW = E2 * WR;            // row words
  static constexpr int NCW = (E2 + 31) / 32;     // words of the face x = P
  static constexpr int NW = NRW + NCW;
  static constexpr int NPW = (NW + 31) / 32;
  static constexpr int NB = (L + 1) * (L + 1) * (L + 1);
  static constexpr bool QUANT = ST == ST_BF16 || ST == ST_I8;
  typedef typename StoreType<ST>::type S;
  static constexpr int SB = sizeof(S);
  static constexpr int RING = 30 * E2 + 12 * E;  // floats exported per patch
  static constexpr int HDR = (16 + 16 * F + 15) / 16 * 16;
  static constexpr int RG = E * WR;              // row groups of the fused z pass
  static constexpr int FG = (E + 31) / 32;       // face groups (x = P)
  static constexpr int NCK = (NW + 31) / 32;     // chunks of 32 mask words
  // Scratch of a field, PITCH floats: its cube with the ghosts; once the new
  // values are gathered, its six export faces and, FACES floats on, its
  // section of the new record, at most SECMAX bytes (coarse block, band mask
  // and scales, presence, all words, every survivor).
  static constexpr int NINT = (P - 1) * (P - 1) * (P - 1);  // nodes not on a face
  static constexpr int SECMAX =
      (4 * NC + (QUANT ? 8 + 4 * NB : 0) + 4 * NPW + 4 * NW + 7 + 4 * (E3 - NINT) + SB * NINT + 15) / 16 * 16;
  static constexpr int FACES = (6 * E2 + 3) / 4 * 4;
  static constexpr int PITCH = ((EG3 > FACES + SECMAX / 4 ? EG3 : FACES + SECMAX / 4) + 3) / 4 * 4;
  // shared memory carve-up (bytes)
  static constexpr size_t OFF_MW = (size_t(E3) * 4 + 7) / 8 * 8;  // per mask word: the word, the survivors before it
  static constexpr size_t OFF_BMAX = OFF_MW + size_t(NW) * 8;
  static constexpr size_t OFF_SCL = OFF_BMAX + size_t(NB) * 4;
  static constexpr size_t OFF_SINV = OFF_SCL + size_t(NB) * 4;
  static constexpr size_t OFF_TAU = OFF_SINV + size_t(NB) * 4;
  static constexpr size_t OFF_WS = OFF_TAU + size_t(2 * NB) * 4;  // scan scratch: totals of the chunks of 32 words
  static constexpr size_t OFF_MISC = OFF_WS + 2 * 64 * 4;
  static constexpr size_t OFF_HEAD = OFF_MISC + 64 * 4;  // per field: section offset, words, edges, band mask (encode: its row of the record's table)
  static constexpr size_t SMEM = OFF_HEAD + size_t(F) * 5 * 4;
  static_assert(SMEM <= 232448, "patch does not fit in shared memory");
  // learned-threshold kernels: per z-line class sums, band totals, the network
  static constexpr int NG = 7 * L, NIN = 2 * NG;
  static constexpr int MLP_NP = 64 * NIN + 64 + 64 * 64 + 64 + 64 + 1;
  static constexpr size_t OFF_LACC = (SMEM + 15) / 16 * 16;                       // E2 x (L+1) x {e, m}
  static constexpr size_t OFF_BAND = OFF_LACC + size_t(E2) * (L + 1) * 2 * 4;    // NB doubles + NB floats
  static constexpr size_t OFF_FV = (OFF_BAND + size_t(NB) * 12 + 15) / 16 * 16;   // NIN features
  static constexpr size_t OFF_W = (OFF_FV + size_t(NIN) * 4 + 15) / 16 * 16;
  static constexpr size_t SMEM_FEAT = OFF_W + size_t(MLP_NP) * 4;
  static_assert(SMEM_FEAT <= 232448, "the learned-threshold patch does not fit in shared memory");
  static_assert(E3 < 65536, "survivor ranks are kept in 16 bits");
  static_assert(NB <= 64, "band masks are 64 bits");
  static_assert(WR == 1 && NCK <= 64 && NPW == NCK && NW <= 2 * NT, "a word per row, at most two chunk totals per lane");
};

// Edge-coefficient bits of mask word w (a node on a face of the patch) and
// the valid bits (nodes, not padding).
template <int P, int E, int WR> __device__ __forceinline__ unsigned int word3_valid(int w) {
  constexpr int NRW = E * E * WR;
  if (w < NRW) {
    const int n = P - 32 * (w % WR);
    return n >= 32 ? 0xffffffffu : ((1u << n) - 1u);
  }
  const int n = E * E - 32 * (w - NRW);
  return n >= 32 ? 0xffffffffu : ((1u << n) - 1u);
}
template <int P, int E, int WR> __device__ __forceinline__ unsigned int word3_edges(int w) {
  constexpr int NRW = E * E * WR;
  const unsigned int vm = word3_valid<P, E, WR>(w);
  if (w < NRW) {
    const int r = w / WR, h = w - r * WR, y = r % E, z = r / E;
    if (y == 0 || y == P || z == 0 || z == P) return vm;
    return h == 0 ? 1u : 0u;  // x = 0
  }
  return vm;  // the face x = P
}

// Exclusive prefix of the chunk totals in ws (n of them, at most 64), value of
// chunk k; `total` gets their sum.  Every warp does this by itself.
__device__ __forceinline__ unsigned int chunk_base(const unsigned int* ws, int n, int k, unsigned int& total) {
  const int lane = threadIdx.x & 31;
  const unsigned int a = lane < n ? ws[lane] : 0u, b = 32 + lane < n ? ws[32 + lane] : 0u;
  const unsigned int ia = warp_incl_scan(a), ib = warp_incl_scan(b);
  const unsigned int ta = __shfl_sync(0xffffffffu, ia, 31);
  total = ta + __shfl_sync(0xffffffffu, ib, 31);
  const unsigned int ea = __shfl_sync(0xffffffffu, ia - a, k & 31), eb = __shfl_sync(0xffffffffu, ib - b, k & 31);
  return k < 32 ? ea : ta + eb;
}

// hi + lo coarse storage (Sec. 2.1.2, eq. conservation): the coarse block of
// one field formed a second time, in FP64, from its FP32 nodes in the tile
// ([z][y][x]); the x pass on every line keeps the coarse-x values (hb,
// [ix][z][y]), the y pass on those keeps the coarse-y ones (hb + NC1 E^2,
// [ix][iy][z]), the z pass leaves the block in c64 ([iz][iy][ix]).  The
// FP32 path's lifting in FP64, so the oracle's FP64 transform bit for bit.
// hb lives in global memory (a few tens of KB per CTA, L2-resident); all
// threads of the block call this.
template <int P, int L, int NT>
__device__ __noinline__ void coarse3_fp64(const float* tile, double* hb, double* c64) {
  constexpr int E = P + 1, E2 = E * E, NC1 = (P >> L) + 1;
  const int tid = threadIdx.x;
  double* hb2 = hb + NC1 * E2;
  for (int l = tid; l < E2; l += NT) {
    const int z = l / E, y = l - z * E;
    double v[E];
#pragma unroll
    for (int x = 0; x < E; ++x) v[x] = double(tile[z * E2 + y * E + x]);
    fwd_levels<WV_BL53, P, 1, L, double>(v);
#pragma unroll
    for (int ix = 0; ix < NC1; ++ix) hb[(ix * E + z) * E + y] = v[ix << L];
  }
  __syncthreads();
  for (int t = tid; t < NC1 * E; t += NT) {
    const int ix = t / E, z = t - ix * E;
    double v[E];
#pragma unroll
    for (int y = 0; y < E; ++y) v[y] = hb[(ix * E + z) * E + y];
    fwd_levels<WV_BL53, P, 1, L, double>(v);
#pragma unroll
    for (int iy = 0; iy < NC1; ++iy) hb2[(ix * NC1 + iy) * E + z] = v[iy << L];
  }
  __syncthreads();
  for (int t = tid; t < NC1 * NC1; t += NT) {
    const int ix = t / NC1, iy = t - ix * NC1;
    double v[E];
#pragma unroll
    for (int z = 0; z < E; ++z) v[z] = hb2[(ix * NC1 + iy) * E + z];
    fwd_levels<WV_BL53, P, 1, L, double>(v);
#pragma unroll
    for (int iz = 0; iz < NC1; ++iz) c64[(iz * NC1 + iy) * NC1 + ix] = v[iz << L];
  }
  __syncthreads();
}

// The record into the arena at dst: its first 16 bytes, the fields' rows
// (head, 4 ints each) and their sections from the scratch slot Sc.  Out of
// line, and two pieces in flight for 16-cell patches: its registers are missing
// elsewhere among the 64 of their kernel (160^3 1515 us a step inlined, 1455 out
// of line with four pieces, 1416 with two; 32-cell patches with every detail,
// 192^3: 2863 with four, 2943 with two).
template <int P, int L, int ST> __device__ __noinline__ void store_record3(const float* Sc, const int* head, uint4 first, uint4* dst) {
  typedef Cfg3<P, L, ST> C;
  constexpr int F = C::F, NT = C::NT;
  static_assert(C::HDR == 16 + 16 * F && C::PITCH % 4 == 0 && C::FACES % 4 == 0, "16-byte pieces of the record");
  const int n16 = int(first.x / 16u);
  int f = 0;
  auto piece = [&](int i) -> uint4 {  // 16 bytes of the record; i grows from call to call
    if (i == 0) return first;
    if (i <= F) {
      const int* h = head + 4 * (i - 1);
      return make_uint4(unsigned(h[0]), unsigned(h[1]), unsigned(h[2]), unsigned(h[3]));
    }
    while (f + 1 < F && 16 * i >= head[4 * (f + 1)]) ++f;
    return *reinterpret_cast<const uint4*>(Sc + size_t(f) * C::PITCH + C::FACES + (4 * i - head[4 * f] / 4));
  };
  constexpr int NP = P >= 32 ? 4 : 2;  // pieces in flight per thread
#pragma unroll 1
  for (int i0 = threadIdx.x; i0 < n16; i0 += NP * NT) {
    uint4 v[NP];
#pragma unroll
    for (int k = 0; k < NP; ++k) v[k] = k == 0 || i0 + k * NT < n16 ? piece(i0 + k * NT) : v[0];
#pragma unroll
    for (int k = 0; k < NP; ++k)
      if (k == 0 || i0 + k * NT < n16) dst[i0 + k * NT] = v[k];
  }
}

// One patch (pid) of one launch.  MODE_INIT encodes the equilibrium of the
// macroscopic fields, MODE_STEP advances one step, MODE_EXPORT decodes.
template <int WV, int ST, int P, int L, int MODE, int FEAT = 0, int HL = 0>
__device__ void patch3_body(const Patch3Args& a, int pid, float* Sc, unsigned char* smem) {
  typedef Cfg3<P, L, ST> C;
  typedef float T;
  typedef typename C::S S;
  constexpr int F = C::F, E = C::E, E2 = C::E2, E3 = C::E3, EG = C::EG, EG2 = C::EG2;
  constexpr int NT = C::NT, NWARP = C::NWARP, NW = C::NW, NRW = C::NRW, NB = C::NB, WR = C::WR, NC = C::NC;
  static_assert(WV == WV_BL53, "the 3-D path uses the folded BL5/3 wavelet");

  T* tile = reinterpret_cast<T*>(smem);
  // mask words and the survivors before each (edge | interior << 16: at most
  // 6 E^2 and (P-1)^3)
  uint2* wp = reinterpret_cast<uint2*>(smem + C::OFF_MW);
  unsigned int* bmax = reinterpret_cast<unsigned int*>(smem + C::OFF_BMAX);
  float* scl = reinterpret_cast<float*>(smem + C::OFF_SCL);
  float* sinv = reinterpret_cast<float*>(smem + C::OFF_SINV);
  float* tau_i = reinterpret_cast<float*>(smem + C::OFF_TAU);
  float* tau_e = tau_i + NB;
  unsigned int* ws = reinterpret_cast<unsigned int*>(smem + C::OFF_WS);
  int* misc = reinterpret_cast<int*>(smem + C::OFF_MISC);
  int* head = reinterpret_cast<int*>(smem + C::OFF_HEAD);

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int px = pid % a.npx, py = (pid / a.npx) % a.npy, pzc = pid / (a.npx * a.npy);
  auto sidx = [&](int x, int y, int z) -> int { return (z + 1) * EG2 + (y + 1) * EG + (x + 1); };
  const T omega = a.omega;
  // hi + lo coarse storage (kernels of their own, HL = 1): this CTA's FP64
  // work space, the FP64 coarse block of the field being encoded at its end
  constexpr bool hilo = HL != 0 && MODE != MODE_EXPORT;
  double* hb = hilo ? a.hbuf + size_t(blockIdx.x) * a.hbuf_doubles : nullptr;
  double* c64 = hilo ? hb + (C::NC1 * E2 + C::NC1 * C::NC1 * E) : nullptr;

  // The warp tasks of a z pass: task y holds the columns (x = lane, y), the
  // face tasks (P, y = lane).  fn(row?, x, y, in, line): `line` has what does
  // not change along z: the bits of a mask word below this lane's that count
  // with it (an interior lane of a row does not count the edge node x = 0),
  // where its rank sits in the packed prefix, its band and whether it is coarse.
  struct ZLine {
    unsigned int lt, mask;
    int shift, cxy;
    bool edge, coarse;
  };
  auto z_tasks = [&](auto fn) {
#pragma unroll 1
    for (int g = warp; g < C::RG + C::FG; g += NWARP) {
      const bool row = g < C::RG;
      const int yl = 32 * (g - C::RG) + lane;
      const int x = row ? lane : P, y = row ? g : (yl < E ? yl : 0);
      const bool in = row ? lane < P : yl < E;
      ZLine zl;
      zl.lt = (1u << lane) - 1u;
      zl.edge = x == 0 || x == P || y == 0 || y == P;
      zl.mask = (y == 0 || y == P) ? zl.lt : (lane == 0 ? 0u : zl.lt & ~1u);
      zl.shift = zl.edge ? 0 : 16;
      zl.cxy = (node_class_rt<L>(x) * (L + 1) + node_class_rt<L>(y)) * (L + 1);
      zl.coarse = in && ((x | y) & ((1 << L) - 1)) == 0;
      if (row) fn(std::true_type(), x, y, in, zl);
      else fn(std::false_type(), x, y, in, zl);
    }
  };

  // every node of the tile (index i, coordinates): a warp per row of 33 nodes
  // (the 33rd by the row's first lane), a thread per node in small patches
  auto copy_rows = [&](auto fn) {
    if constexpr (P == 32) {
#pragma unroll 4
      for (int r = warp; r < E2; r += NWARP) {
        const int z = r / E, y = r - z * E;
        fn(r * E + lane, lane, y, z);
        if (lane == 0) fn(r * E + P, P, y, z);
      }
    } else {
      for (int i = tid; i < E3; i += NT) fn(i, i % E, (i / E) % E, i / E2);
    }
  };

  // lifting of every line of the tile along x (0) or y (1)
  auto lines = [&](int axis, bool inverse) {
    for (int l = tid; l < E2; l += NT) {
      const int u = l % E, v = l / E;
      T* p = tile + v * E2 + (axis == 0 ? u * E : u);
      const int stride = axis == 0 ? 1 : E;
      if (inverse) line_transform<WV, P, L, true, T>(p, stride);
      else line_transform<WV, P, L, false, T>(p, stride);
    }
    __syncthreads();
  };

  // ------------------------------------------------------------ decode
  // Record of the current state -> every field, inverse transformed, in the
  // scratch (STEP) or to the dense output (EXPORT).
  if constexpr (MODE == MODE_STEP || MODE == MODE_EXPORT) {
    const unsigned long long ent = a.tab_in[pid];
    const unsigned char* R = a.arena_in + (ent >> 24);
    if (tid < F) {  // the section headers of every field
      const uint4 fe = *reinterpret_cast<const uint4*>(R + 16 + 16 * tid);  // offset, nwords, nedge, nint
      int* h = head + 5 * tid;
      h[0] = int(fe.x);
      h[1] = int(fe.y);
      h[2] = int(fe.z);
      if constexpr (C::QUANT) {
        h[3] = int(ldg_u32(R + fe.x + NC * 4));
        h[4] = int(ldg_u32(R + fe.x + NC * 4 + 4));
      }
    }
    __syncthreads();
    for (int f = 0; f < F; ++f) {
      if constexpr (MODE == MODE_EXPORT) {
        if (a.field_sel >= 0 && f != a.field_sel) continue;
      }
      const unsigned char* sec = R + head[5 * f];
      int p = NC * 4;
      unsigned long long bm = 0ull;
      if constexpr (C::QUANT) {
        bm = (unsigned long long)(unsigned int)head[5 * f + 3] | ((unsigned long long)(unsigned int)head[5 * f + 4] << 32);
        if (tid < NB) scl[tid] = ((bm >> tid) & 1ull) ? __ldg(reinterpret_cast<const float*>(sec + p + 8) + __popcll(bm & ((1ull << tid) - 1ull))) : 0.0f;
        p += 8 + 4 * __popcll(bm);
      }
      const unsigned char* pres = sec + p;
      const unsigned char* words = pres + 4 * C::NPW;
      // every mask word (absent ones zero) and the survivors before it: a
      // warp takes chunks of 32 words, then adds the chunks before its own
      const unsigned int p0 = lane < C::NPW ? ldg_u32(pres + 4 * lane) : 0u;
      const unsigned int p1 = 32 + lane < C::NPW ? ldg_u32(pres + 4 * (32 + lane)) : 0u;
      const unsigned int n0 = __popc(p0), n1 = __popc(p1);
      const unsigned int i0 = warp_incl_scan(n0), i1 = warp_incl_scan(n1);
      const unsigned int t0 = __shfl_sync(0xffffffffu, i0, 31);
      for (int k = warp; k < C::NCK; k += NWARP) {
        const unsigned int pk = __shfl_sync(0xffffffffu, k < 32 ? p0 : p1, k & 31);
        const unsigned int jk = __shfl_sync(0xffffffffu, k < 32 ? i0 - n0 : t0 + i1 - n1, k & 31);
        const int w = 32 * k + lane;
        const bool has = (pk >> lane) & 1u;
        const unsigned int word = has ? ldg_u32(words + 4 * int(jk + __popc(pk & ((1u << lane) - 1u)))) : 0u;
        const unsigned int em = w < NW ? word3_edges<P, E, WR>(w) : 0u;
        const unsigned int ne = __popc(word & em), v = ne | ((__popc(word) - ne) << 16);
        const unsigned int sc = warp_incl_scan(v);
        if (w < NW) wp[w] = make_uint2(word, sc - v);
        if (lane == 31) ws[k] = sc;
      }
      __syncthreads();
      for (int k = warp; k < C::NCK; k += NWARP) {
        unsigned int tot;
        const unsigned int base = chunk_base(ws, C::NCK, k, tot);
        if (32 * k + lane < NW) wp[32 * k + lane].y += base;
      }
      __syncthreads();
      // decode and inverse z lifting: warp task y holds the columns (x = lane,
      // y), all their values loaded at once; the face tasks hold (P, y = lane)
      const unsigned char* pe = sec + ((p + 4 * C::NPW + 4 * head[5 * f + 1] + 7) & ~7);
      const unsigned char* pi = pe + 4 * head[5 * f + 2];
      const float* coarse = reinterpret_cast<const float*>(sec);
      typedef typename RawType<T, ST>::type Raw;
      z_tasks([&](auto isrow, int x, int y, bool in, const ZLine& zl) {
        constexpr bool ROW = decltype(isrow)::value;
        Raw raw[E];
        unsigned int any = 0u;
#pragma unroll
        for (int z = 0; z < E; ++z) {
          const bool zed = z == 0 || z == P;
          const uint2 q = wp[ROW ? z * E + y : NRW + ((z * E + y) >> 5)];
          const int b = ROW ? lane : (z * E + y) & 31;
          const unsigned int m = ROW ? (zed ? zl.lt : zl.mask) : (1u << b) - 1u;
          const int idx = int(zed ? q.y & 0xffffu : (q.y >> zl.shift) & 0xffffu) + __popc(q.x & m);
          any |= q.x;
          raw[z] = survivor_raw<T, ST>(in && ((q.x >> b) & 1u), zed || zl.edge, idx, pe, pi, false);
        }
        T v[E];
#pragma unroll
        for (int z = 0; z < E; ++z) {
          float sc = 0.0f;
          if constexpr (C::QUANT) sc = scl[zl.cxy + node_class<L>(z)];
          v[z] = survivor_value<T, ST>(raw[z], zl.edge || z == 0 || z == P, false, sc);
          if ((z & ((1 << L) - 1)) == 0 && zl.coarse)
            v[z] = __ldg(coarse + ((z >> L) * C::NC1 + (y >> L)) * C::NC1 + (x >> L));
        }
        if (__any_sync(0xffffffffu, any != 0u || zl.coarse)) inv_levels<WV, P, L, T>(v);
        if (in) {
#pragma unroll
          for (int z = 0; z < E; ++z) tile[z * E2 + y * E + x] = v[z];
        }
      });
      __syncthreads();
      lines(1, true);
      lines(0, true);
      if constexpr (MODE == MODE_STEP) {
        float* Sf = Sc + size_t(f) * C::PITCH;
        copy_rows([&](int i, int x, int y, int z) { Sf[sidx(x, y, z)] = tile[i]; });
      } else {
        const size_t gn = size_t(a.G0) * a.G1 * a.G2;
        const int fo = a.field_sel >= 0 ? 0 : f;
        for (int i = tid; i < E3; i += NT) {
          const int x = i % E, y = (i / E) % E, z = i / E2;
          if (x == P || y == P || z == P) continue;  // owned by the next patch
          const size_t g = size_t(fo) * gn + (size_t(pzc * P + z) * a.G1 + (py * P + y)) * a.G0 + (px * P + x);
          if (a.dense_dtype == 0) reinterpret_cast<double*>(a.dense)[g] = double(tile[i]);
          else reinterpret_cast<float*>(a.dense)[g] = tile[i];
        }
      }
      __syncthreads();
    }
    if constexpr (MODE == MODE_EXPORT) return;
  }

  if constexpr (MODE == MODE_INIT) {
    // equilibrium of the macroscopic fields at every node
    for (int i = tid; i < E3; i += NT) {
      const int x = i % E, y = (i / E) % E, z = i / E2;
      const long long gx = (px * P + x) % a.G0, gy = (py * P + y) % a.G1, gz = (pzc * P + z) % a.G2;
      const size_t g = (size_t(gz) * a.G1 + gy) * a.G0 + gx;
      T fe[19];
      if (a.state) {  // a given state (import): the values themselves
        const size_t vol = size_t(a.G0) * size_t(a.G1) * size_t(a.G2);
#pragma unroll
        for (int q = 0; q < 19; ++q)
          fe[q] = a.state_dtype == 0 ? T(reinterpret_cast<const double*>(a.state)[q * vol + g])
                                     : T(reinterpret_cast<const float*>(a.state)[q * vol + g]);
      } else {
        d3q19_equilibrium<T>(T(a.macro[0][g]), T(a.macro[1][g]), T(a.macro[2][g]), T(a.macro[3][g]), fe);
      }
#pragma unroll
      for (int q = 0; q < 19; ++q) Sc[size_t(q) * C::PITCH + sidx(x, y, z)] = fe[q];
    }
    __syncthreads();
  }

  if constexpr (MODE == MODE_STEP) {
    // ghost layer: the neighbours' exported inward populations
    const int pxm = (px - 1 + a.npx) % a.npx, pxp = (px + 1) % a.npx;
    const int pym = (py - 1 + a.npy) % a.npy, pyp = (py + 1) % a.npy;
    const int pzm = (pzc - 1 + a.npz) % a.npz, pzp = (pzc + 1) % a.npz;
    auto nb = [&](int qx, int qy, int qz) -> const float* {
      return a.ring_in + size_t((qz * a.npy + qy) * a.npx + qx) * C::RING;
    };
    for (int t = tid; t < 30 * E2; t += NT) {
      const int g = t / (5 * E2), r = t - g * 5 * E2, k = r / E2, pos = r - k * E2, u = pos % E, v = pos / E;
      // my ghost face g (0: x = -1, 1: x = P+1, 2: y = -1, ...) is the
      // opposite face of the neighbour on that side
      const int phi = g ^ 1;
      const float* src;
      int x, y, z;
      if (g == 0) { src = nb(pxm, py, pzc); x = -1; y = u; z = v; }
      else if (g == 1) { src = nb(pxp, py, pzc); x = E; y = u; z = v; }
      else if (g == 2) { src = nb(px, pym, pzc); x = u; y = -1; z = v; }
      else if (g == 3) { src = nb(px, pyp, pzc); x = u; y = E; z = v; }
      else if (g == 4) { src = nb(px, py, pzm); x = u; y = v; z = -1; }
      else { src = nb(px, py, pzp); x = u; y = v; z = E; }
      const int pop = d3_face_pop(phi, k);
      Sc[size_t(pop) * C::PITCH + sidx(x, y, z)] = __ldg(src + phi * 5 * E2 + k * E2 + pos);
    }
    for (int t = tid; t < 12 * E; t += NT) {
      const int e = t / E, s = t - e * E, i = 7 + e;
      const int cx = d3_cx(i), cy = d3_cy(i), cz = d3_cz(i);
      const int qx = (px - cx + a.npx) % a.npx, qy = (py - cy + a.npy) % a.npy, qz = (pzc - cz + a.npz) % a.npz;
      const int x = cx > 0 ? -1 : (cx < 0 ? E : s);
      const int y = cy > 0 ? -1 : (cy < 0 ? E : s);
      const int z = cz > 0 ? -1 : (cz < 0 ? E : s);
      Sc[size_t(i) * C::PITCH + sidx(x, y, z)] = __ldg(nb(qx, qy, qz) + 30 * E2 + e * E + s);
    }
    // collision of every node of the patch
    for (int i = tid; i < E3; i += NT) {
      const int x = i % E, y = (i / E) % E, z = i / E2;
      const int s = sidx(x, y, z);
      T fv[19];
#pragma unroll
      for (int q = 0; q < 19; ++q) fv[q] = Sc[size_t(q) * C::PITCH + s];
      d3q19_collide<T>(fv, omega);
#pragma unroll
      for (int q = 0; q < 19; ++q) Sc[size_t(q) * C::PITCH + s] = fv[q];
    }
    __syncthreads();
  }

  // ------------------------------------------------------------ encode
  const double ep = a.eps_patch ? a.eps_patch[pid] : a.eps;
  if (tid < NB) {
    tau_i[tid] = T(ep * a.band_factor[tid]);
    tau_e[tid] = T(a.eps_edge * a.band_factor[tid]);
  }
  if (tid == 0) misc[0] = C::HDR;  // running offset of the next field section
  bool bad = false;
  float* lacc = reinterpret_cast<float*>(smem + C::OFF_LACC);
  double* band_e = reinterpret_cast<double*>(smem + C::OFF_BAND);
  float* band_m = reinterpret_cast<float*>(band_e + NB);
  if constexpr (FEAT) {
    if (tid < NB) {
      band_e[tid] = 0.0;
      band_m[tid] = 0.0f;
    }
  }
  for (int f = 0; f < F; ++f) {
    const float* Sf = Sc + size_t(f) * C::PITCH;
    {
      const int cx = MODE == MODE_STEP ? d3_cx(f) : 0, cy = MODE == MODE_STEP ? d3_cy(f) : 0,
                cz = MODE == MODE_STEP ? d3_cz(f) : 0;
      // pull streaming, copied asynchronously: the whole cube is in flight
      // (by loads and stores of four rows a warp it took 33K cycles a field, now 16K)
      copy_rows([&](int i, int x, int y, int z) {
        const unsigned int d = (unsigned int)__cvta_generic_to_shared(tile + i);
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(Sf + sidx(x - cx, y - cy, z - cz)) : "memory");
      });
      asm volatile("cp.async.wait_all;" ::: "memory");
    }
    for (int w = NRW + tid; w < NW; w += NT) wp[w].x = 0u;  // face words take their bits one by one
    if (tid < NB) bmax[tid] = 0u;
    __syncthreads();
    if constexpr (hilo) coarse3_fp64<P, L, NT>(tile, hb, c64);
    lines(0, false);
    lines(1, false);
    // forward z lifting fused with the threshold (Sec. 2.2)
    for (int g = warp; g < C::RG + C::FG; g += NWARP) {
      if (g < C::RG) {
        const int y = g / WR, h = g - y * WR, x = 32 * h + lane;
        const bool valid = x < P;
        const int cx = node_class<L>(x), cy = node_class<L>(y);
        const bool fedge = x == 0 || y == 0 || y == P;
        T* col = tile + y * E + (valid ? x : 0);
        T thr[L + 1];
#pragma unroll
        for (int c = 0; c <= L; ++c) {
          const int b = (cx * (L + 1) + cy) * (L + 1) + c;
          thr[c] = fedge ? tau_e[b] : tau_i[b];
        }
        unsigned int myw[(E + 31) / 32];
#pragma unroll
        for (int k = 0; k < (E + 31) / 32; ++k) myw[k] = 0u;
        unsigned int mx[L + 1];  // bits + 1 of the largest kept interior detail per z class
#pragma unroll
        for (int c = 0; c <= L; ++c) mx[c] = 0u;
        float acc2[L + 1], accm[L + 1];  // FEAT: this z-line's energy and max per z class
#pragma unroll
        for (int c = 0; c <= L; ++c) { acc2[c] = 0.0f; accm[c] = 0.0f; }
        T v[E];
#pragma unroll
        for (int z = 0; z < E; ++z) v[z] = valid ? col[z * E2] : T(0);
        auto node = [&](int z) {
          const int cz = node_class<L>(z);
          if constexpr (FEAT) {
            acc2[cz] = acc2[cz] + v[z] * v[z];
            accm[cz] = fmaxf(accm[cz], fabsf(v[z]));
          }
          bool keep = false;
          if (valid && (cx | cy | cz)) {
            const bool zedge = z == 0 || z == P;
            const int b = (cx * (L + 1) + cy) * (L + 1) + cz;
            keep = fabsf(v[z]) >= (zedge ? tau_e[b] : thr[cz]);
            if constexpr (C::QUANT) {
              if (keep && !zedge) mx[cz] = max(mx[cz], __float_as_uint(fabsf(v[z])) + 1u);
            }
          }
          const unsigned int bal = __ballot_sync(0xffffffffu, keep);
          if (lane == (z & 31)) myw[z >> 5] = bal;
          // dropped details are not read again
          if (valid && (keep || (cx | cy | cz) == 0)) col[z * E2] = v[z];
        };
        fwd_levels_cb<WV, P, 1, L, T>(v, node);
#pragma unroll
        for (int k = 0; k < (E + 31) / 32; ++k) {
          const int z = 32 * k + lane;
          if (z < E) wp[(z * E + y) * WR + h].x = myw[k];
        }
        if constexpr (C::QUANT) {
          if (!fedge)
#pragma unroll
            for (int c = 0; c <= L; ++c)
              if (mx[c]) atomicMax(bmax + (cx * (L + 1) + cy) * (L + 1) + c, mx[c]);
        }
        if constexpr (FEAT) {
          if (valid)
#pragma unroll
            for (int c = 0; c <= L; ++c) {
              lacc[((y * E + x) * (L + 1) + c) * 2] = acc2[c];
              lacc[((y * E + x) * (L + 1) + c) * 2 + 1] = accm[c];
            }
        }
      } else {
        const int y = 32 * (g - C::RG) + lane;
        const bool valid = y < E;
        const int cy = node_class<L>(valid ? y : 0);
        T* col = tile + (valid ? y : 0) * E + P;
        float acc2[L + 1], accm[L + 1];
#pragma unroll
        for (int c = 0; c <= L; ++c) { acc2[c] = 0.0f; accm[c] = 0.0f; }
        T v[E];
#pragma unroll
        for (int z = 0; z < E; ++z) v[z] = valid ? col[z * E2] : T(0);
        auto node = [&](int z) {
          const int cz = node_class<L>(z);
          if (!valid) return;
          if constexpr (FEAT) {
            acc2[cz] = acc2[cz] + v[z] * v[z];
            accm[cz] = fmaxf(accm[cz], fabsf(v[z]));
          }
          bool keep = true;
          if (cy | cz) {  // x = P is a coarse x-node; every node here is on a face
            const int b = cy * (L + 1) + cz;
            keep = fabsf(v[z]) >= tau_e[b];
            if (keep) {
              const int r = z * E + y;
              atomicOr(&wp[NRW + (r >> 5)].x, 1u << (r & 31));
            }
          }
          if (keep) col[z * E2] = v[z];
        };
        fwd_levels_cb<WV, P, 1, L, T>(v, node);
        if constexpr (FEAT) {
          if (valid)
#pragma unroll
            for (int c = 0; c <= L; ++c) {
              lacc[((y * E + P) * (L + 1) + c) * 2] = acc2[c];
              lacc[((y * E + P) * (L + 1) + c) * 2 + 1] = accm[c];
            }
        }
      }
    }
    __syncthreads();
    if constexpr (FEAT) {  // band sums of this field: band b walks its z-lines in order
      if (tid > 0 && tid < NB) {
        const int b = tid, cx = b / ((L + 1) * (L + 1)), cy = (b / (L + 1)) % (L + 1), cz = b % (L + 1);
        float e = 0.0f, m = 0.0f;
        for (int y = 0; y < E; ++y) {
          if (node_class<L>(y) != cy) continue;
          for (int x = 0; x < E; ++x) {
            if (node_class<L>(x) != cx) continue;
            e = e + lacc[((y * E + x) * (L + 1) + cz) * 2];
            m = fmaxf(m, lacc[((y * E + x) * (L + 1) + cz) * 2 + 1]);
          }
        }
        band_e[b] += double(e);
        band_m[b] = fmaxf(band_m[b], m);
      }
    }

    // band scales (Sec. 2.3 values, quantised): BF16 with a power-of-two
    // scale >= max|d|, int8 with max|d|/127, per band over interior survivors
    unsigned long long bm = 0ull;
    if constexpr (C::QUANT) {
      if (tid < NB) {
        float s = 0.0f, si = 0.0f;
        if (tid > 0 && bmax[tid] != 0u) {
          const float m = __uint_as_float(bmax[tid] - 1u);
          if constexpr (ST == ST_BF16) {
            if (m > 0.0f) {
              const int e = pow2_ceil_exp(m);
              s = exp2_int(e);
              si = exp2_int(-e);
            }
          } else {
            s = m / 127.0f;
          }
        }
        scl[tid] = s;
        sinv[tid] = si;
      }
      const unsigned int b0 = __ballot_sync(0xffffffffu, lane > 0 && lane < NB && bmax[lane < NB ? lane : 0] != 0u);
      const unsigned int b1 = __ballot_sync(0xffffffffu, 32 + lane < NB && bmax[32 + lane < NB ? 32 + lane : 0] != 0u);
      bm = (unsigned long long)b0 | ((unsigned long long)b1 << 32);
    }
    // word counts and their scans, a warp per chunk of 32 words; the ballot
    // of a chunk is its word of the presence bitmap
    unsigned int* wsn = ws + 64;
    for (int k = warp; k < C::NCK; k += NWARP) {
      const int w = 32 * k + lane;
      const unsigned int word = w < NW ? wp[w].x : 0u, em = w < NW ? word3_edges<P, E, WR>(w) : 0u;
      const unsigned int ne = __popc(word & em), v = ne | ((__popc(word) - ne) << 16);
      const unsigned int sc = warp_incl_scan(v), pr = __ballot_sync(0xffffffffu, word != 0u);
      if (w < NW) wp[w].y = sc - v;
      if (lane == 31) {
        ws[k] = sc;
        wsn[k] = __popc(pr);
      }
    }
    __syncthreads();
    unsigned int tot, nwords;
    (void)chunk_base(ws, C::NCK, 0, tot);
    (void)chunk_base(wsn, C::NCK, 0, nwords);
    const unsigned int nedge = tot & 0xffffu, nint = tot >> 16;
    const int p_q = NC * 4;
    const int p_pres = p_q + (C::QUANT ? 8 + 4 * __popcll(bm) : 0);
    const int p_words = p_pres + 4 * C::NPW;
    const int p_wend = p_words + 4 * int(nwords);
    const int p_edge = (p_wend + 7) & ~7;
    const int p_int = p_edge + 4 * int(nedge);
    const int p_iend = p_int + C::SB * int(nint);
    const int size = (p_iend + 15) & ~15;
    unsigned char* sec = reinterpret_cast<unsigned char*>(Sc + size_t(f) * C::PITCH + C::FACES);  // the gather of this field is done
    for (int k = warp; k < C::NCK; k += NWARP) {  // prefix counts, presence bitmap, words
      unsigned int t;
      const unsigned int base = chunk_base(ws, C::NCK, k, t), rank = chunk_base(wsn, C::NCK, k, t);
      const int w = 32 * k + lane;
      const unsigned int word = w < NW ? wp[w].x : 0u, pr = __ballot_sync(0xffffffffu, word != 0u);
      if (w < NW) wp[w].y += base;
      if (word) reinterpret_cast<unsigned int*>(sec + p_words)[rank + __popc(pr & ((1u << lane) - 1u))] = word;
      if (lane == 0) reinterpret_cast<unsigned int*>(sec + p_pres)[k] = pr;
    }
    // coarse block, FP64 coarse sums (2^(3L) x the trapezoid sum: details
    // carry no mass), band mask and scales, presence bitmap, words
    for (int c = tid; c < NC; c += NT) {
      const int ix = c % C::NC1, iy = (c / C::NC1) % C::NC1, iz = c / (C::NC1 * C::NC1);
      const float cv = tile[((iz << L) * E + (iy << L)) * E + (ix << L)];
      // a non-finite coefficient anywhere makes a coarse one non-finite (the
      // updates carry every detail into even nodes, level by level and axis
      // by axis), so the coarse block is the whole check
      if (!isfinite(cv)) bad = true;
      reinterpret_cast<float*>(sec)[c] = cv;
    }
    if (warp == NWARP - 1) {
      double acc = 0.0;
      for (int c = lane; c < NC; c += 32) {
        const int ix = c % C::NC1, iy = (c / C::NC1) % C::NC1, iz = c / (C::NC1 * C::NC1);
        double w = 1.0;
        if (ix == 0 || ix == C::NC1 - 1) w *= 0.5;
        if (iy == 0 || iy == C::NC1 - 1) w *= 0.5;
        if (iz == 0 || iz == C::NC1 - 1) w *= 0.5;
        acc = acc + w * double(tile[((iz << L) * E + (iy << L)) * E + (ix << L)]);
      }
#pragma unroll
      for (int o = 16; o >= 1; o >>= 1) acc = acc + __shfl_down_sync(0xffffffffu, acc, o);
      if (lane == 0 && MODE != MODE_EXPORT) a.pstats[size_t(pid) * F + f] = acc * double(1ll << (3 * L));
      if constexpr (hilo) {  // lo = fl32(c64 - hi) and its share of the mass
        double acc_lo = 0.0;
        for (int c = lane; c < NC; c += 32) {
          const int ix = c % C::NC1, iy = (c / C::NC1) % C::NC1, iz = c / (C::NC1 * C::NC1);
          double w = 1.0;
          if (ix == 0 || ix == C::NC1 - 1) w *= 0.5;
          if (iy == 0 || iy == C::NC1 - 1) w *= 0.5;
          if (iz == 0 || iz == C::NC1 - 1) w *= 0.5;
          const float lo = float(c64[c] - double(tile[((iz << L) * E + (iy << L)) * E + (ix << L)]));
          a.coarse_lo[(size_t(pid) * F + f) * NC + c] = lo;
          acc_lo = acc_lo + w * double(lo);
        }
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) acc_lo = acc_lo + __shfl_down_sync(0xffffffffu, acc_lo, o);
        if (lane == 0) a.pstats_lo[size_t(pid) * F + f] = acc_lo * double(1ll << (3 * L));
      }
    }
    if constexpr (C::QUANT) {
      if (tid == 0) {
        reinterpret_cast<unsigned int*>(sec + p_q)[0] = unsigned(bm & 0xffffffffull);
        reinterpret_cast<unsigned int*>(sec + p_q)[1] = unsigned(bm >> 32);
      }
      if (tid < NB && ((bm >> tid) & 1ull))
        reinterpret_cast<float*>(sec + p_q + 8)[__popcll(bm & ((1ull << tid) - 1ull))] = scl[tid];
    }
    if (tid == 0) {
      for (int b = p_wend; b < p_edge; ++b) sec[b] = 0;
      for (int b = p_iend; b < size; ++b) sec[b] = 0;
      int* h = head + 4 * f;
      h[0] = misc[0];
      h[1] = int(nwords);
      h[2] = int(nedge);
      h[3] = int(nint);
    }
    __syncthreads();
    // survivors in bit order, and the new state's inverse z lifting in the
    // same pass: warp task y holds the columns (x = lane, y) as a decoder of
    // the record would (quantised survivors, zeros, coarse samples)
    float* oe = reinterpret_cast<float*>(sec + p_edge);
    S* oi = reinterpret_cast<S*>(sec + p_int);
    z_tasks([&](auto isrow, int x, int y, bool in, const ZLine& zl) {
      constexpr bool ROW = decltype(isrow)::value;
      T* col = tile + y * E + x;
      T v[E];
      unsigned int any = 0u;
#pragma unroll
      for (int z = 0; z < E; ++z) {
        const bool zed = z == 0 || z == P;
        const uint2 q = wp[ROW ? z * E + y : NRW + ((z * E + y) >> 5)];
        const int b = ROW ? lane : (z * E + y) & 31;
        const unsigned int m = ROW ? (zed ? zl.lt : zl.mask) : (1u << b) - 1u;
        const int idx = int(zed ? q.y & 0xffffu : (q.y >> zl.shift) & 0xffffu) + __popc(q.x & m);
        const bool has = in && ((q.x >> b) & 1u);
        any |= q.x;
        const T t = col[z * E2];  // dropped details hold what they were before the threshold
        T val = has || (zl.coarse && (z & ((1 << L) - 1)) == 0) ? t : T(0);
        if (has) {
          if (!ROW || zed || zl.edge) {
            oe[idx] = val;
          } else if constexpr (ST == ST_F32) {
            oi[idx] = val;
          } else if constexpr (ST == ST_BF16) {
            const int b2 = zl.cxy + node_class<L>(z);
            const float s = scl[b2];
            unsigned short h = 0;
            if (s != 0.0f) h = __bfloat16_as_ushort(__float2bfloat16_rn(val * sinv[b2]));
            oi[idx] = h;
            val = __uint_as_float(unsigned(h) << 16) * s;
          } else {
            const float s = scl[zl.cxy + node_class<L>(z)];
            int h = 0;
            if (s != 0.0f) h = int(fminf(127.0f, fmaxf(-127.0f, rintf(val / s))));
            oi[idx] = (signed char)h;
            val = float(h) * s;
          }
        }
        v[z] = val;
      }
      if (__any_sync(0xffffffffu, any != 0u || zl.coarse)) inv_levels<WV, P, L, T>(v);
      if (in) {
#pragma unroll
        for (int z = 0; z < E; ++z) col[z * E2] = v[z];
      }
    });
    __syncthreads();
    if (tid == 0) misc[0] += size;
    // the rest of the re-decode: the new state of this field, its six export
    // layers to the scratch (the gather of this field is done, so its cube is
    // free)
    lines(1, true);
    lines(0, true);
    float* Sw = Sc + size_t(f) * C::PITCH;  // face phi, node (u, v) at phi E^2 + v E + u
    for (int t = tid; t < 6 * E2; t += NT) {
      const int phi = t / E2, pos = t - phi * E2, u = pos % E, v = pos / E;
      const int l = (phi & 1) ? P - 1 : 1;
      int x, y, z;
      if (phi < 2) { x = l; y = u; z = v; }
      else if (phi < 4) { x = u; y = l; z = v; }
      else { x = u; y = v; z = l; }
      Sw[t] = tile[(z * E + y) * E + x];
    }
    __syncthreads();
  }
  if (bad) {
    if (atomicOr(&a.ctl->status, STAT_NAN) == 0u) a.ctl->err_step = int(a.step);
  }
  if constexpr (FEAT) {
    // features of the new state: group (l, S) = the bands whose largest
    // class is l on exactly the axes S, in band order
    float* fv = reinterpret_cast<float*>(smem + C::OFF_FV);
    if (tid < C::NG) {
      const int g = tid, l = g / 7 + 1, S = g % 7 + 1;
      double e = 0.0;
      float m = 0.0f;
      for (int b = 1; b < NB; ++b) {
        const int c0 = b / ((L + 1) * (L + 1)), c1 = (b / (L + 1)) % (L + 1), c2 = b % (L + 1);
        const int bl = max(c0, max(c1, c2));
        const int bs = (c0 == bl ? 1 : 0) | (c1 == bl ? 2 : 0) | (c2 == bl ? 4 : 0);
        if (bl != l || bs != S) continue;
        e += band_e[b];
        m = fmaxf(m, band_m[b]);
      }
      fv[2 * g] = log10f(float(e) * a.feat_inv_cnt[g] + 1e-30f);
      fv[2 * g + 1] = log10f(m + 1e-30f);
      a.feat[size_t(pid) * C::NIN + 2 * g] = fv[2 * g];
      a.feat[size_t(pid) * C::NIN + 2 * g + 1] = fv[2 * g + 1];
    }
    __syncthreads();
    if (a.mlp_wt && warp == 0) {  // the network, lane j owns hidden units j and j + 32
      constexpr int H = 64, NIN = C::NIN;
      const float* W1T = reinterpret_cast<const float*>(smem + C::OFF_W);
      const float* b1 = W1T + NIN * H;
      const float* W2T = b1 + H;
      const float* b2 = W2T + H * H;
      const float* W3 = b2 + H;
      const float* b3 = W3 + H;
      float h0 = b1[lane], h1 = b1[lane + 32];
      for (int i = 0; i < NIN; ++i) {
        const float xi = fv[i];
        h0 = __fmaf_rn(W1T[i * H + lane], xi, h0);
        h1 = __fmaf_rn(W1T[i * H + lane + 32], xi, h1);
      }
      const float a0 = gelu_f(h0), a1v = gelu_f(h1);
      float z0 = b2[lane], z1 = b2[lane + 32];
#pragma unroll 8
      for (int i = 0; i < 32; ++i) {
        const float u = __shfl_sync(0xffffffffu, a0, i);
        z0 = __fmaf_rn(W2T[i * H + lane], u, z0);
        z1 = __fmaf_rn(W2T[i * H + lane + 32], u, z1);
      }
#pragma unroll 8
      for (int i = 0; i < 32; ++i) {
        const float u = __shfl_sync(0xffffffffu, a1v, i);
        z0 = __fmaf_rn(W2T[(i + 32) * H + lane], u, z0);
        z1 = __fmaf_rn(W2T[(i + 32) * H + lane + 32], u, z1);
      }
      float yv = W3[lane] * gelu_f(z0) + W3[lane + 32] * gelu_f(z1);
#pragma unroll
      for (int o = 16; o >= 1; o >>= 1) yv = yv + __shfl_down_sync(0xffffffffu, yv, o);
      if (lane == 0) {
        double ev = pow(10.0, double(yv + b3[0]));
        if (!isfinite(ev)) ev = a.eps;
        a.eps_next[pid] = ev < a.eps_lo ? a.eps_lo : (ev > a.eps_hi ? a.eps_hi : ev);
      }
    }
  }
  // ring: post-collision inward populations of the export layers
  for (int t = tid; t < 6 * E2 + 12 * E; t += NT) {
    if (t < 6 * E2) {
      const int phi = t / E2, pos = t - phi * E2;
      T fv[19];
#pragma unroll
      for (int q = 0; q < 19; ++q) fv[q] = Sc[size_t(q) * C::PITCH + t];
      d3q19_collide<T>(fv, omega);
      float* dst = a.ring_out + size_t(pid) * C::RING + phi * 5 * E2 + pos;
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        // the face's populations, selected with constant indices
        T val = fv[0];
#pragma unroll
        for (int q = 1; q < 19; ++q)
          if (q == d3_face_pop(phi, k)) val = fv[q];
        dst[k * E2] = val;
      }
    } else {
      // edge e: two velocity components not zero; its nodes lie on the face
      // of the first of them
      const int e = (t - 6 * E2) / E, s = t - 6 * E2 - e * E, i = 7 + e;
      const int cx = d3_cx(i), cy = d3_cy(i), cz = d3_cz(i);
      const int ly = cy > 0 ? P - 1 : (cy < 0 ? 1 : s), lz = cz > 0 ? P - 1 : (cz < 0 ? 1 : s);
      const int at = cx != 0 ? (cx > 0 ? E2 : 0) + lz * E + ly : (cy > 0 ? 3 * E2 : 2 * E2) + lz * E + s;
      T fv[19];
#pragma unroll
      for (int q = 0; q < 19; ++q) fv[q] = Sc[size_t(q) * C::PITCH + at];
      d3q19_collide<T>(fv, omega);
      T val = fv[7];
#pragma unroll
      for (int q = 8; q < 19; ++q)
        if (q == i) val = fv[q];
      a.ring_out[size_t(pid) * C::RING + 30 * E2 + e * E + s] = val;
    }
  }
  // allocation and the copy of the record into the arena
  if (tid == 0) {
    const unsigned long long total = (unsigned long long)misc[0];
    const unsigned long long base = atomicAdd(&a.ctl->cursor[a.cur_out], total);
    int ok = 1;
    if (base + total > a.cap_out || total >= (1ull << 24)) {
      ok = 0;
      if (atomicOr(&a.ctl->status, STAT_ARENA_FULL) == 0u) a.ctl->err_step = int(a.step);
    } else {
      a.tab_out[pid] = (base << 24) | total;
    }
    misc[1] = ok;
    misc[2] = int(base & 0xffffffffull);
    misc[3] = int(base >> 32);
  }
  __syncthreads();
  if (misc[1]) {
    const unsigned long long base = (unsigned long long)(unsigned)misc[2] | ((unsigned long long)(unsigned)misc[3] << 32);
    store_record3<P, L, ST>(Sc, head, make_uint4(unsigned(misc[0]), unsigned(pid), unsigned(F), a.flags),
                            reinterpret_cast<uint4*>(a.arena_out + base));
  }
  __syncthreads();
}

// Persistent launch: CTA b takes patches b, b + grid, ... with its own
// scratch slot.  The learned step (FEAT) is bound to one CTA per SM for 16
// cells too, 168 registers a thread: bound to three (64, with spills) a step of
// 160^3 takes 2345 instead of 2592 us and of 176 x 80 x 112 946 instead of 1155,
// but 64 patches 644 instead of 348.
template <int WV, int ST, int P, int L, int MODE, int FEAT = 0, int HL = 0>
__global__ void __launch_bounds__(Cfg3<P, L, ST>::NT, FEAT ? 1 : Cfg3<P, L, ST>::MINB) patch3_kernel(const Patch3Args a) {
  extern __shared__ __align__(16) unsigned char smem3[];
  const int np = a.npx * a.npy * a.npz;
  float* Sc = a.scratch + size_t(blockIdx.x) * a.slot_floats;
  if constexpr (MODE == MODE_STEP) {
    __shared__ unsigned int st0;
    if (threadIdx.x == 0) {
      st0 = *((volatile unsigned int*)&a.ctl->status);
      if (blockIdx.x == 0 && !(st0 & (STAT_ARENA_FULL | STAT_NAN | STAT_BAD_RECORD))) {
        a.ctl->live[a.cur_rst] = a.ctl->cursor[a.cur_rst];
        a.ctl->cursor[a.cur_rst] = 0ull;
      }
    }
    __syncthreads();
    if (st0 & (STAT_ARENA_FULL | STAT_NAN | STAT_BAD_RECORD)) return;
  }
  if constexpr (FEAT) {  // the network's weights, once per CTA
    typedef Cfg3<P, L, ST> C;
    if (a.mlp_wt) {
      float* W = reinterpret_cast<float*>(smem3 + C::OFF_W);
      for (int i = threadIdx.x; i < C::MLP_NP; i += C::NT) W[i] = __ldg(a.mlp_wt + i);
    }
    __syncthreads();
  }
  for (int pid = blockIdx.x; pid < np; pid += gridDim.x) patch3_body<WV, ST, P, L, MODE, FEAT, HL>(a, pid, Sc, smem3);
}

}  // namespace wcs

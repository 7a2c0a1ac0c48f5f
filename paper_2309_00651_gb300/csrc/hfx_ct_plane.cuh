// Forward and x/Coulomb passes of the compile-time FP32 geometry for edges that are a multiple of 4.
//
// What bounds them: every point of a plane goes through shared memory once per exchange between
// butterflies, and shared-memory throughput and issue slots (not HBM) set these passes' time.  So the
// axes are split to need as few exchanges as registers allow: z and x are (N/4) x 4 -- one large radix
// in registers, then a radix 4 -- and the small last stages of a plane's two axes are taken together on
// a 2-D tile of one thread:
//   forward pass:  product -> [z radix N/4] -> [y first radix] -> [z radix 4 x y last radix] -> W
//   x pass:        W -> [x radix N/4] -> [x radix 4, Coulomb, inverse x radix 4, inverse z radix 4]
//                    -> [inverse z radix N/4] -> [inverse x radix N/4] -> W
// (transforms along different axes commute).  That is three shared-memory round trips a plane where one
// stage at a time takes four.  y keeps the split of stage_plan(N), which the accumulate passes invert.
// Measured against the one-stage-at-a-time form, us per launch of 256 couples: forward / x pass 45 / 45
// -> 28 / 27 (32^3), 108 / 127 -> 90 / 96 (48^3), 231 / 239 -> 194 / 221 (64^3), 338 / 409 -> 292 / 346
// (72^3), 436 / 531 -> 415 / 472 (80^3), 778 / 1012 -> 676 / 892 (96^3), 2262 / 2872 -> 2075 / 2368
// (128^3), before the energy sums of PlaneSum.  At 72^3 the x pass moves 4.4 TB/s of DRAM; with its loads and
// stores taken out it runs in 252 us, with its shared-memory stages taken out in 254, so what is left is how far
// the two overlap.
//
// Layouts, chosen so that the half-warps of every stage touch 16 different 8-byte banks:
//   forward: z = 4 D + e of row y sits at y S + e E + D (E = 4 or 12 mod 16, S = 3 mod 16): four rows x
//            four e of the z stage, runs of D in the last stage, and runs of (D, e) in the y stage.
//            At 96^3 rows go without gaps (kDense; E = 24 = 8, S = 97 = 1 mod 16, eight rows x two e in the z
//            stage, runs of places in the y stage), so that three planes fit an SM instead of two: 721 -> 676 us
//            (at 72^3 a fifth plane by rows without gaps lost, 288 -> 302 us);
//   x pass:  (x, z) sits at x S + z + 2 ((x / 8) mod 2), S = N + 2 (2 or 10 mod 16): eight rows x two z
//            in the z stage, runs of z in the x stages, and in the tile stage 16-byte accesses of which
//            eight consecutive lanes (two x, four z tiles) cover all banks.
// W is [couple][y][x][z] for these edges: the x pass, which reads and writes it, then moves whole
// contiguous planes (with [x][y][z] its rows of N z were N^2 apart), and the forward pass writes its
// planes no slower as rows.
#pragma once
#include "hfx_ct.cuh"

namespace hfx {
namespace ct {

template <int N> struct PlaneGeo {
  static_assert(N % 4 == 0, "plane passes need an edge that is a multiple of 4");
  static constexpr int R = N / 4;                                   // large radix of z and x
  static constexpr StagePlan Y = stage_plan(N);
  static_assert(Y.ns == 2, "two y stages");
  static constexpr int RY0 = Y.r[0], RY1 = Y.r[1];
  static constexpr int TW = 4 * (R + R % 2);                        // z and x twiddles, then y's
  static constexpr int TWY = RY1 * RY0;
  // dynamic shared memory of the forward pass for a row stride, and how many such planes fit an SM (228 KB,
  // of which each block takes 1 KB more than it asks for)
  static constexpr int fwd_bytes(int stride) { return (N * stride + TW + TWY) * 8; }
  static constexpr int fwd_planes(int stride) { return 228 * 1024 / (fwd_bytes(stride) + 1024); }
  static constexpr int kPadE = (R + 3) / 8 * 8 + 4;                 // >= R, 4 mod 8
  // forward rows without gaps, where the digits then lie 8 mod 16 apart (eight rows x two e cover the banks)
  // and a third plane fits an SM that holds two (96 so far); with more planes than that latency is hidden anyway
  static constexpr bool kDense =
      R % 16 == 8 && fwd_planes(4 * kPadE + 3) <= 2 && fwd_planes(4 * R + 1) > fwd_planes(4 * kPadE + 3);
  static constexpr int E = kDense ? R : kPadE;
  static constexpr int SF = 4 * E + (kDense ? 1 : 3);               // forward row stride
  // row and z digit of task `id` of the z stage
  static __device__ __forceinline__ void z_task(int id, int& y, int& e) {
    if constexpr (kDense) {
      e = (id >> 3) & 3;
      y = (id >> 5) * 8 + (id & 7);
    } else {
      e = (id >> 2) & 3;
      y = (id >> 4) * 4 + (id & 3);
    }
  }
  static constexpr int SX = N + 2;                                  // x-pass row stride
  static_assert(E >= R && (kDense || E % 8 == 4), "bank-spreading stride of the z digits");
  // place of output k of the large radix among its R: as two radices the runtime-geometry kernels know
  // (plane_radices) would leave it, so that the tables and the pencil and batch kernels share the order
  static constexpr PlaneRadices P = plane_radices(R);
  static __host__ __device__ constexpr int place(int k) { return (k % P.a) * P.b + k / P.a; }
  static constexpr int smem_fwd = fwd_bytes(SF);
  static constexpr int smem_x = (N * SX + 2 + TW) * 8;
};

// launch shapes: threads per block, resident blocks per SM the kernel is built for, and (forward) steps of
// the product each thread keeps in flight.  Many small blocks, whose barriers and phases are independent,
// beat few large ones as long as a thread keeps its radix in registers (72^3 forward: 160 threads x 4
// blocks 288 us, 288 x 3 320 us, 96 x 4 301 us; x pass: 128 x 5 348 us, 288 x 3 372 us; 96^3 x pass, two
// planes fit an SM: 384 x 2 892 us, 192 x 3 with a spilling radix 24 956 us).  Loading the next plane into
// a second buffer while one is transformed lost (399-425 us against 375): it halves the planes in work.
template <int N> struct PlaneCfg;
template <> struct PlaneCfg<32>  { static constexpr int fnt = 64,  fmb = 12, un = 4, xnt = 64,  xmb = 12; };
template <> struct PlaneCfg<36>  { static constexpr int fnt = 96,  fmb = 8,  un = 2, xnt = 96,  xmb = 9; };
template <> struct PlaneCfg<40>  { static constexpr int fnt = 96,  fmb = 8,  un = 2, xnt = 96,  xmb = 9; };
template <> struct PlaneCfg<48>  { static constexpr int fnt = 96,  fmb = 8,  un = 2, xnt = 96,  xmb = 9; };
template <> struct PlaneCfg<60>  { static constexpr int fnt = 128, fmb = 5,  un = 4, xnt = 128, xmb = 6; };
template <> struct PlaneCfg<64>  { static constexpr int fnt = 128, fmb = 5,  un = 4, xnt = 128, xmb = 6; };
template <> struct PlaneCfg<72>  { static constexpr int fnt = 160, fmb = 4,  un = 3, xnt = 128, xmb = 5; };
template <> struct PlaneCfg<80>  { static constexpr int fnt = 160, fmb = 4,  un = 4, xnt = 160, xmb = 4; };
template <> struct PlaneCfg<96>  { static constexpr int fnt = 128, fmb = 3,  un = 6, xnt = 384, xmb = 2; };
template <> struct PlaneCfg<100> { static constexpr int fnt = 224, fmb = 2,  un = 4, xnt = 256, xmb = 2; };
template <> struct PlaneCfg<108> { static constexpr int fnt = 224, fmb = 2,  un = 4, xnt = 256, xmb = 2; };
template <> struct PlaneCfg<120> { static constexpr int fnt = 480, fmb = 1,  un = 4, xnt = 480, xmb = 1; };
template <> struct PlaneCfg<128> { static constexpr int fnt = 512, fmb = 1,  un = 4, xnt = 512, xmb = 1; };

// v[k] *= w^{e k} (or its conjugate); the table holds two consecutive k of one e in 16 bytes
template <int R, bool CONJ>
__device__ __forceinline__ void twiddle_zx(cpair (&v)[R], const cpair* tw, int e) {
  const float4* t = reinterpret_cast<const float4*>(tw) + e;
#pragma unroll
  for (int k = 0; k < R; k += 2) {
    const float4 w = t[(k / 2) * 4];
    if (k > 0) v[k] = CONJ ? cmulc(v[k], cpair{w.x, w.y}) : cmul(v[k], cpair{w.x, w.y});
    if (k + 1 < R) v[k + 1] = CONJ ? cmulc(v[k + 1], cpair{w.z, w.w}) : cmul(v[k + 1], cpair{w.z, w.w});
  }
}

__device__ __forceinline__ cpair ld_cg(const cpair* p) {
  const float2 v = __ldcg(reinterpret_cast<const float2*>(p));
  return cpair{v.x, v.y};
}

// four consecutive complex values (32 bytes, 32-byte aligned) to global memory in one store
__device__ __forceinline__ void st_c4(float2* p, cpair a, cpair b, cpair c, cpair d) {
  asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(a.x), "f"(a.y), "f"(b.x),
               "f"(b.y), "f"(c.x), "f"(c.y), "f"(d.x), "f"(d.y)
               : "memory");
}

// ----------------------------------------------------------------------------------
// forward pass: pair product, z and y transforms of x-plane x of couple cl
// ----------------------------------------------------------------------------------
// The product of one plane into buf, four z a step.  The first loads are issued before the barrier that
// ends the previous item's use of buf, so that their latency runs beside it.
template <int N, int NT, int UN>
__device__ __forceinline__ void product_to_smem(const float* __restrict__ orb, long long Ntot, int4 cp, int x,
                                                cpair* __restrict__ buf) {
  using G = PlaneGeo<N>;
  constexpr int NV = N * G::R;
  const bool hasa = cp.x >= 0, hasb = cp.z >= 0;
  // full couples of an off-diagonal block pair hold (i, j) and (i, j + 1): three planes are read.  Those of a
  // ragged block pair hold (i, j) and (i + 1, j) and read four.
  const bool same = cp.x == cp.z;
  const long long off = (long long)x * (N * N);
  const float4* a1 = reinterpret_cast<const float4*>(orb + (long long)(hasa ? cp.x : 0) * Ntot + off);
  const float4* a2 = reinterpret_cast<const float4*>(orb + (long long)(hasa ? cp.y : 0) * Ntot + off);
  const float4* b1 = reinterpret_cast<const float4*>(orb + (long long)(hasb ? cp.z : 0) * Ntot + off);
  const float4* b2 = reinterpret_cast<const float4*>(orb + (long long)(hasb ? cp.w : 0) * Ntot + off);
#pragma unroll 1
  for (int i0 = threadIdx.x; i0 < NV; i0 += UN * NT) {
    float4 p[UN], q[UN], s[UN];
#pragma unroll
    for (int u = 0; u < UN; ++u) {
      const int i = i0 + u * NT;
      const bool in = (NV % (UN * NT) == 0) || i < NV;
      const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
      p[u] = (in && hasa) ? __ldg(a1 + i) : zero;
      q[u] = (in && hasa) ? __ldg(a2 + i) : zero;
      s[u] = (in && hasb) ? __ldg(b2 + i) : zero;
    }
    if (same) {
#pragma unroll
      for (int u = 0; u < UN; ++u) {
        s[u].x *= p[u].x; s[u].y *= p[u].y; s[u].z *= p[u].z; s[u].w *= p[u].w;
      }
    } else if (hasb) {
#pragma unroll
      for (int u = 0; u < UN; ++u) {
        const int i = i0 + u * NT;
        if ((NV % (UN * NT) == 0) || i < NV) {
          const float4 r = __ldg(b1 + i);
          s[u].x *= r.x; s[u].y *= r.y; s[u].z *= r.z; s[u].w *= r.w;
        }
      }
    }
    if (i0 == threadIdx.x) __syncthreads();  // the previous item is done with buf
#pragma unroll
    for (int u = 0; u < UN; ++u) {
      const int i = i0 + u * NT;
      if ((NV % (UN * NT) == 0) || i < NV) {
        const int y = i / G::R, D = i - y * G::R;  // z = 4 D .. 4 D + 3
        cpair* d = buf + y * G::SF + D;
        d[0] = cpair{p[u].x * q[u].x, s[u].x};
        d[G::E] = cpair{p[u].y * q[u].y, s[u].y};
        d[2 * G::E] = cpair{p[u].z * q[u].z, s[u].z};
        d[3 * G::E] = cpair{p[u].w * q[u].w, s[u].w};
      }
    }
  }
}

template <int N, int NT, int UN>
__device__ __forceinline__ void fwd_plane_item(const float* __restrict__ orb, long long Ntot, int4 cp,
                                               float2* __restrict__ W, cpair* buf, const cpair* tw, int cl, int x) {
  using G = PlaneGeo<N>;
  constexpr int R = G::R, E = G::E, S = G::SF, PLANE = N * N, RY0 = G::RY0, RY1 = G::RY1;
  product_to_smem<N, NT, UN>(orb, Ntot, cp, x, buf);
  __syncthreads();
  // z: elements e + 4 k of row y
#pragma unroll 1
  for (int id = threadIdx.x; id < 4 * N; id += NT) {
    int y, e;
    G::z_task(id, y, e);
    cpair* p = buf + y * S + e * E;
    cpair v[R];
#pragma unroll
    for (int k = 0; k < R; ++k) v[k] = p[k];
    Dft<R, -1, cpair>::run(v);
    twiddle_zx<R, false>(v, tw, e);
#pragma unroll
    for (int k = 0; k < R; ++k) p[G::place(k)] = v[k];
  }
  __syncthreads();
  // y: rows j + RY1 k of one column
#pragma unroll 1
  for (int id = threadIdx.x; id < RY1 * N; id += NT) {
    const int j = id / N, c = id - j * N;
    cpair* p = buf + j * S + (G::kDense ? c : (c & 3) * E + (c >> 2));
    cpair v[RY0];
#pragma unroll
    for (int k = 0; k < RY0; ++k) v[k] = p[k * (RY1 * S)];
    Dft<RY0, -1, cpair>::run(v);
    const cpair* t = tw + G::TW + j * RY0;
#pragma unroll
    for (int k = 1; k < RY0; ++k) v[k] = cmul(v[k], t[k]);
#pragma unroll
    for (int k = 0; k < RY0; ++k) p[k * (RY1 * S)] = v[k];
  }
  __syncthreads();
  // last z and y stages of the tile z = 4 D .. 4 D + 3, y = RY1 Dy .. RY1 Dy + RY1 - 1, to W[cl][y][x][z]
  float2* w = W + (long long)cl * N * PLANE + x * N;
#pragma unroll 1
  for (int id = threadIdx.x; id < R * RY0; id += NT) {
    const int Dy = id / R, D = id - Dy * R;
    const cpair* p = buf + Dy * (RY1 * S) + D;
    cpair v[4][RY1];
#pragma unroll
    for (int f = 0; f < RY1; ++f) {
      cpair t[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) t[e] = p[f * S + e * E];
      Dft<4, -1, cpair>::run(t);
#pragma unroll
      for (int e = 0; e < 4; ++e) v[e][f] = t[e];
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) Dft<RY1, -1, cpair>::run(v[e]);
    float2* d = w + Dy * (RY1 * PLANE) + 4 * D;
#pragma unroll
    for (int f = 0; f < RY1; ++f) st_c4(d + f * PLANE, v[0][f], v[1][f], v[2][f], v[3][f]);
  }
}

template <int N, int NT, int MINB, int UN>
__global__ void __launch_bounds__(NT, MINB)
k_fwd_plane(const float* __restrict__ orb, long long Ntot, const int4* __restrict__ couples, int c0, int c1,
            float2* __restrict__ W, const float2* __restrict__ twg, int prefetch) {
  using G = PlaneGeo<N>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cpair* tw = reinterpret_cast<cpair*>(smem_raw);
  cpair* buf = tw + G::TW + G::TWY;
  for (int i = threadIdx.x; i < G::TW + G::TWY; i += NT) tw[i] = cpair{twg[i].x, twg[i].y};
  const int ncl = c1 - c0, items = ncl * N;
  // x-major order: the blocks in flight work on the same x-plane of many couples, whose orbital planes
  // (the batch's orbitals at that x) are then read from DRAM once and from L2 after
  int it = blockIdx.x;
  int x = it / ncl, cl = it - x * ncl;
  int4 cp = it < items ? couples[c0 + cl] : make_int4(-1, -1, -1, -1);
  __syncthreads();
  while (it < items) {
    // the next item's couple is read, and its orbital planes head for L2, while this item runs
    const int nx = it + gridDim.x;
    const int x2 = nx / ncl, cl2 = nx - x2 * ncl;
    int4 cp2 = make_int4(-1, -1, -1, -1);
    if (nx < items) {
      cp2 = couples[c0 + cl2];
      if (prefetch && threadIdx.x < 4) {
        const int o = threadIdx.x == 0 ? cp2.x : threadIdx.x == 1 ? cp2.y : threadIdx.x == 2 ? cp2.z : cp2.w;
        if (o >= 0 && !(threadIdx.x == 2 && cp2.z == cp2.x))
          prefetch_l2(orb + (long long)o * Ntot + (long long)x2 * N * N, N * N * sizeof(float));
      }
    }
    if (!couple_empty(cp)) fwd_plane_item<N, NT, UN>(orb, Ntot, cp, W, buf, tw, cl, x);
    it = nx;
    x = x2;
    cl = cl2;
    cp = cp2;
  }
}

// ----------------------------------------------------------------------------------
// x pass: forward x, Coulomb multiply and energy, inverse x and z of y-plane y of couple cl
// ----------------------------------------------------------------------------------
// red: [2][32] pairs of floats in shared memory used alternately (par) by consecutive items of a block
template <int N, int NT>
__device__ __forceinline__ void x_plane_item(int c0, float2* __restrict__ W, const float* __restrict__ vtab,
                                             double* __restrict__ epart, int energy_only, cpair* buf,
                                             const cpair* tw, float2 (*red)[32], int par, int cl, int y) {
  using G = PlaneGeo<N>;
  constexpr int R = G::R, S = G::SX, PLANE = N * N;
  float2* wc = W + ((long long)cl * N + y) * PLANE;
  // forward x: elements j + 4 k of column z, straight from W; the loads go through L2 only (each is read
  // once), and the first ones are issued before the barrier that ends the previous item's use of buf
  if constexpr (NT > 4 * N) __syncthreads();
#pragma unroll 1
  for (int id = threadIdx.x; id < 4 * N; id += NT) {
    const int j = id / N, z = id - j * N;
    const cpair* src = reinterpret_cast<const cpair*>(wc) + j * N + z;
    cpair* p = buf + j * S + z;
    cpair v[R];
#pragma unroll
    for (int k = 0; k < R; ++k) v[k] = ld_cg(src + k * (4 * N));
    Dft<R, -1, cpair>::run(v);
    twiddle_zx<R, false>(v, tw, j);
    if (NT <= 4 * N && id == threadIdx.x) __syncthreads();
#pragma unroll
    for (int k = 0; k < R; ++k) p[G::place(k) * (4 * S) + 2 * ((G::place(k) >> 1) & 1)] = v[k];
  }
  // the tile x = 4 X .. 4 X + 3, z = 4 Z .. 4 Z + 3: last forward x stage, v(G) and the energy, first
  // inverse x stage, first inverse z stage.  The plane's energy: FP32 within a butterfly, then PlaneSum;
  // planes and couples are summed in FP64
  PlaneSum energy;
  const float* vy = vtab + (long long)y * N;
  __syncthreads();
#pragma unroll 1
  for (int id = threadIdx.x; id < R * R; id += NT) {
    // lanes alternate between two x tiles whose rows are shifted against each other
    const int q = id & 1, m = R % 2 != 0 ? id : id >> 1, g = m / R, Z = m - g * R;
    // (g of a pair of tiles two apart; what R leaves over: neighbours, or for odd R one by one)
    constexpr int R4 = R / 4 * 4;
    const int X = R % 2 != 0 ? id / R : (g >= R4 / 2 ? R4 + 2 * (g - R4 / 2) + q : (g & 1) + 4 * (g >> 1) + 2 * q);
    float4* p = reinterpret_cast<float4*>(buf + (4 * X) * S + 4 * Z + 2 * ((X >> 1) & 1));
    const float* vp = vy + (4 * X) * PLANE + 4 * Z;
    float4 vg4[4];
#pragma unroll
    for (int f = 0; f < 4; ++f) vg4[f] = __ldg(reinterpret_cast<const float4*>(vp + f * PLANE));
    cpair v[4][4];
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      const float4 a = p[f * (S / 2)], b = p[f * (S / 2) + 1];
      v[0][f] = cpair{a.x, a.y};
      v[1][f] = cpair{a.z, a.w};
      v[2][f] = cpair{b.x, b.y};
      v[3][f] = cpair{b.z, b.w};
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      float en = 0.f;
      Dft<4, -1, cpair>::run(v[e]);
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        const float vg = e == 0 ? vg4[f].x : e == 1 ? vg4[f].y : e == 2 ? vg4[f].z : vg4[f].w;
        en += vg * (v[e][f].x * v[e][f].x + v[e][f].y * v[e][f].y);
        v[e][f].x *= vg;
        v[e][f].y *= vg;
      }
      energy.add(en);
    }
    if (!energy_only) {
#pragma unroll
      for (int e = 0; e < 4; ++e) Dft<4, 1, cpair>::run(v[e]);
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        cpair t[4] = {v[0][f], v[1][f], v[2][f], v[3][f]};
        Dft<4, 1, cpair>::run(t);
        p[f * (S / 2)] = make_float4(t[0].x, t[0].y, t[1].x, t[1].y);
        p[f * (S / 2) + 1] = make_float4(t[2].x, t[2].y, t[3].x, t[3].y);
      }
    }
  }
  // block sum without barriers of its own: the warps' sums to red[par] now, and warp 0 adds them after the
  // barrier that the inverse stages need anyway (at the end of the item instead it cost the x pass 2% more where
  // one or two planes fit an SM)
  energy.warp(red[par]);
  __syncthreads();
  if (threadIdx.x < 32) PlaneSum::block<NT / 32>(red[par], epart + (long long)(c0 + cl) * N + y);
  if (energy_only) return;
  // inverse z: elements e + 4 k of row x
#pragma unroll 1
  for (int id = threadIdx.x; id < (N + 7) / 8 * 32; id += NT) {
    const int e = (id >> 3) & 3, xg = id >> 5, x = xg * 8 + (id & 7);
    if (N % 8 != 0 && x >= N) continue;
    cpair* p = buf + x * S + 2 * (xg & 1) + e;
    cpair v[R];
#pragma unroll
    for (int k = 0; k < R; ++k) v[k] = p[4 * G::place(k)];
    twiddle_zx<R, true>(v, tw, e);
    Dft<R, 1, cpair>::run(v);
#pragma unroll
    for (int k = 0; k < R; ++k) p[4 * k] = v[k];
  }
  __syncthreads();
  // inverse x: elements j + 4 k of column z, straight to W
#pragma unroll 1
  for (int id = threadIdx.x; id < 4 * N; id += NT) {
    const int j = id / N, z = id - j * N;
    const cpair* p = buf + j * S + z;
    cpair v[R];
#pragma unroll
    for (int k = 0; k < R; ++k) v[k] = p[G::place(k) * (4 * S) + 2 * ((G::place(k) >> 1) & 1)];
    twiddle_zx<R, true>(v, tw, j);
    Dft<R, 1, cpair>::run(v);
    cpair* dst = reinterpret_cast<cpair*>(wc) + j * N + z;
#pragma unroll
    for (int k = 0; k < R; ++k) dst[k * (4 * N)] = v[k];
  }
}

template <int N, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB)
k_x_plane(const int4* __restrict__ couples, int c0, int c1, float2* __restrict__ W, const float* __restrict__ vtab,
          const float2* __restrict__ twg, double* __restrict__ epart, int energy_only, int prefetch) {
  using G = PlaneGeo<N>;
  static_assert(NT % 32 == 0, "whole warps");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cpair* tw = reinterpret_cast<cpair*>(smem_raw);
  cpair* buf = tw + G::TW;
  __shared__ float2 red[2][32];  // warp partials of the plane energy, double-buffered by item parity
  for (int i = threadIdx.x; i < G::TW; i += NT) tw[i] = cpair{twg[i].x, twg[i].y};
  int par = 0;
  const int items = (c1 - c0) * N;
  int it = blockIdx.x, cl = it / N;
  bool empty = it < items ? couple_empty(couples[c0 + cl]) : true;
  __syncthreads();
  while (it < items) {
    // this block's next y-plane heads for L2 while this one runs (a row at a time)
    const int nx = it + gridDim.x, cl2 = nx / N;
    bool empty2 = true;
    if (nx < items) {
      empty2 = couple_empty(couples[c0 + cl2]);
      if (prefetch && !empty2)
        for (int r = threadIdx.x; r < N; r += NT)
          prefetch_l2(W + (long long)nx * N * N + r * N, N * sizeof(float2));
    }
    if (!empty) {
      x_plane_item<N, NT>(c0, W, vtab, epart, energy_only, buf, tw, red, par, cl, it - cl * N);
      par ^= 1;
    }
    it = nx;
    cl = cl2;
    empty = empty2;
  }
}

}  // namespace ct
}  // namespace hfx

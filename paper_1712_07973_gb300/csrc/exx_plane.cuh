// Plane pipeline of the pair Poisson solves (sm_103a): the x transforms as
// streaming line kernels, and the whole (y, z) part of a pair's solve for one
// kx on chip.
//
//   xfwd   (one CTA per y, block of ZB z and pair)
//          rho = psi_i psi_j on the lines, real-to-complex FFT along x of
//          length 2n (x >= n zero).  Writes X[pair][kx][y][z], kx <= n.
//   plane  (one CTA per plane (pair, kx))
//          y: pruned forward FFT; z: pruned forward FFT, kernel multiply and
//          Parseval energy, inverse keeping z < n; y: inverse keeping y < n.
//   xinv   (one CTA per y, block of ZB z and pair)
//          complex-to-real FFT along x keeping x < n: V[pair][z][y][x].
//
// The padded (y, z) part of a spectrum never reaches memory: per pair X (8 n^3
// bytes in FP32) is written and read twice, where spectra X[kx][z][ky] padded
// along y move twice that four times.  Planes that go through in halves (128^3,
// 160^3) are read once more and their partial outputs written and read once more
// by the plane kernel, most of that in L2: at 160^3 it moves 47 MB in and 41 out per
// pair, its spectrum being 33.
//
// What bounds it, per pair in FP32 (HBM at 6.8 TB/s, the FMA pipe, shared memory at
// 128 bytes a cycle and SM; measured): plane 96^3 2.1, 6.1, 6.8; 9.9 us (slab pipeline:
// 8.2 for z alone, 17.5 with the y passes of its kernels), 160^3 9.7, 34, 32; 59 us.
// xfwd 96^3 1.0 us of HBM, 1.9 measured; 160^3 4.9 and 9.0 (exchange through shared
// memory 60% busy).  xinv 96^3 1.6 and 1.9; 160^3 7.3 and 8.2.
#pragma once

#include <cstring>

#include "exx_kernels.cuh"

namespace exx {

// Split of the plane kernel's lines with G samples: G = H1 * L2, L2 the
// smallest divisor >= sqrt(G) (12 = 3 x 4, 96 = 8 x 12, 160 = 10 x 16).  A
// free line (padded to 2G) has sub-DFTs of length L1 = 2 H1 with half their
// inputs zero, so its even and odd frequencies come from two DFTs of length
// H1; a periodic line (G long) has L1 = H1.
__host__ __device__ constexpr int plane_l2(int G) {
  for (int b = 1; b <= 16; ++b)
    if (G % b == 0 && b * b >= G && smooth7(b) && smooth7(G / b)) return b;
  return 0;
}
template <int G_, bool PER_> struct PLine {
  static constexpr int G = G_;
  static constexpr bool PER = PER_;
  static constexpr int L = PER ? G : 2 * G;  // line length
  static constexpr int L2 = plane_l2(G), H1 = L2 ? G / L2 : 0, L1 = PER ? H1 : 2 * H1;
};

// Twiddles of one line of the plane kernel (w = exp(-2 pi i / L)):
//   TA[s][n2][k1] = w^(n2 (2 k1 + s)) (free; s = 0, 1) or [n2][k1] = w^(n2 k1)
//   TB[k1][m2] = w^(k1 m2), k1 < L1
// L entries each; consecutive entries are what one thread multiplies in turn.
template <int CNT, typename C> __device__ __forceinline__ void load_tw(const C* t, C (&w)[CNT]) {
  if constexpr (sizeof(C) == 8 && CNT % 2 == 0) {
#pragma unroll
    for (int i = 0; i < CNT; i += 2) {
      const float4 q = *reinterpret_cast<const float4*>(t + i);
      w[i] = mkc<C>(q.x, q.y);
      w[i + 1] = mkc<C>(q.z, q.w);
    }
  } else {
#pragma unroll
    for (int i = 0; i < CNT; ++i) w[i] = t[i];
  }
}

// Products by a unit's twiddles, v[k] w[k]; ONE0: w[0] = 1.  FP64, bound by its
// arithmetic, leaves out those of the units whose twiddles are all one (unit):
// 64^3 120.2 -> 118.4 us per pair.
template <bool ONE0, int CNT, typename C>
__device__ __forceinline__ void twiddle(C (&v)[CNT], const C* t, bool unit) {
  if (sizeof(C) == 16 && unit) return;
  C w[CNT];
  load_tw(t, w);
#pragma unroll
  for (int k = ONE0 ? 1 : 0; k < CNT; ++k) v[k] = cmul(v[k], w[k]);
}
template <int CNT, typename C> __device__ __forceinline__ void twiddle_conj(C (&v)[CNT], const C* t, bool unit) {
  if (sizeof(C) == 16 && unit) return;
  C w[CNT];
  load_tw(t, w);
#pragma unroll
  for (int k = 1; k < CNT; ++k) v[k] = cmulc(v[k], w[k]);
}

// lane by lane a * b + c (FP32 on the device: one packed instruction)
template <typename C> __device__ __forceinline__ C cfma2(C a, C b, C c) {
  if constexpr (sizeof(C) == 8) return __ffma2_rn(a, b, c);
  else return mkc<C>(a.x * b.x + c.x, a.y * b.y + c.y);
}

// ------------------------------------------------------------ tensor memory
// Tensor memory as a stash of values private to a thread (32x32b accesses: a
// warp reaches the 32 lanes 32 (warp % 4) .., one 32-bit word per column).
__device__ __forceinline__ void tmem_alloc(unsigned* smem_slot, unsigned cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(smem_slot)),
               "r"(cols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(unsigned addr, unsigned cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(addr), "r"(cols) : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory"); }

template <int W> __device__ __forceinline__ void tmem_st(unsigned a, const unsigned* r) {
  if constexpr (W >= 16) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16};\n" ::"r"(a),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
    tmem_st<W - 16>(a + 16, r + 16);
  } else if constexpr (W >= 8) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};\n" ::"r"(a), "r"(r[0]),
                 "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
                 : "memory");
    tmem_st<W - 8>(a + 8, r + 8);
  } else if constexpr (W >= 4) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};\n" ::"r"(a), "r"(r[0]), "r"(r[1]),
                 "r"(r[2]), "r"(r[3])
                 : "memory");
    tmem_st<W - 4>(a + 4, r + 4);
  } else if constexpr (W >= 2) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1, %2};\n" ::"r"(a), "r"(r[0]), "r"(r[1]) : "memory");
    tmem_st<W - 2>(a + 2, r + 2);
  }
}
template <int W> __device__ __forceinline__ void tmem_ld(unsigned a, unsigned* r) {
  if constexpr (W >= 16) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(a)
        : "memory");
    tmem_ld<W - 16>(a + 16, r + 16);
  } else if constexpr (W >= 8) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(a)
                 : "memory");
    tmem_ld<W - 8>(a + 8, r + 8);
  } else if constexpr (W >= 4) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a)
                 : "memory");
    tmem_ld<W - 4>(a + 4, r + 4);
  } else if constexpr (W >= 2) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];\n" : "=r"(r[0]), "=r"(r[1]) : "r"(a) : "memory");
    tmem_ld<W - 2>(a + 2, r + 2);
  }
}
// H complex values of a thread to / from its stash at column address a
template <int H, typename C> __device__ __forceinline__ void stash_put(unsigned a, const C (&v)[H]) {
  constexpr int W = H * (int)sizeof(C) / 4;
  unsigned r[W];
  memcpy(r, v, sizeof(r));
  tmem_st<W>(a, r);
}
template <int H, typename C> __device__ __forceinline__ void stash_get(unsigned a, C (&v)[H]) {
  constexpr int W = H * (int)sizeof(C) / 4;
  unsigned r[W];
  tmem_ld<W>(a, r);
  tmem_wait_ld();
  memcpy(v, r, sizeof(r));
}

// -------------------------------------------------------------------- plane
// Shared memory is 78% busy at 96^3 and 66% at 160^3, the FMA pipe and instruction
// issue 56 to 59%, HBM 20%.  Hence: every pass in place (the plane is all the shared memory there
// is), odd pitch and lanes across lines (no bank conflicts, warp-uniform
// twiddles read two at a time), barriers of groups rather than of the CTA, and
// the z samples and partial outputs in tensor memory rather than a second half
// of every z spectrum in shared memory.
//
// Launch shape and on-chip layout of the plane kernel for grids of G points,
// (y, z) lines periodic or free.  The plane P[row][z] holds the y spectrum
// (row = ky in natural order) of the G z-samples, row pitch ZP odd, so that
// lanes along z (y passes) and lanes along ky (z passes) both touch distinct
// banks.  RY = 2 (large free grids): the even and the odd ky, independent
// halves of the spectrum whose inverse y transforms add up, go through the
// same half-size plane one after the other.
template <typename R, int G, bool PERY, bool PERZ, int RY, int NT_, int MINB_, int NG_> struct PlaneCfg {
  using C = cplx<R>;
  using Y = PLine<G, PERY>;
  using Z = PLine<G, PERZ>;
  static constexpr int YU = RY == 2 ? Y::H1 : Y::L1;  // units of y pass 2 = row stride of its inputs
  static constexpr int ROWS = YU * Y::L2;
  static constexpr int ZP = G | 1;
  static constexpr bool SAME = PERY == PERZ;  // one twiddle table
  static constexpr int TWN = 2 * Y::L + (SAME ? 0 : 2 * Z::L);
  static constexpr size_t smem = ((size_t)TWN + (size_t)ROWS * ZP) * sizeof(C);
  static constexpr size_t limit = 227 * 1024 - 1024 - NT_ * sizeof(double);
  static constexpr bool fits = Y::L2 > 0 && (RY == 1 || !PERY) && smem + 4096 + 1024 <= 227 * 1024;
  static constexpr bool ok = G % NG_ == 0 && ROWS % NG_ == 0 && NT_ % (32 * NG_) == 0 && Y::L2 > 0 && (RY == 1 || !PERY) && smem <= limit;
  static constexpr int NT = NT_, MINB = MINB_;
  // NG groups of NTG threads: each owns G / NG of the z in the y passes and
  // ROWS / NG rows in the z passes
  static constexpr int NG = NG_, NTG = NT / NG;
  static constexpr int SWZ = G / NG, SWR = ROWS / NG;
  static constexpr int NE = NT < 128 ? NT / 32 : 4;  // energy partials per plane
  static constexpr int WST = PERZ ? 0 : (int)(Z::H1 * sizeof(C) / 4);  // stash words per z unit
  static constexpr int ZUNITS = SWR * Z::L2;  // per group
  static constexpr int ZROUNDS = (ZUNITS + NTG - 1) / NTG;
  static constexpr int tneed = ((NT + 127) / 128) * ZROUNDS * WST;
  static constexpr int tcols = tneed <= 32 ? 32 : tneed <= 64 ? 64 : tneed <= 128 ? 128 : tneed <= 256 ? 256 : 512;
  static constexpr bool tok = PERZ || tneed <= 512;
};

// Launch shape.  The whole spectrum plane in one CTA where it fits (RY = 1),
// else its halves in turn.  With c CTAs per SM (shared memory), the threads
// are what the registers of the longest sub-DFT allow without spills; grids
// of 32 k points run k groups of 32 lines each, so that a group's barrier
// stops a few warps only.  Measured in FP32 (us per pair, best against the
// neighbours): 96^3 768 threads in 3 groups 10.3 (512 in 2: 11.5), 160^3 640 in 5
// groups 60.4 (one group 64.8, 320 threads 69.9), 128^3 512 in 4 groups 28.7
// (640: 33.6, spills), 112^3 448 in 7 groups of 16 lines 19.1 (one group 20.1),
// 80^3 320 x 2 CTAs 6.4 (384: 7.3, spills), 64^3 256 x 3 CTAs 2.9, 48^3 192 x 4
// 1.36.  FP64 is bound by its arithmetic whatever the shape.
struct PlaneShape {
  int ry, nt, minb, ng;
};
template <typename R, int G, bool PERY, bool PERZ> constexpr PlaneShape plane_shape() {
  using P1 = PlaneCfg<R, G, PERY, PERZ, 1, 128, 1, 1>;
  using P2 = PlaneCfg<R, G, PERY, PERZ, 2, 128, 1, 1>;
  const int ry = P1::fits ? 1 : 2;
  const size_t smem = ry == 1 ? P1::smem : P2::smem;
  const int rows = ry == 1 ? P1::ROWS : P2::ROWS, l2 = plane_l2(G), wst = P1::WST;
  for (int c = 8; c >= 1; --c) {
    int ng = 1, nt = c == 1 ? 512 : c == 2 ? 320 : c == 3 ? 256 : c == 4 ? 192 : 128;
    if (sizeof(R) == 8) {
      nt = c == 1 ? 256 : 128;
    } else if (c == 1) {
      ng = G % 32 == 0 ? G / 32 : G % 16 == 0 ? G / 16 : 1;
      if (ng > 1) nt = ng * (l2 > 12 ? 4 * G / ng : 256);
    } else if (c <= 3 && G % 32 == 0) {
      ng = G / 32;
      nt = (c == 2 ? 384 : 288) / (32 * ng) * (32 * ng);
    } else if (c == 4 && G % 7 == 0) {
      continue;  // the length-7 sub-DFTs spill at 80 registers
    }
    if (c > 1 && c * (smem + nt * sizeof(double) + 16 + 1024) > 228 * 1024) continue;
    // the tensor memory of c CTAs (powers of two of 512 columns)
    const int rounds = (rows / ng * l2 + nt / ng - 1) / (nt / ng);
    int cols = 32;
    while (cols < (nt + 127) / 128 * rounds * wst) cols *= 2;
    if (c * cols <= 512 || c == 1) return PlaneShape{ry, nt, c, ng};
  }
  return PlaneShape{ry, 128, 1, 1};
}

template <typename R, int G, bool PERY, bool PERZ> struct PlaneBuilt {
  static constexpr PlaneShape s = plane_shape<R, G, PERY, PERZ>();
  using K = PlaneCfg<R, G, PERY, PERZ, s.ry, s.nt, s.minb, s.ng>;
  static constexpr bool value = K::ok && K::tok;
};

template <typename R, int G, bool PERY, bool PERZ, int RY, int NT_, int MINB_, int NG_, bool EO>
__global__ void __launch_bounds__(NT_, MINB_)
k_plane(const cplx<R>* X_, cplx<R>* Yo_, const R* __restrict__ Gs, const cplx<R>* __restrict__ tw_g,
        double* __restrict__ epart, int npair, int nkx) {
  using C = cplx<R>;
  using K = PlaneCfg<R, G, PERY, PERZ, RY, NT_, MINB_, NG_>;
  using Y = PLine<G, PERY>;
  using Z = PLine<G, PERZ>;
  constexpr int NT = K::NT, ZP = K::ZP, YU = K::YU;
  constexpr int YH = Y::H1, YL1 = Y::L1, YL2 = Y::L2, ZH = Z::H1, ZL1 = Z::L1, ZL2 = Z::L2;
  constexpr int NTG = K::NTG, SWZ = K::SWZ, SWR = K::SWR;
  constexpr int U1 = YL2 * SWZ;     // a group's units of y forward pass 1 and y inverse pass 2
  constexpr int U2 = YU * SWZ;      // of y forward pass 2 and y inverse pass 1
  constexpr int UZ1 = K::ZUNITS;    // of z passes 1 and 3
  constexpr int UZ2 = ZH * SWR;     // of z pass 2
  // The tensor-memory instructions are warp-wide (.sync.aligned), and so are the
  // groups' named barriers: a warp is brought together ahead of them wherever its
  // lanes may have parted (a last round that not all lanes take, FP64's
  // left-out twiddles where a warp holds units of two n2); groups hold whole
  // warps of units.
  constexpr bool PARTS = UZ1 % NTG != 0 || sizeof(C) == 16;
  static_assert(K::NG == 1 || (NTG % 32 == 0 && U1 % 32 == 0 && U2 % 32 == 0 && UZ1 % 32 == 0 && UZ2 % 32 == 0 &&
                               sizeof(C) == 8), "a group's barrier needs whole warps");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* ta_y = reinterpret_cast<C*>(smem_raw);
  C* tb_y = ta_y + Y::L;
  C* ta_z = K::SAME ? ta_y : tb_y + Y::L;
  C* tb_z = ta_z + Z::L;
  C* P = reinterpret_cast<C*>(smem_raw) + K::TWN;
  __shared__ double red[NT];
  __shared__ unsigned tslot;
  const int tid = threadIdx.x, warp = tid >> 5;
  const int gid = K::NG == 1 ? 0 : tid / NTG, gt = tid - gid * NTG;
  const int zg = gid * SWZ, rg = gid * SWR;  // the group's first z and row
  auto gsync = [&]() {
    if constexpr (K::NG == 1) __syncthreads();
    else asm volatile("bar.sync %0, %1;\n" ::"r"(gid + 1), "n"(NTG) : "memory");
  };
  for (int t = tid; t < K::TWN; t += NT) ta_y[t] = tw_g[t];
  unsigned stash = 0;
  if constexpr (!PERZ) {
    __syncwarp();
    if (warp == 0) tmem_alloc(&tslot, K::tcols);
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  }
  __syncthreads();
  if constexpr (!PERZ) {
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    stash = tslot + ((unsigned)(warp & 3) << 21) + (unsigned)(warp >> 2) * (K::ZROUNDS * K::WST);
  }
  dep_wait();
  const C* X = after_wait(X_);
  C* Yo = after_wait(Yo_);
  const int nplane = npair * nkx;
  // plane pl: kx = pl / npair, pair pl % npair (the pairs of one kx together:
  // its kernel-table rows stay in L2)
  auto plane_at = [&](int pl) { return ((long long)(pl % npair) * nkx + pl / npair) * (G * G); };
  for (int pl = blockIdx.x; pl < nplane; pl += gridDim.x) {
    const int kx = pl / npair, p = pl - kx * npair;
    const C* in = X + plane_at(pl);
    C* out = Yo + plane_at(pl);
    const R* __restrict__ Gk = Gs + (long long)kx * Z::L * Y::L;
    double eacc = 0.0;
#pragma unroll 1
    for (int sy = 0; sy < RY; ++sy) {
      // y forward, pass 1: units (n2, z), lanes along z
#pragma unroll 1
      for (int u = gt; u < U1; u += NTG) {
        const int n2 = u / SWZ, z = zg + u - n2 * SWZ;
        C v[YH];
#pragma unroll
        for (int n1 = 0; n1 < YH; ++n1) v[n1] = in[(YL2 * n1 + n2) * G + z];  // samples y = YL2 n1 + n2
        C* o = P + (YU * n2) * ZP + z;
        if constexpr (PERY) {
          dft<YH, 1, -1>(v);
          twiddle<true>(v, ta_y + n2 * YH, n2 == 0);
#pragma unroll
          for (int k = 0; k < YH; ++k) o[k * ZP] = v[k];
        } else if constexpr (RY == 1) {
          C e[YH];
#pragma unroll
          for (int k = 0; k < YH; ++k) e[k] = v[k];
          dft<YH, 1, -1>(e);
          twiddle<true>(e, ta_y + n2 * YH, n2 == 0);
#pragma unroll
          for (int k = 0; k < YH; ++k) o[2 * k * ZP] = e[k];
          sfor<YH>([&](auto J) { v[J] = twmul<-1, YL1, (int)J>(v[J]); });
          dft<YH, 1, -1>(v);
          twiddle<false>(v, ta_y + (YL2 + n2) * YH, n2 == 0);
#pragma unroll
          for (int k = 0; k < YH; ++k) o[(2 * k + 1) * ZP] = v[k];
        } else {
          if (sy) sfor<YH>([&](auto J) { v[J] = twmul<-1, YL1, (int)J>(v[J]); });
          dft<YH, 1, -1>(v);
          twiddle<false>(v, ta_y + (sy * YL2 + n2) * YH, n2 == 0);
#pragma unroll
          for (int k = 0; k < YH; ++k) o[k * ZP] = v[k];
        }
      }
      gsync();
      // y forward, pass 2: units (k1, z), in place: row k1 + YU k2 = ky
#pragma unroll 1
      for (int u = gt; u < U2; u += NTG) {
        const int k1 = u / SWZ, z = zg + u - k1 * SWZ;
        C* o = P + k1 * ZP + z;
        C v[YL2];
#pragma unroll
        for (int n2 = 0; n2 < YL2; ++n2) v[n2] = o[YU * n2 * ZP];
        dft<YL2, 1, -1>(v);
#pragma unroll
        for (int k2 = 0; k2 < YL2; ++k2) o[YU * k2 * ZP] = v[k2];
      }
      __syncthreads();
      // the next plane's samples into L2
      if (RY == 1 || sy == 1) {
        const int pn = pl + (int)gridDim.x;
        if (pn < nplane) {
          const unsigned char* nx = reinterpret_cast<const unsigned char*>(X + plane_at(pn));
          for (int t = tid * 128; t < G * G * (int)sizeof(C); t += NT * 128)
            asm volatile("prefetch.global.L2 [%0];\n" ::"l"(nx + t));
        }
      }
      __syncwarp();
      // z forward, pass 1: units (n2, row), lanes along ky; in place: samples
      // z = ZL2 n1 + n2 become slots ZL2 k1 + n2.  Free lines: the even
      // frequencies first; the samples go to the thread's stash for the odd ones
#pragma unroll 1
      for (int r = 0; r < K::ZROUNDS; ++r) {
        const int u = gt + r * NTG;
        const bool on = UZ1 % NTG == 0 || u < UZ1;
        const int n2 = u / SWR, row = rg + u - n2 * SWR;
        C* o = P + row * ZP + n2;
        C v[ZH];
        if (on) {
#pragma unroll
          for (int n1 = 0; n1 < ZH; ++n1) v[n1] = o[ZL2 * n1];
        }
        if constexpr (!PERZ) {
          if constexpr (PARTS) __syncwarp();
          stash_put(stash + r * K::WST, v);
        }
        if (on) {
          dft<ZH, 1, -1>(v);
          twiddle<true>(v, ta_z + n2 * ZH, n2 == 0);
#pragma unroll
          for (int k = 0; k < ZH; ++k) o[ZL2 * k] = v[k];
        }
      }
      if constexpr (!PERZ) {
        if constexpr (PARTS) __syncwarp();
        tmem_wait_st();
      }
      gsync();
#pragma unroll 1
      for (int sz = 0; sz < (PERZ ? 1 : 2); ++sz) {
        // z forward pass 2, kernel multiply, energy, inverse pass 1: units (k1, row)
#pragma unroll 1
        for (int u = gt; u < UZ2; u += NTG) {
          const int k1 = u / SWR, row = rg + u - k1 * SWR;
          const int kf = PERZ ? k1 : 2 * k1 + sz;
          const R* __restrict__ g = Gk + kf * Y::L + (RY == 2 ? sy * G : 0) + row;
          R gv[ZL2];
#pragma unroll
          for (int k2 = 0; k2 < ZL2; ++k2) gv[k2] = __ldg(g + (ZL1 * k2) * Y::L);
          C* o = P + row * ZP + ZL2 * k1;
          C v[ZL2];
#pragma unroll
          for (int n2 = 0; n2 < ZL2; ++n2) v[n2] = o[n2];
          dft<ZL2, 1, -1>(v);
          C es = mkc<C>(R(0), R(0));
#pragma unroll
          for (int k2 = 0; k2 < ZL2; ++k2) {
            const C t = cscale(v[k2], gv[k2]);
            es = cfma2(t, v[k2], es);
            v[k2] = t;
          }
          eacc += (double)(es.x + es.y);
          if constexpr (!EO) {
            dft<ZL2, 1, 1>(v);
            twiddle_conj(v, tb_z + kf * ZL2, kf == 0);
#pragma unroll
            for (int m2 = 0; m2 < ZL2; ++m2) o[m2] = v[m2];
          }
        }
        if (sy == RY - 1 && (PERZ || sz == 1)) red[tid] = eacc;
        if (!EO || (!PERZ && sz == 0)) gsync();
        if constexpr (PERZ) {
          if constexpr (!EO) {
            // z inverse, pass 2: units (m2, row)
#pragma unroll 1
            for (int u = gt; u < UZ1; u += NTG) {
              const int m2 = u / SWR, row = rg + u - m2 * SWR;
              C* o = P + row * ZP + m2;
              C v[ZH];
#pragma unroll
              for (int k = 0; k < ZH; ++k) v[k] = o[ZL2 * k];
              dft<ZH, 1, 1>(v);
#pragma unroll
              for (int m1 = 0; m1 < ZH; ++m1) o[ZL2 * m1] = v[m1];
            }
            __syncthreads();
          }
        } else if (sz == 0) {
          // inverse pass 2 of the even frequencies (partial outputs to the
          // stash) and forward pass 1 of the odd ones (samples from it)
#pragma unroll 1
          for (int r = 0; r < K::ZROUNDS; ++r) {
            const int u = gt + r * NTG;
            const bool on = UZ1 % NTG == 0 || u < UZ1;
            const int n2 = u / SWR, row = rg + u - n2 * SWR;
            C* o = P + row * ZP + n2;
            C v[ZH], a[ZH];
            if constexpr (PARTS) __syncwarp();
            stash_get(stash + r * K::WST, v);
            if constexpr (!EO) {
              if (on) {
#pragma unroll
                for (int k = 0; k < ZH; ++k) a[k] = o[ZL2 * k];
                dft<ZH, 1, 1>(a);
              }
              if constexpr (PARTS) __syncwarp();
              stash_put(stash + r * K::WST, a);
            }
            if (on) {
              sfor<ZH>([&](auto J) { v[J] = twmul<-1, ZL1, (int)J>(v[J]); });
              dft<ZH, 1, -1>(v);
              twiddle<false>(v, ta_z + (ZL2 + n2) * ZH, n2 == 0);
#pragma unroll
              for (int k = 0; k < ZH; ++k) o[ZL2 * k] = v[k];
            }
          }
          if constexpr (!EO) {
            if constexpr (PARTS) __syncwarp();
            tmem_wait_st();
          }
          gsync();
        } else if constexpr (!EO) {
          // inverse pass 2 of the odd frequencies, added to the even part
#pragma unroll 1
          for (int r = 0; r < K::ZROUNDS; ++r) {
            const int u = gt + r * NTG;
            const bool on = UZ1 % NTG == 0 || u < UZ1;
            const int m2 = u / SWR, row = rg + u - m2 * SWR;
            C* o = P + row * ZP + m2;
            C v[ZH], a[ZH];
            if constexpr (PARTS) __syncwarp();
            stash_get(stash + r * K::WST, a);
            if (on) {
#pragma unroll
              for (int k = 0; k < ZH; ++k) v[k] = o[ZL2 * k];
              dft<ZH, 1, 1>(v);
              sfor<ZH>([&](auto J) { o[ZL2 * J] = twadd<1, ZL1, (int)J>(a[J], v[J]); });
            }
          }
          __syncthreads();
        }
      }
      if constexpr (EO) __syncthreads();
      if (sy == RY - 1 && warp < 4) {
        // Parseval energy of the plane: warp w adds the sums of threads 32 w ..
        // + 128 i (fixed order), one partial per warp; the other warps go on
        double s = 0.0;
#pragma unroll 1
        for (int t = tid; t < NT; t += 128) s += red[t];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((tid & 31) == 0)
          epart[((long long)p * nkx + kx) * K::NE + warp] = ((kx == 0 || kx == nkx - 1) ? 1.0 : 2.0) * s;
      }
      if constexpr (!EO) {
        // RY = 2, odd half: the even half's partial outputs, written by this
        // thread, requested one round ahead
        C na[RY == 2 ? YH : 1];
        auto fetch_a = [&](int u) {
          if constexpr (RY == 2) {
            if (sy && u < U1) {
              const int m2 = u / SWZ, z = zg + u - m2 * SWZ;
#pragma unroll
              for (int k = 0; k < YH; ++k) na[k] = out[(YL2 * k + m2) * G + z];
            }
          }
        };
        // y inverse, pass 1: units (k1, z), in place (rows k1 + YU k2 -> slots k1 + YU m2)
#pragma unroll 1
        for (int u = gt; u < U2; u += NTG) {
          const int k1 = u / SWZ, z = zg + u - k1 * SWZ;
          const int kf = RY == 2 ? 2 * k1 + sy : k1;
          C* o = P + k1 * ZP + z;
          C v[YL2];
#pragma unroll
          for (int k2 = 0; k2 < YL2; ++k2) v[k2] = o[YU * k2 * ZP];
          dft<YL2, 1, 1>(v);
          twiddle_conj(v, tb_y + kf * YL2, kf == 0);
#pragma unroll
          for (int m2 = 0; m2 < YL2; ++m2) o[YU * m2 * ZP] = v[m2];
        }
        fetch_a(gt);
        gsync();
        // y inverse, pass 2: units (m2, z): outputs y = YL2 m1 + m2
#pragma unroll 1
        for (int u = gt; u < U1; u += NTG) {
          const int m2 = u / SWZ, z = zg + u - m2 * SWZ;
          const C* o = P + (YU * m2) * ZP + z;
          C* q = out + m2 * G + z;
          C v[YH];
          if constexpr (PERY) {
#pragma unroll
            for (int k = 0; k < YH; ++k) v[k] = o[k * ZP];
            dft<YH, 1, 1>(v);
#pragma unroll
            for (int m1 = 0; m1 < YH; ++m1) q[YL2 * m1 * G] = v[m1];
          } else if constexpr (RY == 1) {
            C e[YH];
#pragma unroll
            for (int k = 0; k < YH; ++k) {
              e[k] = o[2 * k * ZP];
              v[k] = o[(2 * k + 1) * ZP];
            }
            dft<YH, 1, 1>(e);
            dft<YH, 1, 1>(v);
            sfor<YH>([&](auto J) { q[YL2 * J * G] = twadd<1, YL1, (int)J>(e[J], v[J]); });
          } else {
#pragma unroll
            for (int k = 0; k < YH; ++k) v[k] = o[k * ZP];
            dft<YH, 1, 1>(v);
            if (sy) {
              sfor<YH>([&](auto J) { v[J] = twadd<1, YL1, (int)J>(na[J], v[J]); });
              fetch_a(u + NTG);
            }
#pragma unroll
            for (int k = 0; k < YH; ++k) q[YL2 * k * G] = v[k];
          }
        }
        gsync();
      }
    }
  }
  if constexpr (!PERZ) {
    __syncthreads();
    if (warp == 0) tmem_dealloc(tslot, K::tcols);
  }
}

// ------------------------------------------------------------- x line kernels
// Split of the complex length-N line (N = half the padded x line, or half the
// periodic one): N = X1 * X2, X1 the smallest even divisor >= sqrt(N) (96 = 12 x
// 8, 160 = 16 x 10).
__host__ __device__ constexpr int plane_x1(int N) {
  for (int a = 2; a <= 16; a += 2)
    if (N % a == 0 && a * a >= N && smooth7(a) && smooth7(N / a)) return a;
  return 0;
}
// z-lines per CTA: 32 where that divides the grid (X[kx][y][z] in runs of 256
// bytes), else its largest divisor up to 16, so that no CTA is partial (160^3:
// 9.0 and 8.1 us per pair forward and inverse with 32, 9.9 and 12.0 with 16)
__host__ __device__ constexpr int plane_zb(int G) {
  if (G % 32 == 0) return 32;
  for (int b = 16; b > 1; --b)
    if (G % b == 0) return b;
  return 1;
}
// One CTA per (pair, y, block of ZB lines).  The transform takes two passes
// and one exchange through S.  On the spectrum side a thread holds the two
// sub-DFTs q and X1 - q (q = 0: 0 and X1 / 2) of a line: the frequencies k and
// N - k that the split into the Hermitian half spectrum (and its inverse)
// combines are both its own, so the spectrum goes from registers to memory
// (from memory to registers) with no further pass.
// Forward, the samples come in whole rows through T[zl][x] (pairs of samples,
// odd pitch) and every pass keeps its lanes along zl: read straight from memory,
// eight or ten lanes per row and orbital, they kept the load/store unit 80% busy
// at 160^3 (11.3 -> 9.0 us per pair; 64^3 0.87 -> 0.75).  Inverse, the samples of
// one orbital pair go straight from registers to memory (a stage and its
// barrier cost more: 8.1 -> 8.9 us at 160^3), lanes along x.
template <typename R, int N, bool PER> struct XCfg {
  static constexpr int G = PER ? 2 * N : N;
  static constexpr int ZB = plane_zb(G), NZB = G / ZB;
  static constexpr int X1 = plane_x1(N), X2 = X1 ? N / X1 : 1;
  static constexpr int GC = G / 2, TP = GC | 1;  // sample pairs per line, pitch of T
  static constexpr bool ok = X1 != 0 && X2 <= 16 && G % 2 == 0;
  static constexpr int UA = X2 * ZB;         // units (n2, line) of the sample side
  static constexpr int UB = (X1 / 2) * ZB;   // units (q, line) of the spectrum side
  static constexpr int most = UA > UB ? UA : UB;
  static constexpr int NT = most >= 320 ? 320 : (most + 31) / 32 * 32;
  static constexpr int MINB = (sizeof(R) == 8 ? 512 : 1024) / NT;
  // forward: twiddles w^k (k < 2N) and TX[k1][n2] = w^(2 n2 k1) (N), T, S[row][zl]
  static constexpr size_t smem_f = (3 * (size_t)N + (size_t)ZB * TP + (size_t)N * ZB) * sizeof(cplx<R>);
  // inverse: w^k, S with row r at srow(r) (pitch SP, skewed every X1 rows)
  static constexpr int SP = ZB | 1;
  static constexpr size_t smem_i = (2 * (size_t)N + (size_t)N * SP + (X1 ? N / X1 : 0) + 1) * sizeof(cplx<R>);
};

template <typename R, int N, bool PER>
__global__ void __launch_bounds__(XCfg<R, N, PER>::NT, XCfg<R, N, PER>::MINB)
k_xfwd(const R* psi0, const R* const* __restrict__ psi_tab, const int4* __restrict__ pairs,
       cplx<R>* __restrict__ X, const cplx<R>* __restrict__ tw_g, long long n3) {
  using C = cplx<R>;
  using K = XCfg<R, N, PER>;
  constexpr int G = K::G, ZB = K::ZB, X1 = K::X1, X2 = K::X2, NT = K::NT, GC = K::GC, TP = K::TP;
  constexpr int XIN = PER ? X1 : X1 / 2;  // nonzero inputs of the length-X1 DFTs
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* tw = reinterpret_cast<C*>(smem_raw);
  C* tx = tw + 2 * N;
  C* T = tx + N;
  C* S = T + ZB * TP;
  const int tid = threadIdx.x;
  const int p = blockIdx.x / K::NZB, y = blockIdx.y, z0 = (blockIdx.x - p * K::NZB) * ZB;
  const int4 pr = pairs[p];
  const R* psi = psi_tab ? psi_tab[pr.w] : psi0;
  dep_wait();
  psi = after_wait(psi);
  const R* pi = psi + (long long)pr.x * n3 + (long long)z0 * G * G + y * G;
  const R* pj = psi + (long long)pr.y * n3 + (long long)z0 * G * G + y * G;
  // rho[2m] + i rho[2m+1], whole rows; paired loads where the caller's orbitals
  // are aligned for them
  if ((reinterpret_cast<size_t>(psi) & (sizeof(C) - 1)) == 0) {
    constexpr int NL = (ZB * GC + NT - 1) / NT;
    C a[NL], b[NL];
#pragma unroll
    for (int i = 0; i < NL; ++i) {
      const int t = tid + i * NT, zl = t / GC, c = t - zl * GC;
      if (ZB * GC % NT == 0 || t < ZB * GC) {
        a[i] = *(reinterpret_cast<const C*>(pi + (long long)zl * G * G) + c);
        b[i] = *(reinterpret_cast<const C*>(pj + (long long)zl * G * G) + c);
      }
    }
    for (int t = tid; t < 3 * N; t += NT) tw[t] = tw_g[t];
#pragma unroll
    for (int i = 0; i < NL; ++i) {
      const int t = tid + i * NT, zl = t / GC, c = t - zl * GC;
      if (ZB * GC % NT == 0 || t < ZB * GC) T[zl * TP + c] = mkc<C>(a[i].x * b[i].x, a[i].y * b[i].y);
    }
  } else {
    for (int t = tid; t < 3 * N; t += NT) tw[t] = tw_g[t];
    for (int t = tid; t < ZB * GC; t += NT) {
      const int zl = t / GC, c = t - zl * GC;
      const R* ri = pi + (long long)zl * G * G + 2 * c;
      const R* rj = pj + (long long)zl * G * G + 2 * c;
      T[zl * TP + c] = mkc<C>(ri[0] * rj[0], ri[1] * rj[1]);
    }
  }
  __syncthreads();
  // sample side: units (n2, zl), zl fastest; m = X2 n1 + n2
#pragma unroll 1
  for (int u = tid; u < K::UA; u += NT) {
    const int n2 = u / ZB, zl = u - n2 * ZB;
    C v[X1];
#pragma unroll
    for (int n1 = 0; n1 < XIN; ++n1) v[n1] = T[zl * TP + X2 * n1 + n2];
    if constexpr (PER) dft<X1, 1, -1>(v);
    else dft_halfin<X1, -1>(v);
    C* col = S + n2 * X1 * ZB + zl;
    col[0] = v[0];
#pragma unroll
    for (int k1 = 1; k1 < X1; ++k1) col[k1 * ZB] = cmul(v[k1], tx[k1 * X2 + n2]);
  }
  __syncthreads();
  // spectrum side: units (q, zl), zl fastest; Z[a + X1 k2], Z[b + X1 k2]
  C* Xo = X + ((long long)p * (N + 1) * G + y) * G + z0;
  constexpr int KS = G * G;  // stride of kx
#pragma unroll 1
  for (int u = tid; u < K::UB; u += NT) {
    const int q = u / ZB, zl = u - q * ZB;
    const int a = q, b = q == 0 ? X1 / 2 : X1 - q;
    C va[X2], vb[X2];
#pragma unroll
    for (int n2 = 0; n2 < X2; ++n2) {
      va[n2] = S[(n2 * X1 + a) * ZB + zl];
      vb[n2] = S[(n2 * X1 + b) * ZB + zl];
    }
    dft<X2, 1, -1>(va);
    dft<X2, 1, -1>(vb);
    C* o = Xo + zl;
    if (q == 0) {
      // frequencies X1 k2 pair with X1 (X2 - k2) (0 with N, the Nyquist row),
      // X1/2 + X1 k2 with X1/2 + X1 (X2 - 1 - k2)
      o[0] = mkc<C>(va[0].x + va[0].y, R(0));
      o[(long long)N * KS] = mkc<C>(va[0].x - va[0].y, R(0));
#pragma unroll
      for (int k2 = 1; 2 * k2 <= X2; ++k2) {
        if (2 * k2 == X2) {
          o[(long long)(X1 * k2) * KS] = mkc<C>(va[k2].x, -va[k2].y);
        } else {
          C xk, xm;
          split_step(va[k2], va[X2 - k2], tw[X1 * k2], xk, xm);
          o[(long long)(X1 * k2) * KS] = xk;
          o[(long long)(X1 * (X2 - k2)) * KS] = xm;
        }
      }
#pragma unroll
      for (int k2 = 0; 2 * k2 < X2; ++k2) {
        if (2 * k2 == X2 - 1) {
          o[(long long)(X1 / 2 + X1 * k2) * KS] = mkc<C>(vb[k2].x, -vb[k2].y);
        } else {
          C xk, xm;
          split_step(vb[k2], vb[X2 - 1 - k2], tw[X1 / 2 + X1 * k2], xk, xm);
          o[(long long)(X1 / 2 + X1 * k2) * KS] = xk;
          o[(long long)(X1 / 2 + X1 * (X2 - 1 - k2)) * KS] = xm;
        }
      }
    } else {
#pragma unroll
      for (int k2 = 0; k2 < X2; ++k2) {  // k = a + X1 k2, N - k = b + X1 (X2 - 1 - k2)
        C xk, xm;
        split_step(va[k2], vb[X2 - 1 - k2], tw[a + X1 * k2], xk, xm);
        o[(long long)(a + X1 * k2) * KS] = xk;
        o[(long long)(b + X1 * (X2 - 1 - k2)) * KS] = xm;
      }
    }
  }
}

// Inverse of split_step (times 2): zk = E + i O, zm = conj(E) + i conj(O) with
// E = xk + conj xm, O = (xk - conj xm) conj(w).
template <typename C> EXX_HD void fold_step(C xk, C xm, C w, C& zk, C& zm) {
  const C e = mkc<C>(xk.x + xm.x, xk.y - xm.y);
  const C o = cmulc(mkc<C>(xk.x - xm.x, xk.y + xm.y), w);
  zk = mkc<C>(e.x - o.y, e.y + o.x);
  zm = mkc<C>(e.x + o.y, o.x - e.y);
}

template <typename R, int N, bool PER>
__global__ void __launch_bounds__(XCfg<R, N, PER>::NT, XCfg<R, N, PER>::MINB)
k_xinv(const cplx<R>* X, R* __restrict__ V, const cplx<R>* __restrict__ tw_g) {
  using C = cplx<R>;
  using K = XCfg<R, N, PER>;
  constexpr int G = K::G, ZB = K::ZB, X1 = K::X1, X2 = K::X2, SP = K::SP, NT = K::NT;
  constexpr int XOUT = PER ? X1 : X1 / 2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* tw = reinterpret_cast<C*>(smem_raw);
  C* S = tw + 2 * N;
  const int tid = threadIdx.x;
  const int p = blockIdx.x / K::NZB, y = blockIdx.y, z0 = (blockIdx.x - p * K::NZB) * ZB;
  dep_wait();
  const C* Xi = after_wait(X) + ((long long)p * (N + 1) * G + y) * G + z0;
  constexpr int KS = G * G;
  // spectrum side: units (q, zl), zl fastest; the first unit's values are under
  // way during the set-up
  C va[X2], vb[X2];
  R xn = R(0);
  auto load = [&](int u) {
    const int q = u / ZB, zl = u - q * ZB;
    const int a = q, b = q == 0 ? X1 / 2 : X1 - q;
    const C* in = Xi + zl;
#pragma unroll
    for (int k2 = 0; k2 < X2; ++k2) {
      va[k2] = __ldcs(in + (long long)(a + X1 * k2) * KS);
      vb[k2] = __ldcs(in + (long long)(b + X1 * k2) * KS);
    }
    if (q == 0) xn = __ldcs(&in[(long long)N * KS].x);
  };
  if (tid < K::UB) load(tid);
  for (int t = tid; t < 2 * N; t += NT) tw[t] = tw_g[t];
  __syncthreads();
#pragma unroll 1
  for (int u = tid; u < K::UB; u += NT) {
    const int q = u / ZB, zl = u - q * ZB;
    const int a = q, b = q == 0 ? X1 / 2 : X1 - q;
    if (u != tid) load(u);
    if (q == 0) {
      const R x0 = va[0].x;
      va[0] = mkc<C>(x0 + xn, x0 - xn);
#pragma unroll
      for (int k2 = 1; 2 * k2 <= X2; ++k2) {
        if (2 * k2 == X2) va[k2] = mkc<C>(R(2) * va[k2].x, R(-2) * va[k2].y);
        else fold_step(va[k2], va[X2 - k2], tw[X1 * k2], va[k2], va[X2 - k2]);
      }
#pragma unroll
      for (int k2 = 0; 2 * k2 < X2; ++k2) {
        if (2 * k2 == X2 - 1) vb[k2] = mkc<C>(R(2) * vb[k2].x, R(-2) * vb[k2].y);
        else fold_step(vb[k2], vb[X2 - 1 - k2], tw[X1 / 2 + X1 * k2], vb[k2], vb[X2 - 1 - k2]);
      }
    } else {
#pragma unroll
      for (int k2 = 0; k2 < X2; ++k2)
        fold_step(va[k2], vb[X2 - 1 - k2], tw[a + X1 * k2], va[k2], vb[X2 - 1 - k2]);
    }
    dft<X2, 1, 1>(va);
    dft<X2, 1, 1>(vb);
#pragma unroll
    for (int m2 = 0; m2 < X2; ++m2) {
      S[srow<SP, X1>(m2 * X1) + a * SP + zl] = m2 ? cmulc(va[m2], tw[2 * m2 * a]) : va[0];
      S[srow<SP, X1>(m2 * X1) + b * SP + zl] = m2 ? cmulc(vb[m2], tw[2 * m2 * b]) : vb[0];
    }
  }
  __syncthreads();
  // sample side: units (zl, m2), m2 fastest
  R* Vz = V + (((long long)p * G + z0) * G + y) * G;
#pragma unroll 1
  for (int u = tid; u < K::UA; u += NT) {
    const int zl = u / X2, m2 = u - zl * X2;
    C v[X1];
#pragma unroll
    for (int k1 = 0; k1 < X1; ++k1) v[k1] = S[srow<SP, X1>(m2 * X1) + k1 * SP + zl];
    if constexpr (PER) dft<X1, 1, 1>(v);
    else dft_halfout<X1, 1>(v);
    C* row = reinterpret_cast<C*>(Vz + (long long)zl * G * G) + m2;
#pragma unroll
    for (int m1 = 0; m1 < XOUT; ++m1) row[X2 * m1] = v[m1];
  }
}

}  // namespace exx

// hydro_mixed_planes.cuh -- one sub-grid of the mixed-precision hydro step as
// a plane sweep: each of the 13 lines through a cell is reconstructed once,
// and what a flux needs of a line's end is computed once with it.
//
// The row sweep (hydro_mixed_body.cuh) gives every thread one row of cells
// along one axis and reconstructs, at each cell of the row, the 9 lines that
// cross its faces of that axis: 27 line evaluations per cell for 13 distinct
// lines, and the sound speed and energy of an edge's or corner's state once
// per face at it, 54 per cell for 26.  Here one CTA of kThreadsPl threads per
// SM sweeps the sub-grid plane by plane along z (k = -1 .. N), each step in
// two phases:
//   A  reconstruct plane k: the 13 lines of its interior cells, the 9 lines
//      of the face-adjacent ghost cells around it (x = -1, N and y = -1, N)
//      and, on the planes k = -1 and N, the 9 lines that cross the z-faces;
//      both ends of every line go to shared memory as records of 13 floats
//      (rho v | E tau p c^2 | z species | 1/c), the ends towards +z into one of
//      two z-buffers that the next step reads;
//   B  the fluxes of the x- and y-faces of plane k and of the z-faces between
//      planes k-1 and k, one thread per group of a face's points (the groups
//      of its summation order, listed group by group so that a warp's threads
//      have equal work), into group sums in shared memory; meanwhile the next
//      primitive plane arrives;
//   C  (in the interval of phase A of the next step) per cell and quantity, the
//      FP64 differences of the face sums: x plus y of plane k, and z of plane
//      k - 1, whose total goes to the CTA's scratch in global memory; two steps
//      later two warps finish the plane from there (divergence, sources and
//      update: finish_cell).
// The FP64 pipe takes 16 cycles for a warp's instruction, so its work (C, the
// finish, the conversion of the next plane's state) is spread over the steps,
// beside the lines' FP32 work of other warps, and C's operands are widened on
// the integer pipes.
//
// What bounds it: the latency of its intervals with 20 warps and one tile per
// SM (phase A alone 25 us of a tile's 90, the face fluxes 14, phase C 15, the
// conversion of a padded FP64 state 14, the first planes and the last finish
// 25; measured with the others left out).  A row sweep with two tiles on the
// SM overlaps them and takes 146 us for the two, but 105 for one alone, so the
// dispatch gives this sweep the batches of at most one tile per SM (77 leaves
// with contact steepening and spin: 173 -> 102 us).  Two fields of a line share
// each packed instruction in phase A, and two fields of a point in phase B:
// the records' float4 quarters are register pairs as they are loaded.  The
// primitives live in a ring of six FP32 planes (the five planes a line of
// plane k reaches, and the one arriving), so the CTA holds 225 KB of shared
// memory.
//
// The arithmetic is the row sweep's own: the same ppm32x2 on the same samples
// (exactly symmetric under reversal of a line, so the orientation in which a
// line is evaluated does not matter; each lane rounds alike whichever field
// or line shares its instruction), the same point flux on the same points
// in the same order, the same grouping of each face sum, the same FP64 differences and finish_cell.  The two
// decompositions therefore give the same bits.
#pragma once
#include <type_traits>

#include "hydro_mixed_body.cuh"

namespace hyd {

// 20 warps, one CTA per SM, at 96 registers a thread: phase A's 35 warps of
// lines are two rounds, with phase C's second items on the warps that have one
// line; phase B's 21 warps of face groups go one to a warp, the last beside
// another of two points.
constexpr int kThreadsPl = 640;
constexpr int kWarpsPl = kThreadsPl / 32;
constexpr int kPl = S * S;                // 196 cells of a padded plane
constexpr int kRing = 6;                  // primitive planes held
constexpr int kNN = N * N;                // 64 cells of an interior plane
constexpr int kNFaceXY = 2 * (N + 1) * N; // x- and y-faces of a plane (144)
constexpr int kNFace = kNFaceXY + kNN;    // and the z-faces below it (208)
constexpr int kFaceWarps = (kNFace + 31) / 32;  // 7
constexpr int kSlots = 36;                // line-end slots of a plane's cells (r_slot)
// A slot holds the records of one direction's ends at the 64 cells of a plane
// (kBndB: at the 8 ghost cells along a side): three float4 quarters, then 1/c.
constexpr int kSlotB = 52 * kNN, kBndB = 52 * N;

// Shared-memory layout of one CTA (offsets in bytes).
struct PlaneSmem {
  static constexpr int ring = 0;                                    // float2 [kRing][5][kPl]
  static constexpr int ends = ring + 8 * kRing * 5 * kPl;           // [kSlots] of kSlotB bytes
  static constexpr int bnd = ends + kSlots * kSlotB;                // [4][9] of kBndB bytes
  static constexpr int sums = bnd + 4 * 9 * kBndB;                  // float [3][F + 3][kNFace]
  static constexpr int coord = sums + 4 * 3 * (F + 3) * kNFace;     // float [2][N + 2]
  static constexpr int red = coord + 4 * 2 * (N + 2);               // float [kWarpsPl]
  static constexpr int stage = (red + 4 * kWarpsPl + 15) / 16 * 16; // double [F][kPl] (Io without primitives)
  static constexpr int total = stage + 8 * F * kPl;
};
constexpr size_t kPlaneSmemBytes = PlaneSmem::total;
static_assert(kPlaneSmemBytes <= 227 * 1024, "plane sweep shared memory");

// Direction code of d in {-1,0,1}^3: (dz+1)*9 + (dy+1)*3 + (dx+1); 13 is 0.
// The ends of a plane's interior cells lie in slot `code`, those towards +z
// (code >= 18) in slot code or code + 9 by the parity of the plane.
__device__ __forceinline__ int r_slot(int code, int k) { return code + (code >= 18 ? 9 * (k & 1) : 0); }
// Ghost cells: side sd (0: x = -1, 1: x = N, 2: y = -1, 3: y = N), the side's
// 9 directions into the sub-grid bi = (u2+1)*3 + (u1+1) ((+-1, u1, u2) for x
// sides, (u1, +-1, u2) for y sides), position pos along the side.
__device__ __forceinline__ int bnd_off(int sd, int bi, int pos) { return (sd * 9 + bi) * kBndB + 16 * pos; }

// Lane l of a warp that covers half of an 8 x 8 plane (half hf): x runs
// fastest and the two rows a half-warp reads as 8-byte pairs are four rows
// (448 bytes of the ring) apart, on the other half of the banks.
__device__ __forceinline__ int half_cell(int l, int hf) {
  const int y = ((l >> 3) & 1) * 4 + (l >> 4) + 2 * hf;
  return y * N + (l & 7);
}

// One work item of phase A: the line of the cell at padded plane coordinates
// (ix, iy) along (dx, dy, dz); zo: the ring offsets of the planes k-2 .. k+2.
// dp, dm: the records of the ends towards +d and -d (dm null: not needed), of
// position pos among cnt (the slot's cells).  kContact as line10fc: the
// density and species lines (lane x of pair 0, lane y of pair 4) are
// steepened.
template <bool kContact, bool kSpin>
__device__ __forceinline__ void plane_line(const float2* __restrict__ ring, int ix, int iy, const int zo[5], int dx,
                                           int dy, int dz, unsigned char* dp, unsigned char* dm, int pos, int cnt,
                                           const StepParamsF& PF) {
  const float2* v[5];
  const int c = iy * S + ix, cd = dy * S + dx;
#pragma unroll
  for (int m = 0; m < 5; ++m) v[m] = ring + ((dz == 0 ? zo[2] : dz > 0 ? zo[m] : zo[4 - m]) + c + (m - 2) * cd);
  bool contact = false;
  if (kContact)
    contact = contact_line32(v[1][0].x, v[3][0].x, __fmul_rn(PF.gm1, v[1][2 * kPl].x),
                             __fmul_rn(PF.gm1, v[3][2 * kPl].x), __fmul_rn(PF.gamma, 0.1f));
  // pair f (fields 2f, 2f + 1)
  auto pair = [&](auto fc, float2& qp, float2& qm) {
    constexpr int f = decltype(fc)::value;
    const float2 s0 = v[0][f * kPl], s1 = v[1][f * kPl], s2 = v[2][f * kPl], s3 = v[3][f * kPl], s4 = v[4][f * kPl];
    if constexpr (kContact && (f == 0 || f == 4)) {
      const float eta = !contact ? 0.f
                        : f == 0 ? contact_eta32(s0.x, s1.x, s2.x, s3.x, s4.x)
                                 : contact_eta32(s0.y, s1.y, s2.y, s3.y, s4.y);
      ppm32x2<f == 0 ? 2 : 3>(s0, s1, s2, s3, s4, qp, qm, f2(eta));
    } else {
      ppm32x2(s0, s1, s2, s3, s4, qp, qm);
    }
  };
  using std::integral_constant;
  auto quarter = [&](unsigned char* d, int i, float2 a, float2 b) {
    *reinterpret_cast<float4*>(d + i * 16 * cnt) = make_float4(a.x, a.y, b.x, b.y);
  };
  float2 p0, m0, p1, m1, p2, m2;
  pair(integral_constant<int, 3>{}, p0, m0);
  pair(integral_constant<int, 4>{}, p1, m1);
  quarter(dp, 2, p0, p1);
  if (dm) quarter(dm, 2, m0, m1);
  pair(integral_constant<int, 0>{}, p0, m0);
  pair(integral_constant<int, 1>{}, p1, m1);
  if constexpr (kSpin) {
    // the cell's spin fed back into the velocity at both ends (spin_dv32;
    // the row sweep's values, bit for bit)
    float dv[3];
    spin_dv32(v[2][0].x, v[2][2 * kPl].x, v[2][3 * kPl].x, v[2][3 * kPl].y, v[2][4 * kPl].x, PF.k3h,
              __fmul_rn(PF.gamma, PF.gm1), dx, dy, dz, dv);
    p0.y = __fadd_rn(p0.y, dv[0]);
    m0.y = __fsub_rn(m0.y, dv[0]);
    p1.x = __fadd_rn(p1.x, dv[1]);
    m1.x = __fsub_rn(m1.x, dv[1]);
    p1.y = __fadd_rn(p1.y, dv[2]);
    m1.y = __fsub_rn(m1.y, dv[2]);
  }
  quarter(dp, 0, p0, p1);
  if (dm) quarter(dm, 0, m0, m1);
  pair(integral_constant<int, 2>{}, p2, m2);
  // E, p, c^2 and 1/c of an end (point32's operations)
  auto end = [&](unsigned char* d, float2 q0, float2 q1, float2 q2) {
    const float v2 = __fmaf_rn(q1.y, q1.y, __fmaf_rn(q1.x, q1.x, __fmul_rn(q0.y, q0.y)));
    const float E = __fmaf_rn(__fmul_rn(0.5f, q0.x), v2, q2.x);
    const float p = __fmul_rn(PF.gm1, q2.x);
    const float c2 = __fdividef(__fmul_rn(PF.gamma, p), q0.x);
    quarter(d, 1, f2(E, q2.y), f2(p, c2));
    *reinterpret_cast<float*>(d + 48 * cnt - 12 * pos) = rsqrtf(c2);
  };
  end(dp, p0, p1, p2);
  if (dm) end(dm, m0, m1, m2);
}

// One face side of a thread's points: where the record of point (u1, u2)
// lies, base + u1 s1 + u2 s2 + (u2 == 1 ? s3 : 0) bytes, quarters qst bytes
// apart, its 1/c at dr.
struct SideRef {
  const unsigned char* base;
  int s1, s2, s3, qst, dr;
  template <int u1, int u2>
  __device__ __forceinline__ void load(float4 q[3], float& rs) const {
    const unsigned char* p = base + u1 * s1 + u2 * s2 + (u2 == 1 ? s3 : 0);
#pragma unroll
    for (int i = 0; i < 3; ++i) q[i] = *reinterpret_cast<const float4*>(p + i * qst);
    rs = *reinterpret_cast<const float*>(p + dr);
  }
};

// One quadrature point of a face (point32's operations,
// two fields in the two lanes), added to a group's sums G (field pairs) and
// the torque about the left cell TL.  w: the point's weight.
template <int u1, int u2>
__device__ __forceinline__ void plane_point(const SideRef& sl, const SideRef& sr, int a, float om, float r,
                                            float half_h, float w, float2 G[5], float TL[3], float& amax) {
  float4 L[3], R[3];
  float rsL, rsR;
  sl.load<u1, u2>(L, rsL);
  sr.load<u1, u2>(R, rsR);
  const float hw = 0.5f * w, hq = 0.5f * __fmul_rn(w, half_h);
  const float vaL = a == 0 ? L[0].y : a == 1 ? L[0].z : L[0].w, vaR = a == 0 ? R[0].y : a == 1 ? R[0].z : R[0].w;
  const float unL = __fmaf_rn(om, r, vaL), unR = __fmaf_rn(om, r, vaR);
  const float aq = fmaxf(__fmaf_rn(L[1].w, rsL, fabsf(unL)), __fmaf_rn(R[1].w, rsR, fabsf(unR)));
  amax = fmaxf(amax, aq);
  const float2 uL2 = f2(unL), uR2 = f2(unR), na2 = f2(-aq), hw2 = f2(hw);
  const float pp = __fadd_rn(L[1].z, R[1].z);
  const float pw = __fmaf_rn(L[1].z, vaL, __fmul_rn(R[1].z, vaR));
  // 2 F_q of two fields with conserved values cL, cR and the pressure term x
  auto flux = [&](float2 cL, float2 cR, float2 x) {
    const float2 sum = fma2(cL, uL2, fma2(cR, uR2, x));
    return fma2(na2, sub2(cR, cL), sum);
  };
  auto flux0 = [&](float2 cL, float2 cR) {
    const float2 sum = fma2(cL, uL2, mul2(cR, uR2));
    return fma2(na2, sub2(cR, cL), sum);
  };
  const float2 f01 = flux(f2(L[0].x, __fmul_rn(L[0].x, L[0].y)), f2(R[0].x, __fmul_rn(R[0].x, R[0].y)),
                          f2(0.f, a == 0 ? pp : 0.f));
  const float2 f23 = flux(mul2(f2(L[0].x), f2(L[0].z, L[0].w)), mul2(f2(R[0].x), f2(R[0].z, R[0].w)),
                          f2(a == 1 ? pp : 0.f, a == 2 ? pp : 0.f));
  const float2 f45 = flux(f2(L[1].x, L[1].y), f2(R[1].x, R[1].y), f2(pw, 0.f));
  const float2 f67 = flux0(f2(L[2].x, L[2].y), f2(R[2].x, R[2].y));
  const float2 f89 = flux0(f2(L[2].z, L[2].w), f2(R[2].z, R[2].w));
  G[0] = fma2(hw2, f01, G[0]);
  G[1] = fma2(hw2, f23, G[1]);
  G[2] = fma2(hw2, f45, G[2]);
  G[3] = fma2(hw2, f67, G[3]);
  G[4] = fma2(hw2, f89, G[4]);
  const float d0 = a == 0 ? 1.f : (float)u1, d1 = a == 1 ? 1.f : (a == 0 ? (float)u1 : (float)u2),
              d2 = a == 2 ? 1.f : (float)u2;
  const float fx = f01.y, fy = f23.x, fz = f23.y;
  TL[0] = __fmaf_rn(hq, __fmaf_rn(d1, fz, __fmul_rn(-d2, fy)), TL[0]);
  TL[1] = __fmaf_rn(hq, __fmaf_rn(d2, fx, __fmul_rn(-d0, fz)), TL[1]);
  TL[2] = __fmaf_rn(hq, __fmaf_rn(d0, fy, __fmul_rn(-d1, fx)), TL[2]);
}

// Phase C's item j (0 or 1) of a thread: the second ones go to the last warps.
__device__ __forceinline__ int phase_c_item(int tid, int j) {
  constexpr int kFirst2 = 2 * kThreadsPl - (F + 3) * kNN;  // the first thread with a second item
  static_assert(kFirst2 >= 0 && kFirst2 % 32 == 0, "phase C items");
  return j == 0 ? tid : tid >= kFirst2 ? kThreadsPl + tid - kFirst2 : (F + 3) * kNN;
}

// cp.async of 8 or 16 bytes to shared memory, and the wait for all of the
// thread's copies.
template <int kBytes>
__device__ __forceinline__ void cp_async(void* dst, const void* src) {
  if constexpr (kBytes == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(smem_u32(dst)), "l"(src), "n"(kBytes) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// One 8^3 tile (work unit s) as a plane sweep; Io as for mixed_subgrid, plus
//   Io::kPrims: io.prim_pairs(sub, c) the five primitive pairs of padded cell
//     c (float2, io.kPairStride apart);
//   else, Io::kRows: io.row(sub, k, z, y) the row of field k of the padded
//     state (14 doubles, 16-byte aligned);
//   else io.load_fields(sub, c, f0, nf, u), fields f0 .. f0+nf-1 of cell c.
// sm: the CTA's dynamic shared memory (kPlaneSmemBytes); D: its scratch
// (kScratchPerSub doubles).  Ends with a barrier.  Must be called by all
// kThreadsPl threads.
template <bool kContact, bool kSpin, class Io>
__device__ __forceinline__ void mixed_subgrid_planes(const StepArgs64& A, const Io& io, int s, unsigned char* sm,
                                                     double* __restrict__ D) {
  float2* ring = reinterpret_cast<float2*>(sm + PlaneSmem::ring);
  unsigned char* ends = sm + PlaneSmem::ends;
  unsigned char* bnd = sm + PlaneSmem::bnd;
  float* sums = reinterpret_cast<float*>(sm + PlaneSmem::sums);
  float* coord = reinterpret_cast<float*>(sm + PlaneSmem::coord);
  float* red = reinterpret_cast<float*>(sm + PlaneSmem::red);
  double* stage = reinterpret_cast<double*>(sm + PlaneSmem::stage);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const typename Io::Sub sub = io.begin(s);
  const int si = io.sidx(sub), offx = io.offx(sub), offy = io.offy(sub);
  const double hd = A.h[si];
  const StepParamsF PF{(float)A.P.gamma, (float)A.P.gm1, (float)A.P.omega, kSpin ? 1 : 0,
                       kSpin ? (float)(3.0 / hd) : 0.f};
  const float h = (float)hd, half_h = 0.5f * h;
  const int npt = A.P.face_points;
  float amax = 0.f;
  bool bad = false;

  // primitives of one padded cell into the ring (cell q of padded plane z)
  auto convert = [&](const double* u, int z, int q) {
    float pq[F];
    bad |= !prims_mixed(u, A.P.eta1, PF.gamma, pq);
    float2* dst = ring + (z % kRing) * (5 * kPl) + q;
#pragma unroll
    for (int f = 0; f < 5; ++f) dst[f * kPl] = f2(pq[2 * f], pq[2 * f + 1]);
  };
  // the asynchronous copies of cell q of padded plane z's primitives
  auto copy_prims = [&](int z, int q) {
    if constexpr (Io::kPrims) {
      const float2* src = io.prim_pairs(sub, z * kPl + q);
      float2* dst = ring + (z % kRing) * (5 * kPl) + q;
#pragma unroll
      for (int f = 0; f < 5; ++f) cp_async<8>(dst + f * kPl, src + (size_t)f * Io::kPairStride);
    }
  };

  {
    const double ox = A.origin[3 * si + 0], oy = A.origin[3 * si + 1];
    sub_coords(coord, hd, ox, oy, offx, offy);
  }

  // ---- planes 0..4 of the padded sub-grid, straight into the ring --------
  for (int e = tid; e < 5 * kPl; e += kThreadsPl) {
    if constexpr (Io::kPrims) {
      copy_prims(e / kPl, e % kPl);
    } else {
      double u[F];
      io.load_fields(sub, e, 0, 5, u);
      io.load_fields(sub, e, 5, 5, u + 5);
      convert(u, e / kPl, e % kPl);
    }
  }
  if constexpr (Io::kPrims) cp_async_wait();
  __syncthreads();

  // phase C's items: quantity q (the F fluxes, then the torque's components)
  // of one cell of the plane; each carries the x plus y difference of the
  // plane before and the z-face sum below the plane after
  constexpr int kItems = 2;
  double d01[kItems];
  float zlo[kItems];
#pragma unroll
  for (int j = 0; j < kItems; ++j) {
    d01[j] = 0.0;
    zlo[j] = 0.f;
  }
  auto phase_c = [&](int k) {
    // the face's sum (G0 + G1) + G2 of value q (the centre alone with one point)
    auto total = [&](int q, int face) {
      const float* g = sums + q * kNFace + face;
      constexpr int kG = (F + 3) * kNFace;
      return npt == 1 ? g[2 * kG] : __fadd_rn(__fadd_rn(g[0], g[kG]), g[2 * kG]);
    };
    // component m of the torque about the right cell (right_torque32)
    auto right = [&](int m, int a, int face) {
      const float tl = total(F + m, face);
      if (m == a) return tl;
      const bool plus = m == (a == 2 ? 0 : a + 1);
      return __fmaf_rn(plus ? h : -h, total(SX + 3 - a - m, face), tl);
    };
#pragma unroll
    for (int j = 0; j < kItems; ++j) {
      const int i = phase_c_item(tid, j);
      if (i < (F + 3) * kNN) {
        const int q = i / kNN, cell = i % kNN, x = cell % N, y = cell / N;
        auto lower = [&](int a, int face) { return q < F ? total(q, face) : right(q - F, a, face); };
        const float zu = total(q, kNFaceXY + cell), zl = lower(2, kNFaceXY + cell);
        if (k >= 1)
          D[(size_t)q * N3 + (k - 1) * kNN + cell] = __dadd_rn(d01[j], __dsub_rn(widen(zu), widen(zlo[j])));
        zlo[j] = zl;
        float xu = 0.f, xl = 0.f, yu = 0.f, yl = 0.f;
        if (k < N) {
          const int fx = y * (N + 1) + x, fy = N * (N + 1) + cell;  // the lower faces
          xu = total(q, fx + 1);
          xl = lower(0, fx);
          yu = total(q, fy + N);
          yl = lower(1, fy);
          d01[j] = __dadd_rn(__dsub_rn(widen(xu), widen(xl)), __dsub_rn(widen(yu), widen(yl)));
        }
        if (A.face_flux) {
          // sub-grid boundary faces: sums and the torque about the interior cell
          if (k < N) {
            if (x == 0) io.face(sub, 0, q, k, y, widen(xl));
            if (x == N - 1) io.face(sub, 1, q, k, y, widen(xu));
            if (y == 0) io.face(sub, 2, q, k, x, widen(yl));
            if (y == N - 1) io.face(sub, 3, q, k, x, widen(yu));
          }
          if (k == 0) io.face(sub, 4, q, y, x, widen(zl));
          if (k == N) io.face(sub, 5, q, y, x, widen(zu));
        }
      }
    }
  };

  // the copies of padded plane z's state into the stage (Io without
  // primitives): rows asynchronously, else through this thread's registers
  double pf[5];
  const int pf_q = tid % kPl, pf_f0 = (tid / kPl) * 5;
  auto stage_issue = [&](int z) {
    if constexpr (Io::kRows) {
      // 14 rows of 7 16-byte pieces per field
      for (int i = tid; i < F * kPl / 2; i += kThreadsPl) {
        const int f = i / (kPl / 2), r = i % (kPl / 2), y = r / (S / 2), x2 = r % (S / 2);
        cp_async<16>(stage + f * kPl + 2 * r, io.row(sub, f, z, y) + 2 * x2);
      }
    } else if constexpr (!Io::kPrims) {
      if (tid < 2 * kPl) io.load_fields(sub, z * kPl + pf_q, pf_f0, 5, pf);
    }
  };
  auto stage_arrive = [&]() {
    if constexpr (Io::kRows || Io::kPrims) {
      cp_async_wait();
    } else {
      if (tid < 2 * kPl) {
#pragma unroll
        for (int f = 0; f < 5; ++f) stage[(pf_f0 + f) * kPl + pf_q] = pf[f];
      }
    }
  };
  // the finish of plane p, by the 64 threads t0 .. t0 + 63
  const double inv_h = 1.0 / hd;
  auto finish_plane = [&](int p, int t0) {
    const int c2 = tid - t0, c = p * kNN + c2;
    if (c2 < 0 || c2 >= kNN) return;
    const double o[3] = {A.origin[3 * si + 0], A.origin[3 * si + 1], A.origin[3 * si + 2]};
    finish_cell(A, io, sub, offx, offy, c2 % N, c2 / N, p, [&](int q) { return D[(size_t)q * N3 + c]; }, hd, inv_h, o);
  };
  // warps with one line item (the last five) finish a plane (two of them) and
  // convert the staged one (the others)
  constexpr int kOneLine = 35 - kWarpsPl;  // 15: the first warp with one item
  constexpr int kConvT0 = (kOneLine + 2) * 32;

  if constexpr (!Io::kPrims) {
    stage_issue(5);
    stage_arrive();
    __syncthreads();
  }
#pragma unroll 1
  for (int k = -1; k <= N; ++k) {
    const int zpk = k + G;  // padded index of plane k
    // the next padded plane, k + 6 (its ring slot is plane k's own padded
    // index, which phase A no longer reads)
    const int znew = k + 6;
    if constexpr (Io::kPrims) {
      if (znew < S && tid < kPl) copy_prims(znew, tid);
    }

    // ---- A: reconstruct plane k; C of the step before; the finish of plane
    // k - 3; the conversion of padded plane k + 6.  The FP64 pipe serves C, the
    // finish and the conversion while the lines run: even warps take C first.
    const bool c_first = (warp & 1) == 0;
    if (k >= 1 && c_first) phase_c(k - 1);
    const bool inner = k >= 0 && k < N;
    const int n_int = inner ? (npt == 1 ? 6 : 26) : (npt == 1 ? 2 : 18);     // halves of planes of cells
    const int n_bnd = inner ? (npt == 1 ? 1 : 9) : 0;                        // 32 ghost-cell lines each
    int zo[5];
#pragma unroll
    for (int m = 0; m < 5; ++m) zo[m] = ((zpk + m - 2) % kRing) * (5 * kPl);
#pragma unroll 1
    for (int i = warp; i < n_int + n_bnd; i += kWarpsPl) {
      int ix, iy, dx, dy, dz, pos, cnt;
      unsigned char *dp, *dm;
      if (i < n_int) {
        const int cell = half_cell(lane, i & 1), L = i >> 1;
        int code;
        if (inner)
          code = npt == 1 ? (L == 0 ? 14 : L == 1 ? 16 : 22) : 14 + L;  // the lines with d's code above 13
        else
          code = (k < 0 ? 18 : 0) + (npt == 1 ? 4 : L);  // towards +z from k = -1, towards -z from k = N
        dx = code % 3 - 1;
        dy = (code / 3) % 3 - 1;
        dz = code / 9 - 1;
        ix = cell % N + G;
        iy = cell / N + G;
        pos = cell;
        cnt = kNN;
        dp = ends + r_slot(code, k) * kSlotB + 16 * cell;
        dm = inner ? ends + r_slot(26 - code, k) * kSlotB + 16 * cell : nullptr;
      } else {
        // face-adjacent ghost cells: the 9 lines into the sub-grid (the middle
        // one alone with one point)
        const int j = (i - n_int) * 32 + lane;
        const int sd = npt == 1 ? j / N : j / (9 * N), bi = npt == 1 ? 4 : (j / N) % 9;
        const int u1 = bi % 3 - 1, in = (sd & 1) ? -1 : 1, out = (sd & 1) ? N : -1;
        pos = j % N;
        cnt = N;
        dz = bi / 3 - 1;
        dx = sd < 2 ? in : u1;
        dy = sd < 2 ? u1 : in;
        ix = (sd < 2 ? out : pos) + G;
        iy = (sd < 2 ? pos : out) + G;
        dp = bnd + bnd_off(sd, bi, pos);
        dm = nullptr;
      }
      plane_line<kContact, kSpin>(ring, ix, iy, zo, dx, dy, dz, dp, dm, pos, cnt, PF);
    }
    if (k >= 1 && !c_first) phase_c(k - 1);
    if (k >= 3) finish_plane(k - 3, kOneLine * 32);
    if constexpr (!Io::kPrims) {
      if (znew < S && tid >= kConvT0) {
#pragma unroll 1
        for (int q = tid - kConvT0; q < kPl; q += kThreadsPl - kConvT0) {
          double u[F];
#pragma unroll
          for (int f = 0; f < F; ++f) u[f] = stage[f * kPl + q];
          convert(u, znew, q);
        }
      }
    }
    __syncthreads();

    // ---- B: face fluxes; the copies of the next padded plane --------------------
    if constexpr (!Io::kPrims) {
      if (znew + 1 < S) stage_issue(znew + 1);
    }
    if (k >= 0) {
      // items: face `slot` for group 0 (points 0-3), 2 (points 6-8), 1 (4, 5);
      // with one point per face the centre (group 2) alone
      const int n_faces = k < N ? kNFace : kNN, fw = k < N ? kFaceWarps : kNN / 32;
      // (a 21st item goes to a warp of the smallest group, of two points)
      static_assert(3 * kFaceWarps == kWarpsPl + 1, "phase B items");
#pragma unroll 1
      for (int wi = warp; wi < (npt == 1 ? fw : 3 * fw);
           wi = (wi == 2 * kFaceWarps && fw == kFaceWarps) ? 3 * kFaceWarps - 1 : 3 * kFaceWarps) {
        const int part = npt == 1 ? 1 : wi / fw;  // 0, 1, 2: groups 0, 2, 1
        const int f = (npt == 1 ? wi : wi % fw) * 32 + lane;
        if (f >= n_faces) continue;
        const int slot = k < N ? f : kNFaceXY + f;
        // the face's axis and its left cell (fx, fy) in plane k (k - 1 for z)
        int a, fx, fy;
        if (slot < N * (N + 1)) {
          a = 0;
          fy = slot / (N + 1);
          fx = slot % (N + 1) - 1;
        } else if (slot < kNFaceXY) {
          a = 1;
          const int t = slot - N * (N + 1);  // x fastest: neighbouring lanes read neighbouring cells
          fx = t % N;
          fy = t / N - 1;
        } else {
          a = 2;
          fx = (slot - kNFaceXY) % N;
          fy = (slot - kNFaceXY) / N;
        }
        // interior records: code of (1, u1, u2) along (a, b, c), b < c
        const int par = 9 * (k & 1) * kSlotB, parl = 9 * ((k - 1) & 1) * kSlotB;
        const int cb = a == 0 ? 3 : 1, cc = a == 2 ? 3 : 9, ca = a == 0 ? 1 : a == 1 ? 3 : 9;
        const int cell = fy * N + fx;
        SideRef sl, sr;
        sl.base = ends + (13 + ca) * kSlotB + 16 * cell + (a == 2 ? parl : 0);
        sr.base = ends + (13 - ca) * kSlotB + 16 * (cell + (a == 0 ? 1 : a == 1 ? N : 0));
        sl.s1 = sr.s1 = cb * kSlotB;
        sl.s2 = sr.s2 = cc * kSlotB;
        sl.s3 = sr.s3 = a == 2 ? 0 : par;
        sl.qst = sr.qst = 16 * kNN;
        sl.dr = 48 * kNN - 12 * cell;
        sr.dr = 48 * kNN - 12 * (cell + (a == 0 ? 1 : a == 1 ? N : 0));
        if (a < 2) {
          const int fa = a == 0 ? fx : fy, pos = a == 0 ? fy : fx;
          if (fa < 0) {
            sl.base = bnd + bnd_off(2 * a, 4, pos);
            sl.s1 = bnd_off(0, 1, 0);
            sl.s2 = bnd_off(0, 3, 0);
            sl.s3 = 0;
            sl.qst = 16 * N;
            sl.dr = 48 * N - 12 * pos;
          }
          if (fa + 1 >= N) {
            sr.base = bnd + bnd_off(2 * a + 1, 4, pos);
            sr.s1 = bnd_off(0, 1, 0);
            sr.s2 = bnd_off(0, 3, 0);
            sr.s3 = 0;
            sr.qst = 16 * N;
            sr.dr = 48 * N - 12 * pos;
          }
        }
        // the coordinate that the frame velocity's normal component takes (y_q
        // for x-faces, x_q for y-faces; none for z) by the offset along b
        const float om = a == 0 ? PF.omega : a == 1 ? -PF.omega : 0.f;
        const float cen = a == 0 ? coord[(N + 2) + fy + 1] : coord[fx + 1];
        const float rp = __fmaf_rn(half_h, 1.f, cen), rm = __fmaf_rn(half_h, -1.f, cen);
        constexpr float w1 = 1.f / 36.f, w4 = 4.f / 36.f, w16 = 16.f / 36.f;
        float2 Gs[5];
        float TL[3] = {0.f, 0.f, 0.f};
#pragma unroll
        for (int q = 0; q < 5; ++q) Gs[q] = f2(0.f);
        int g;
        // the points of the groups in the face's order (face_u1, face_u2)
        if (part == 0) {
          g = 0;
          plane_point<1, 1>(sl, sr, a, om, rp, half_h, w1, Gs, TL, amax);
          plane_point<-1, -1>(sl, sr, a, om, rm, half_h, w1, Gs, TL, amax);
          plane_point<1, 0>(sl, sr, a, om, rp, half_h, w4, Gs, TL, amax);
          plane_point<-1, 0>(sl, sr, a, om, rm, half_h, w4, Gs, TL, amax);
        } else if (part == 1) {
          g = 2;
          if (npt != 1) {
            plane_point<0, 1>(sl, sr, a, om, cen, half_h, w4, Gs, TL, amax);
            plane_point<0, -1>(sl, sr, a, om, cen, half_h, w4, Gs, TL, amax);
          }
          plane_point<0, 0>(sl, sr, a, om, cen, half_h, npt == 1 ? 1.f : w16, Gs, TL, amax);
        } else {
          g = 1;
          plane_point<1, -1>(sl, sr, a, om, rp, half_h, w1, Gs, TL, amax);
          plane_point<-1, 1>(sl, sr, a, om, rm, half_h, w1, Gs, TL, amax);
        }
        float* out = sums + g * (F + 3) * kNFace + slot;
#pragma unroll
        for (int q = 0; q < 5; ++q) {
          out[(2 * q) * kNFace] = Gs[q].x;
          out[(2 * q + 1) * kNFace] = Gs[q].y;
        }
#pragma unroll
        for (int m = 0; m < 3; ++m) out[(F + m) * kNFace] = TL[m];
      }
    }
    if (Io::kPrims || znew + 1 < S) stage_arrive();
    __syncthreads();
  }
  phase_c(N);
  // ---- amax and the status ------------------------------------------------
#pragma unroll
  for (int o2 = 16; o2 > 0; o2 >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o2));
  if (lane == 0) red[warp] = amax;
  if (bad) atomicOr(A.status, 1u);
  __syncthreads();
  // the last two planes
  finish_plane(N - 2, 0);
  finish_plane(N - 1, 2 * 32);
  if (tid == kThreadsPl - 1) {
    float m = red[0];
#pragma unroll
    for (int w = 1; w < kWarpsPl; ++w) m = fmaxf(m, red[w]);
    io.amax(sub, (double)m);
  }
  __syncthreads();
}

}  // namespace hyd

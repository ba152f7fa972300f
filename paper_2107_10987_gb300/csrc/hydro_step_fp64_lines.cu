// hydro_step_fp64_lines.cu -- the per-sub-grid hydro step in FP64 with every
// PPM line evaluated once per cell.
//
// The same method, arithmetic and face-sum order as hydro_step_fp64.cu (and
// the same bits), organised around the 13 line directions of Sec. III-B
// instead of the three axis sweeps.  A face point lies on the surface of its
// two cells: the face centres use the axis lines, the edge midpoints (shared
// by two faces of a cell) the 6 edge lines and the corners (shared by three
// faces) the 4 vertex lines, so an axis sweep that reconstructs its own 9
// lines per cell evaluates 27 line-fields per cell where 13 are unique.
// A team of T CTAs of 384 threads, one CTA per SM, works on one 8^3 tile at a
// time (T = 1: a persistent loop of independent CTAs; T > 1: a cooperative
// launch, the CTAs of a team meeting at bounded barriers in global memory):
//   1. the tile's primitives into shared memory: T = 1 stages the
//      ghost-padded state by bulk TMA copies (the next tile's copies are
//      issued as soon as phase 3 no longer reads it, so they overlap phases 4
//      and 5) and converts in place; a larger team converts each cell once,
//      into a buffer in global memory that every CTA then copies;
//   2. (learned smoothness indicator, optional) its per-cell decisions;
//   3. lines: one work item per (field group, run), a run being a maximal segment
//      of consecutive cells along one of the 13 directions d among the cells
//      that need that line (the interior, and the face-adjacent ghost cells
//      of the faces whose normal component of d is nonzero).  The item walks
//      its run with a sliding window, so that the differences, the MC slopes
//      and the unlimited interface value between two cells of the run are
//      computed once for both cells (PPM's interface value at x + d/2 is one
//      number for the cell x and its neighbour x + d), then applies the
//      per-cell steepening and monotonicity fix-ups and stores both
//      interface values of the cell in a per-team buffer in global memory
//      (read back from L2 or DRAM in phase 4).  The group of rho, v, eps and
//      tau also stores what the flux needs of the state (end64: p, E, c), once
//      per line end where the up to three faces at it would each compute it;
//   4. faces: one work item per face sums its 9 Kurganov-Tadmor point fluxes
//      with the Simpson weights from the stored ends, into the team's buffer
//      of face sums;
//   5. divergence, sources and dU/dt as in hydro_step_fp64.cu.
// Runs are listed once per device, longest first, so that the lanes of a
// warp mostly walk runs of equal length; items are dealt out a warp at a time
// over the team.  The walk's arithmetic is ppm64's, operation for operation,
// on the same operands (the reversed line gives the mirrored values bit for
// bit), so the stored values are those the axis sweeps compute, and the
// results depend neither on T nor on the number of teams.
//
// What bounds it: the FP64 pipe, which issues a warp's instruction every 16
// cycles per SM.  12 warps keep it busy without prefetching (6 warps held it
// at 83 %), and the work is cut to the pipe's: decisions on bit patterns,
// masks instead of |x| and -x, an interface value from both its sides at once,
// line ends' sound speeds shared, unread ends of ghost cells left out, and the
// flux in two fused steps per field.  A tile of random data takes a CTA 0.664
// ms (about 1.09 before); the RK3 step of a 512-sub-grid blast 13.0 -> 7.05 ms.
// Teams serve the batches that do not fill whole rounds of the SMs
// (step_fp64_choose_team): 512 tiles take pairs of CTAs 2.45 ms and single
// ones 2.62, one tile takes a team of 46 CTAs 0.081 ms and one CTA 0.647.
#include <algorithm>
#include <vector>

#include "hydro.h"
#include "hydro_common.cuh"
#include "hydro_fp64.cuh"
#include "hydro_mixed.cuh"

namespace hyd {

constexpr int kLThreads = 384;
constexpr int kLWarps = kLThreads / 32;
constexpr long kLWaitPolls = 1L << 24;

// The line-end buffer of one team: for each of the 26 (direction, end) slots
// and each cell of the 10^3 box of interior cells and their face-adjacent
// ghost layer, a record of 12 doubles in three 32-byte sectors, each written
// whole by one thread: rho v | p E c tau | z species (point64's operands; eps
// itself is not needed past end64): [slot][box cell][kRec] doubles.  Then the
// tile's face sums [kFv][kFaces] (fluxes, torques about the left and the
// right cell), and the padded tile's primitives [F][S3] (teams of more than
// one CTA).
constexpr int kBox = (N + 2) * (N + 2) * (N + 2);  // 1000
constexpr int kRec = 12;
constexpr int kFaces = 3 * (N + 1) * N * N;  // 1728, face (a, j, pc, pb): ((a * 9 + j) * 8 + pc) * 8 + pb
constexpr int kFv = F + 6;
constexpr size_t kEndsPerTeam = (size_t)26 * kBox * kRec;
constexpr size_t kSumsPerTeam = (size_t)kFv * kFaces;
constexpr size_t kLinesPerTeam = kEndsPerTeam + kSumsPerTeam + (size_t)F * S3;

// Directions d with components in {-1, 0, 1}, the first nonzero one
// positive; index 9 dx + 3 dy + dz - 1 in [0, 13).  Slot 2 dd + 0 holds the
// value at x + d/2 of cell x, slot 2 dd + 1 the value at x - d/2.
__host__ __device__ constexpr int dir_index(int dx, int dy, int dz) { return 9 * dx + 3 * dy + dz - 1; }

// Slot of the value at x + w/2 for a nonzero w with components in {-1, 0, 1}.
__device__ __forceinline__ int end_slot(int wx, int wy, int wz) {
  const int sg = wx != 0 ? wx : (wy != 0 ? wy : wz);
  return 2 * dir_index(sg * wx, sg * wy, sg * wz) + (sg > 0 ? 0 : 1);
}

// Run list: one 32-bit word per run, bits 0-11 the shared-memory index of its
// first cell (14^3 layout), 12-21 that cell's box index, 22-25 its length
// (1..10), 26-31 the direction's components plus one (2 bits each, x first).
constexpr int kMaxRuns = 2048;
__device__ uint32_t g_line_runs[kMaxRuns];

// Whether box cell (x, y, z) in [-1, N]^3 needs the line along d: interior
// cells need all 13, a ghost cell only the lines that reach its one face
// (exactly one coordinate outside [0, N), and d nonzero along that axis).
static bool needs_line(int x, int y, int z, int dx, int dy, int dz) {
  const int c[3] = {x, y, z}, d[3] = {dx, dy, dz};
  int out = 0;
  for (int i = 0; i < 3; ++i) {
    if (c[i] < -1 || c[i] > N) return false;
    if (c[i] < 0 || c[i] >= N) {
      if (d[i] == 0) return false;
      ++out;
    }
  }
  return out <= 1;
}

// The runs of all 13 directions, the axis lines' first (they alone serve the
// single-point face flux), each group longest first.
static std::vector<uint32_t> build_line_runs(int* n_axis) {
  struct R {
    int len, axis;
    uint32_t word;
  };
  std::vector<R> runs;
  for (int dx = -1; dx <= 1; ++dx)
    for (int dy = -1; dy <= 1; ++dy)
      for (int dz = -1; dz <= 1; ++dz) {
        const int sg = dx != 0 ? dx : (dy != 0 ? dy : dz);
        if (sg <= 0) continue;  // the zero vector and the reversed directions
        const int axis = (dx != 0) + (dy != 0) + (dz != 0) == 1;
        for (int z = -1; z <= N; ++z)
          for (int y = -1; y <= N; ++y)
            for (int x = -1; x <= N; ++x) {
              if (!needs_line(x, y, z, dx, dy, dz) || needs_line(x - dx, y - dy, z - dz, dx, dy, dz)) continue;
              int len = 0;
              while (needs_line(x + len * dx, y + len * dy, z + len * dz, dx, dy, dz)) ++len;
              const uint32_t smem = (uint32_t)(((z + G) * S + (y + G)) * S + (x + G));
              const uint32_t box = (uint32_t)(((z + 1) * (N + 2) + (y + 1)) * (N + 2) + (x + 1));
              const uint32_t dirs = (uint32_t)(dx + 1) | ((uint32_t)(dy + 1) << 2) | ((uint32_t)(dz + 1) << 4);
              runs.push_back({len, axis, smem | (box << 12) | ((uint32_t)len << 22) | (dirs << 26)});
            }
      }
  std::stable_sort(runs.begin(), runs.end(), [](const R& p, const R& q) {
    if (p.axis != q.axis) return p.axis > q.axis;
    return p.len > q.len;
  });
  std::vector<uint32_t> words;
  *n_axis = 0;
  for (const R& r : runs) {
    words.push_back(r.word);
    *n_axis += r.axis;
  }
  return words;
}

static int g_runs_total = 0, g_runs_axis = 0;

// Four doubles of one 32-byte sector, in one access.
__device__ __forceinline__ void st_sector(double* p, double a, double b, double c, double d) {
  asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p), "d"(a), "d"(b), "d"(c), "d"(d) : "memory");
}
__device__ __forceinline__ void ld_sector(const double* p, double& a, double& b, double& c, double& d) {
  asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];" : "=d"(a), "=d"(b), "=d"(c), "=d"(d) : "l"(p) : "memory");
}

// One work item of phase 3: fields k0 .. k0 + NG - 1 along run word e.  The
// window holds, per field, the samples S(i-2..i+2) of cell i of the run, the
// differences and MC slopes around it and w = S(i) - Q(i - 1/2) of the
// interface value Q; each step loads one sample per field and forms one
// difference, one slope and one interface value from both its sides (ppm64's
// operations on the same operands), then the cell's fix-ups, and stores the group's sectors of both records of the
// cell: fields 0 .. 5 with end64's values the first two, fields 6 .. 9 the
// last.
template <bool kGate, bool kContact, int NG>
__device__ __forceinline__ void line_run(const double* __restrict__ Q, const uint8_t* __restrict__ smooth,
                                         const StepParams& P, double* __restrict__ R, uint32_t e, int k0,
                                         double k3h) {
  const int c0 = (int)(e & 0xfffu), b0 = (int)((e >> 12) & 0x3ffu), n = (int)((e >> 22) & 0xfu);
  const int dx = (int)((e >> 26) & 3u) - 1, dy = (int)((e >> 28) & 3u) - 1, dz = (int)(e >> 30) - 1;
  const int sv = dx + S * dy + S * S * dz;                             // shared-memory stride along d
  const int bv = (dx + (N + 2) * dy + (N + 2) * (N + 2) * dz) * kRec;  // line-buffer stride along d
  static_assert(NG == 6 || NG == 4, "field groups 0 .. 5 and 6 .. 9");
  double* Rp = R + ((size_t)(2 * dir_index(dx, dy, dz)) * kBox + b0) * kRec + (NG == 6 ? 0 : 8);
  double* Rm = Rp + (size_t)kBox * kRec;
  // A ghost cell (the first or the last of a run) has only the end at its face
  // read: towards +d where d points into the tile from it, else towards -d.
  auto outward = [&](int i) {  // bit 0: the +d end is not read, bit 1: the -d end
    const int x = b0 % (N + 2) + i * dx, y = (b0 / (N + 2)) % (N + 2) + i * dy, z = b0 / ((N + 2) * (N + 2)) + i * dz;
    const int in = x == 0 ? dx : x == N + 1 ? -dx : y == 0 ? dy : y == N + 1 ? -dy : z == 0 ? dz : z == N + 1 ? -dz : 0;
    return in == 0 ? 0 : in > 0 ? 2 : 1;
  };
  const int out0 = outward(0), outn = outward(n - 1);
  const double* q = Q + k0 * S3 + c0;
  // the group's steepened field: rho in the first, the species in the second
  const bool steep_group = kContact;
  double sm2[NG], sm1[NG], s0[NG], s1[NG], dr[NG], Dm[NG], Dc[NG], wl[NG];
#pragma unroll
  for (int f = 0; f < NG; ++f) {
    const double* qf = q + f * S3;
    sm2[f] = qf[-2 * sv];
    sm1[f] = qf[-sv];
    s0[f] = qf[0];
    s1[f] = qf[sv];
    const double dl = rsub(s0[f], sm1[f]);
    Dm[f] = slope64(rsub(sm1[f], sm2[f]), dl);  // slope at cell i - 1
    dr[f] = rsub(s1[f], s0[f]);
    Dc[f] = slope64(dl, dr[f]);  // slope at cell i
    double u;
    ppm_sides64(dl, Dm[f], Dc[f], u, wl[f]);  // interface value at i - 1/2
  }
#pragma unroll 1
  for (int i = 0; i < n; ++i) {
    const int ci = c0 + i * sv;
    const bool smooth_i = kGate && smooth[ci];
    const bool contact = steep_group && !smooth_i && contact_line64(Q, ci, sv, P);
    double p[NG], m[NG];
#pragma unroll
    for (int f = 0; f < NG; ++f) {
      const int k = k0 + f;
      const double s2 = q[f * S3 + (i + 2) * sv];
      const double d2 = rsub(s2, s1[f]);
      const double Dp = slope64(dr[f], d2);  // slope at cell i + 1
      double up, wn;
      ppm_sides64(dr[f], Dc[f], Dp, up, wn);
      if (kGate && smooth_i && !(k == ZX || k == ZY || k == ZZ)) {
        // the indicator's unlimited 4-point values (line10u)
        const double c7 = 7.0 / 12.0, c1 = 1.0 / 12.0;
        p[f] = rsub(rmul(c7, radd(s0[f], s1[f])), rmul(c1, radd(sm1[f], s2)));
        m[f] = rsub(rmul(c7, radd(s0[f], sm1[f])), rmul(c1, radd(s1[f], sm2[f])));
      } else {
        if (kContact && contact && (k == RHO || k == SP0)) {
          const double eta = contact_eta64(sm2[f], sm1[f], s0[f], s1[f], s2);
          if (eta > 0.0) ppm_steep_sides64(sm1[f], s0[f], s1[f], Dm[f], Dp, eta, up, wl[f]);
        }
        ppm_limit64(s0[f], up, wl[f], p[f], m[f]);
      }
      sm2[f] = sm1[f];
      sm1[f] = s0[f];
      s0[f] = s1[f];
      s1[f] = s2;
      dr[f] = d2;
      Dm[f] = Dc[f];
      Dc[f] = Dp;
      wl[f] = wn;
    }
    if (NG == 6 && P.spin) {
      // the cell's spin fed back into the velocity at both ends (spin_dv64)
      double dv[3];
      spin_dv64(Q[RHO * S3 + ci], Q[EGAS * S3 + ci], Q[ZX * S3 + ci], Q[ZY * S3 + ci], Q[ZZ * S3 + ci], k3h,
                rmul(P.gamma, P.gm1), dx, dy, dz, dv);
#pragma unroll
      for (int m3 = 0; m3 < 3; ++m3) {
        p[(1 + m3) % NG] = radd(p[(1 + m3) % NG], dv[m3]);
        m[(1 + m3) % NG] = rsub(m[(1 + m3) % NG], dv[m3]);
      }
    }
    const int out = (i == 0 ? out0 : 0) | (i == n - 1 ? outn : 0);
    auto put = [&](double* d, const double(&q)[NG]) {
      st_sector(d, q[0], q[1], q[2], q[3]);
      if (NG == 6) {
        const End64 e = end64(q[0], q[1], q[2], q[3], q[NG > 4 ? 4 : 0], P);
        st_sector(d + 4, e.p, e.E, e.c, q[NG > 5 ? 5 : 0]);
      }
    };
    if (!(out & 1)) put(Rp + i * bv, p);
    if (!(out & 2)) put(Rm + i * bv, m);
  }
}

// line_run of a wild tile (WildTile), both field groups in one item, a cell at a
// time from shared memory; out of line: the ordinary runs keep their registers.
// Both ends of every cell are stored, also those of a ghost cell that are not
// read, and a number at a time: st_sector in an out-of-line function stored its
// first number and zeros.
static __device__ __noinline__ void line_run_wild(const double* __restrict__ Q, const uint8_t* __restrict__ smooth,
                                                  bool contact, const StepParams& P, double* __restrict__ R, uint32_t e,
                                                  double k3h) {
  const int c0 = (int)(e & 0xfffu), b0 = (int)((e >> 12) & 0x3ffu), n = (int)((e >> 22) & 0xfu);
  const int dx = (int)((e >> 26) & 3u) - 1, dy = (int)((e >> 28) & 3u) - 1, dz = (int)(e >> 30) - 1;
  const int sv = dx + S * dy + S * S * dz, bv = dx + (N + 2) * dy + (N + 2) * (N + 2) * dz;
#pragma unroll 1
  for (int i = 0; i < n; ++i) {
    const int ci = c0 + i * sv;
    double q[2][F], dv[3] = {0.0, 0.0, 0.0};
    line10_wild(Q, ci, sv, smooth && smooth[ci], contact, P, q[0], q[1]);
    if (P.spin)
      spin_dv64(Q[RHO * S3 + ci], Q[EGAS * S3 + ci], Q[ZX * S3 + ci], Q[ZY * S3 + ci], Q[ZZ * S3 + ci], k3h,
                rmul(P.gamma, P.gm1), dx, dy, dz, dv);
#pragma unroll 1
    for (int side = 0; side < 2; ++side) {
      const double* v = q[side];
      double vel[3];
#pragma unroll
      for (int m = 0; m < 3; ++m)
        vel[m] = P.spin ? (side ? rsub(v[SX + m], dv[m]) : radd(v[SX + m], dv[m])) : v[SX + m];
      double* d = R + ((size_t)(2 * dir_index(dx, dy, dz) + side) * kBox + b0 + i * bv) * kRec;
      const End64 w = end64(v[RHO], vel[0], vel[1], vel[2], v[EGAS], P);
      const double rec[kRec] = {v[RHO], vel[0], vel[1], vel[2], w.p, w.E, w.c, v[TAU], v[ZX], v[ZY], v[ZZ], v[SP0]};
#pragma unroll
      for (int k = 0; k < kRec; ++k) d[k] = rec[k];
    }
  }
}

// Barrier of a team (T = 1: of the CTA): every thread's earlier writes are
// visible to the team's threads after it.  k counts the team's barriers since
// the launch; sync[0] is the launch's abort word, sync[32 (1 + team)] the
// team's arrivals (zero at the launch).  False, for all threads, if a wait
// expired anywhere.
struct TeamSync {
  unsigned* sync;
  unsigned team, size, k;
  long long wait_ns;
  unsigned* status;
};
__device__ __forceinline__ bool team_barrier(TeamSync& B, int* sh_ok) {
  __syncthreads();
  if (B.size == 1) return true;
  ++B.k;
  if (threadIdx.x == 0) {
    unsigned* arrive = B.sync + 32 * (1 + (size_t)B.team);
    __threadfence();
    atomicAdd(arrive, 1u);
    const bool ok = wait_geq(arrive, B.k * B.size, B.sync, B.wait_ns);
    if (!ok) {
      atomicOr(B.status, 2u);
      atomicExch(B.sync, 1u);
    }
    *sh_ok = ok;
  }
  __syncthreads();
  return *sh_ok != 0;
}

// kGate, kContact, NN: as for hydro_step_fp64_kernel.  A.lines: the per-team
// buffers (kLinesPerTeam doubles each); n_runs: the runs of g_line_runs that
// phase 3 walks (the axis runs alone for the single-point face flux); T: the
// CTAs of a team; sync: TeamSync's words (T > 1), zero at the launch.
template <bool kGate, bool kContact = false, int NN = N>
__global__ void __launch_bounds__(kLThreads, 1)
    hydro_step_fp64_lines_kernel(StepArgs64 A, int n_runs, int T, unsigned* sync, long long wait_ns) {
  using Tl = Tile<NN>;
  extern __shared__ __align__(128) double Q[];  // [F][S3], then the indicator's flags
  uint8_t* smooth = reinterpret_cast<uint8_t*>(Q + F * S3);
  __shared__ __align__(8) uint64_t bar;
  __shared__ double red[kLWarps];
  __shared__ int bail, sh_ok;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int team = blockIdx.x / T, rank = blockIdx.x % T, n_teams = gridDim.x / T;
  double* R = A.lines + (size_t)team * kLinesPerTeam;
  double* Fs = R + kEndsPerTeam;
  double* Pb = Fs + kSumsPerTeam;
  const int n_units = A.n_sub * Tl::kTiles;
  TeamSync B{sync, (unsigned)team, (unsigned)T, 0u, wait_ns, A.status};

  // bulk copies of tile u into Q, completing on bar (warp 0; as in
  // hydro_step_fp64_kernel)
  auto stage = [&](int u) {
    if (tid < 32) {
      const Tl tile(u);
      if (tid == 0) {
        fence_proxy_async();
        mbar_expect_tx(&bar, (uint32_t)(F * S3 * sizeof(double)));
      }
      __syncwarp();
      const double* src = A.U + (size_t)tile.s * F * Tl::kS3;
      if (NN == N) {
        if (tid == 0)
#pragma unroll 1
          for (int k = 0; k < F; ++k) bulk_g2s(Q + k * S3, src + (size_t)k * S3, S3 * sizeof(double), &bar);
      } else {
#pragma unroll 1
        for (int w = tid; w < F * S * S; w += 32) {
          const int k = w / (S * S), z = (w / S) % S, y = w % S;
          bulk_g2s(Q + k * S3 + (z * S + y) * S, src + (size_t)k * Tl::kS3 + tile.pad(0, y, z), S * sizeof(double),
                   &bar);
        }
      }
    }
  };

  if (tid == 0) {
    mbar_init(&bar, 1);
    fence_mbar_init();
    bail = 0;
  }
  __syncthreads();
  if (T == 1 && team < n_units) stage(team);

  uint32_t phase = 0;
  for (int u = team; u < n_units; u += n_teams) {
    const Tl tile(u);
    const int s = tile.s;

    // ---- 1. primitives ------------------------------------------------------
    bool bad = false;
    WildTile seen;
    if (T == 1) {
      if (!mbar_wait_bounded(&bar, phase, kLWaitPolls)) {
        atomicOr(A.status, 2u);
        bail = 1;
      }
      phase ^= 1u;
      __syncthreads();
      if (bail) break;
      for (int c = tid; c < S3; c += kLThreads) {
        double w[EGAS + 1];
#pragma unroll
        for (int k = 0; k <= EGAS; ++k) w[k] = Q[k * S3 + c];
        bad |= !prims64(w, Q[TAU * S3 + c], A.P);
#pragma unroll
        for (int k = SX; k <= EGAS; ++k) Q[k * S3 + c] = w[k];
#pragma unroll
        for (int k = 0; k < F; ++k) seen.see(k <= EGAS ? w[k] : Q[k * S3 + c]);
      }
    } else {
      // the team converts each cell once; Pb was last read before the
      // previous tile's lines, which every CTA of the team has passed
      const double* src = A.U + (size_t)s * F * Tl::kS3;
      for (int c = rank * kLThreads + tid; c < S3; c += T * kLThreads) {
        const int pc = tile.pad(c);
        double w[F];
#pragma unroll
        for (int k = 0; k < F; ++k) w[k] = __ldg(src + (size_t)k * Tl::kS3 + pc);
        bad |= !prims64(w, w[TAU], A.P);
#pragma unroll
        for (int k = 0; k < F; ++k) Pb[k * S3 + c] = w[k];
      }
      if (!team_barrier(B, &sh_ok)) break;
      const double2* pb2 = reinterpret_cast<const double2*>(Pb);
      double2* q2 = reinterpret_cast<double2*>(Q);
#pragma unroll 6
      for (int c = tid; c < F * S3 / 2; c += kLThreads) {
        const double2 v = __ldcg(pb2 + c);
        seen.see(v.x);
        seen.see(v.y);
        q2[c] = v;
      }
    }
    if (bad) atomicOr(A.status, 1u);
    const bool wild = __syncthreads_or(seen.wild());

    // ---- 2. learned smoothness indicator -----------------------------------
    if (kGate)
      gate_phase<double, kLThreads>(Q, (float)A.P.gm1, A.gate_w, A.gate_logit_thr, A.gate_zero_smooth, smooth,
                                    smooth + S3);

    // ---- 3. every line once: (field group, run) items, group-major ----------
    {
      const double k3h = 3.0 / A.h[s];  // the spin feedback's 3 / h
      const int n_items = 2 * n_runs;
#pragma unroll 1
      for (int it = (rank + T * warp) * 32 + lane; it < n_items; it += T * kLThreads) {
        if (wild) {
          if (it < n_runs) line_run_wild(Q, kGate ? smooth : nullptr, kContact, A.P, R, g_line_runs[it], k3h);
        } else if (it < n_runs)
          line_run<kGate, kContact, 6>(Q, smooth, A.P, R, g_line_runs[it], 0, k3h);
        else
          line_run<kGate, kContact, 4>(Q, smooth, A.P, R, g_line_runs[it - n_runs], 6, k3h);
      }
    }
    // the last reads of Q for this tile are done: order them before the bulk
    // copies of the next tile, which overlap phases 4 and 5
    fence_proxy_async();
    if (!team_barrier(B, &sh_ok)) break;  // the line ends are visible to the whole team
    if (T == 1 && u + n_teams < n_units) stage(u + n_teams);

    // ---- 4. faces from the stored line ends ----------------------------------
    const int ox = tile.o[0], oy = tile.o[1];
    const double h = A.h[s];
    const double half_h = 0.5 * h;
    const double o[3] = {A.origin[3 * s + 0], A.origin[3 * s + 1], A.origin[3 * s + 2]};
    double amax = 0.0;
    const bool one_point = A.P.face_points == 1;
#pragma unroll 1
    for (int f = (rank + T * warp) * 32 + lane; f < kFaces; f += T * kLThreads) {
      // face j - 1/2 of row (pb, pc) along a, between the cells j - 1 (left)
      // and j (right); transverse axes b < c
      const int a = f / ((N + 1) * N * N), j = (f / (N * N)) % (N + 1), pc = (f / N) % N, pb = f % N;
      const int b = (a == 0) ? 1 : 0;
      const int ba = a == 0 ? 1 : (a == 1 ? N + 2 : (N + 2) * (N + 2));
      // box index of the right cell
      const int boxr = ((axis_comp(2, a, b, j, pb, pc) + 1) * (N + 2) + (axis_comp(1, a, b, j, pb, pc) + 1)) * (N + 2) +
                       (axis_comp(0, a, b, j, pb, pc) + 1);
      // the coordinate that the frame velocity's normal component takes (y_q
      // for x-faces, x_q for y-faces), at the three offsets along b
      const double cb = (pb + (a == 0 ? oy : ox)) + 0.5, ob = a == 0 ? o[1] : o[0];
      const double rm = fma(h, cb - 0.5, ob), r0 = fma(h, cb, ob), rp = fma(h, cb + 0.5, ob);
      const double om = frame_om(a, A.P);
      double fsum[F], Mt[4];
#pragma unroll
      for (int k = 0; k < F; ++k) fsum[k] = 0.0;
      Mt[0] = Mt[1] = Mt[2] = Mt[3] = 0.0;
      // the points in the summation order of hydro_step_fp64_kernel: q = 2p +
      // side for the mirrored pairs p = 0..3 (side 0: the point (-t1,-t2),
      // side 1: (t1,t2), with (t1,t2) = (p/3 - 1, p%3 - 1)), then the centre
      // q = 8; the single-point face flux takes the centre alone
#pragma unroll 1
      for (int qq = one_point ? 8 : 0; qq <= 8; ++qq) {
        const int pp = qq >> 1, t1 = pp / 3 - 1, t2 = pp % 3 - 1;
        const int u1 = (qq & 1) ? t1 : -t1, u2 = (qq & 1) ? t2 : -t2;
        const int d0 = axis_comp(0, a, b, 1, u1, u2), d1 = axis_comp(1, a, b, 1, u1, u2),
                  d2 = axis_comp(2, a, b, 1, u1, u2);
        // the value at x + w/2 of cell j - 1, w = e_a + u1 e_b + u2 e_c (left),
        // and at x + w'/2 of cell j, w' = w - 2 e_a (right)
        const int sl = end_slot(d0, d1, d2);
        const int sr = end_slot(a == 0 ? -1 : d0, a == 1 ? -1 : d1, a == 2 ? -1 : d2);
        const double* pl = R + ((size_t)sl * kBox + boxr - ba) * kRec;
        const double* pr = R + ((size_t)sr * kBox + boxr) * kRec;
        double qL[F], qR[F];
        End64 eL, eR;
        ld_sector(pl, qL[RHO], qL[SX], qL[SY], qL[SZ]);
        ld_sector(pr, qR[RHO], qR[SX], qR[SY], qR[SZ]);
        ld_sector(pl + 4, eL.p, eL.E, eL.c, qL[TAU]);
        ld_sector(pr + 4, eR.p, eR.E, eR.c, qR[TAU]);
        ld_sector(pl + 8, qL[ZX], qL[ZY], qL[ZZ], qL[SP0]);
        ld_sector(pr + 8, qR[ZX], qR[ZY], qR[ZZ], qR[SP0]);
        qL[EGAS] = qR[EGAS] = 0.0;  // not read
        const double r = u1 == 0 ? r0 : (u1 > 0 ? rp : rm);
        // half the Simpson weight (1, 4, 1) x (1, 4, 1) / 36 of the point; 1/2
        // for the single-point face flux
        const double hw = one_point                ? 0.5
                          : (u1 == 0 && u2 == 0) ? (8.0 / 36.0)
                          : (u1 == 0 || u2 == 0) ? (2.0 / 36.0)
                                                 : (0.5 / 36.0);
        point64(qL, eL, qR, eR, a, om, r, hw, u1, u2, fsum, Mt, amax);
      }
      double tl[3], tr[3];
      face_torques64(Mt, fsum, a, half_h, tl, tr);
#pragma unroll
      for (int k = 0; k < F; ++k) Fs[k * kFaces + f] = fsum[k];
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        Fs[(F + m) * kFaces + f] = tl[m];
        Fs[(F + 3 + m) * kFaces + f] = tr[m];
      }
      if (A.face_flux && (j == 0 || j == N) && tile.outer(2 * a + (j == N ? 1 : 0))) {
        // sub-grid boundary face: sums and the torque about the interior cell
        const int fo = 2 * a + (j == N ? 1 : 0);
#pragma unroll
        for (int k = 0; k < F; ++k) A.face_flux[tile.face(fo, k, pc, pb)] = fsum[k];
#pragma unroll
        for (int m = 0; m < 3; ++m) A.face_flux[tile.face(fo, F + m, pc, pb)] = (j == N) ? tl[m] : tr[m];
      }
    }
    amax = warp_max(amax);
    if (lane == 0) red[warp] = amax;
    if (!team_barrier(B, &sh_ok)) break;  // the face sums are visible, line-end reads finished

    // ---- 5. divergence + sources, one thread per interior cell -----------
    const double inv_h = 1.0 / h;
    const double om = A.P.omega;
    const double* Us = A.U + (size_t)s * F * Tl::kS3;
    double* dU = A.dUdt + (size_t)s * F * Tl::kN3;
    for (int c = (rank + T * warp) * 32 + lane; c < N3; c += T * kLThreads) {
      const int x = c % N, y = (c / N) % N, z = c / (N * N);
      const int uc = tile.pad(x + G, y + G, z + G);  // in the sub-grid's padded array
      const int cs = tile.cell(c);                   // in its compact NN^3 array
      // the cell's lower faces; the upper ones are N*N further
      const double* f0 = Fs + (x * N + z) * N + y;
      const double* f1 = Fs + (((N + 1) + y) * N + z) * N + x;
      const double* f2 = Fs + ((2 * (N + 1) + z) * N + y) * N + x;
      // differences of value q between the upper and the lower face (ql: its
      // slot for the lower face, whose torques are about its right cell)
      auto dif = [&](const double* fa, int q, int ql) {
        return __ldcg(fa + q * kFaces + N * N) - __ldcg(fa + ql * kFaces);
      };
      double du[F];
#pragma unroll
      for (int k = 0; k < F; ++k) {
        const double div = (dif(f0, k, k) + dif(f1, k, k)) + dif(f2, k, k);
        du[k] = -(div * inv_h);
      }
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        const double tq = (dif(f0, F + m, F + 3 + m) + dif(f1, F + m, F + 3 + m)) + dif(f2, F + m, F + 3 + m);
        du[ZX + m] = du[ZX + m] - tq * inv_h;
      }
      const double sx = Us[SX * Tl::kS3 + uc], sy = Us[SY * Tl::kS3 + uc], sz = Us[SZ * Tl::kS3 + uc];
      du[SX] = du[SX] + om * sy;
      du[SY] = du[SY] - om * sx;
      du[ZX] = du[ZX] + om * Us[ZY * Tl::kS3 + uc];
      du[ZY] = du[ZY] - om * Us[ZX * Tl::kS3 + uc];
      {
        // spin source w(x_c) x s, w = -omega z_hat x x_c: removes the torque
        // that the frame part s w_n of the momentum flux leaves in the face
        // torques, so that sum (x_c x s + z)_z is conserved for omega != 0
        const double xc = __dadd_rn(o[0], __dmul_rn(h, (x + ox) + 0.5));
        const double yc = __dadd_rn(o[1], __dmul_rn(h, (y + oy) + 0.5));
        const double wx = om * yc, wy = -(om * xc);
        du[ZX] = du[ZX] + wy * sz;
        du[ZY] = du[ZY] - wx * sz;
        du[ZZ] = du[ZZ] + (wx * sy - wy * sx);
      }
      if (A.g) {
        const double* gs = A.g + (size_t)s * 3 * Tl::kN3 + cs;
        const double gx = gs[0], gy = gs[Tl::kN3], gz = gs[2 * Tl::kN3];
        const double rho = Us[RHO * Tl::kS3 + uc];
        du[SX] = du[SX] + rho * gx;
        du[SY] = du[SY] + rho * gy;
        du[SZ] = du[SZ] + rho * gz;
        du[EGAS] = du[EGAS] + ((sx * gx + sy * gy) + sz * gz);
      }
#pragma unroll
      for (int k = 0; k < F; ++k) dU[k * Tl::kN3 + cs] = du[k];
    }
    if (tid == 0) {
      double m = red[0];
#pragma unroll
      for (int w = 1; w < kLWarps; ++w) m = fmax(m, red[w]);
      if (Tl::kTiles == 1 && T == 1)
        A.amax[s] = m;
      else
        atomic_max_nonneg(A.amax + s, m);  // cleared before the launch
    }
    // face sums and red are rewritten after the next tile's lines, whose
    // barrier every thread of the team reaches after its reads above
  }
  __syncthreads();
  if (tid == 0) mbar_inval(&bar);
}

size_t step_fp64_lines_smem_bytes(bool gate) { return (size_t)F * S3 * sizeof(double) + (gate ? 2 * S3 : 0); }

template <int NN>
static cudaError_t fp64_lines_attrs() {
  cudaError_t e = cudaSuccess;
  const void* fns[4] = {(const void*)hydro_step_fp64_lines_kernel<false, false, NN>,
                        (const void*)hydro_step_fp64_lines_kernel<true, false, NN>,
                        (const void*)hydro_step_fp64_lines_kernel<false, true, NN>,
                        (const void*)hydro_step_fp64_lines_kernel<true, true, NN>};
  for (int i = 0; i < 4 && e == cudaSuccess; ++i)
    e = cudaFuncSetAttribute(fns[i], cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)step_fp64_lines_smem_bytes(i & 1));
  return e;
}

// Once per device: the shared-memory opt-in and the run list (no
// allocation; call before any stream capture).
cudaError_t prepare_step_fp64_lines() {
  static unsigned long long done = 0;
  return once_per_device(&done, [] {
    cudaError_t e = fp64_lines_attrs<8>();
    if (e == cudaSuccess) e = fp64_lines_attrs<16>();
    if (e != cudaSuccess) return e;
    int n_axis = 0;
    const std::vector<uint32_t> runs = build_line_runs(&n_axis);
    if (runs.size() > (size_t)kMaxRuns) return cudaErrorInvalidValue;
    e = cudaMemcpyToSymbol(g_line_runs, runs.data(), runs.size() * sizeof(uint32_t));
    if (e == cudaSuccess) {
      g_runs_total = (int)runs.size();
      g_runs_axis = n_axis;
    }
    return e;
  });
}

size_t step_fp64_lines_per_team() { return kLinesPerTeam; }
size_t step_fp64_lines_sync_words(int teams) { return 32 * (1 + (size_t)teams); }

// CTAs per team for `units` tiles on num_sms SMs: the smallest estimate of
//   rounds of the teams over the batch x (a tile's time on T SMs),
// the latter its FP64 work shared out (kTileUs on one SM), not below the
// chain of the longest line run and a face (kChainUs), plus the team's
// barriers and copies (kTeamUs).  A batch that fills whole rounds of single
// CTAs keeps T = 1; 512 tiles on 152 SMs take 3.4 rounds' work in 4 rounds
// alone, and one tile alone leaves 151 SMs idle.  The three are the model's
// weights and not times: a tile takes 647 us on one SM (with contact steepening
// 960, and spin feedback 1,110), and the least that a team takes for one is 81
// (118), so the estimates lie 15 to 70 % below the times, and no team has
// more than 46 CTAs, where the shared work meets the chain.
// Measured on 152 SMs, teams against single CTAs: 1 tile 81 against 647 us,
// 8 tiles 84 and 647, 16 tiles 110 and 648, 38 tiles 204 and 650, 77 tiles 471
// and 659, 512 tiles 2,454 and 2,618.
int step_fp64_choose_team(int units, int num_sms, int face_points) {
  const double kTileUs = face_points == 1 ? 120.0 : 560.0, kChainUs = 12.0, kTeamUs = 12.0;
  int best = 1;
  double best_us = 1e300;
  for (int T = 1; T <= num_sms; ++T) {
    const int teams = num_sms / T;
    const int rounds = (units + teams - 1) / teams;
    double us = kTileUs / T;
    if (T > 1) us = (us > kChainUs ? us : kChainUs) + kTeamUs;
    // a larger team has to gain 2 %
    if (rounds * us < 0.98 * best_us) {
      best_us = rounds * us;
      best = T;
    }
  }
  return best;
}

template <int NN>
static cudaError_t launch_fp64_lines_nn(const StepArgs64& A, int grid, int n_runs, int T, unsigned* sync,
                                        long long wait_ns, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(kLThreads);
  cfg.dynamicSmemBytes = step_fp64_lines_smem_bytes(A.gate);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = T > 1 ? 1 : 0;
  if (A.gate && A.P.contact)
    return cudaLaunchKernelEx(&cfg, hydro_step_fp64_lines_kernel<true, true, NN>, A, n_runs, T, sync, wait_ns);
  if (A.gate)
    return cudaLaunchKernelEx(&cfg, hydro_step_fp64_lines_kernel<true, false, NN>, A, n_runs, T, sync, wait_ns);
  if (A.P.contact)
    return cudaLaunchKernelEx(&cfg, hydro_step_fp64_lines_kernel<false, true, NN>, A, n_runs, T, sync, wait_ns);
  return cudaLaunchKernelEx(&cfg, hydro_step_fp64_lines_kernel<false, false, NN>, A, n_runs, T, sync, wait_ns);
}

// The FP64 step with every line once, over the A.n_sub * (nn/8)^3 tiles:
// `teams` teams of T CTAs (T > 1: teams * T at most the SMs, a cooperative
// launch, and sync holds step_fp64_lines_sync_words(teams) words); A.lines
// holds teams * step_fp64_lines_per_team() doubles.  Where several CTAs share
// a sub-grid its amax is the atomic maximum over them, cleared here first.
cudaError_t launch_step_fp64_lines(const StepArgs64& A, int teams, int T, unsigned* sync, int nn, cudaStream_t st) {
  cudaError_t e = prepare_step_fp64_lines();
  if (e != cudaSuccess) return e;
  if (!A.lines || T < 1 || (T > 1 && !sync)) return cudaErrorInvalidValue;
  const int n_runs = A.P.face_points == 1 ? g_runs_axis : g_runs_total;
  if (T > 1) {
    e = cudaMemsetAsync(sync, 0, step_fp64_lines_sync_words(teams) * sizeof(unsigned), st);
    if (e != cudaSuccess) return e;
  }
  if (nn == 16 || T > 1) {
    e = cudaMemsetAsync(A.amax, 0, (size_t)A.n_sub * sizeof(double), st);
    if (e != cudaSuccess) return e;
  }
  // a second: far above the longest phase of a tile on one SM
  const long long wait_ns = 1000000000ll;
  return nn == 16 ? launch_fp64_lines_nn<16>(A, teams * T, n_runs, T, sync, wait_ns, st)
                  : launch_fp64_lines_nn<8>(A, teams * T, n_runs, T, sync, wait_ns, st);
}

}  // namespace hyd

namespace hyd {

__global__ void selftest_arith_kernel(const double* __restrict__ x, const double* __restrict__ y, int n,
                                      double* __restrict__ out) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const double a = x[i], b = y[i];
    out[2 * i] = half64(a);
    out[2 * i + 1] = slope64(a, b);
  }
}

__global__ void selftest_scalar_kernel(const double* __restrict__ x, const double* __restrict__ y, double eta, int n,
                                       double* __restrict__ out) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const double a = x[i], b = y[i];
    double u[EGAS + 1] = {b, a, 0.0, 0.0, 1.0};
    const StepParams P = {};
    prims64(u, 1.0, P);
    out[5 * i + 0] = u[SX];
    out[5 * i + 1] = rsqrt64(b);
    out[5 * i + 2] = (double)narrow(a);
    out[5 * i + 3] = widen((float)a);
    out[5 * i + 4] = above(a, narrow(a), eta, b, narrow(b)) ? 1.0 : 0.0;
  }
}

}  // namespace hyd

extern "C" int hydro_selftest_arith(const double* x, const double* y, int n, double* out, void* stream) {
  if (n < 0 || (n > 0 && (!x || !y || !out))) return HYDRO_EINVAL;
  if (n == 0) return HYDRO_OK;
  const int grid = (n + 255) / 256 < 1024 ? (n + 255) / 256 : 1024;
  hyd::selftest_arith_kernel<<<grid, 256, 0, (cudaStream_t)stream>>>(x, y, n, out);
  return cudaGetLastError() == cudaSuccess ? HYDRO_OK : HYDRO_ECUDA;
}

extern "C" int hydro_selftest_scalar(const double* x, const double* y, double eta, int n, double* out, void* stream) {
  if (n < 0 || (n > 0 && (!x || !y || !out))) return HYDRO_EINVAL;
  if (n == 0) return HYDRO_OK;
  const int grid = (n + 255) / 256 < 1024 ? (n + 255) / 256 : 1024;
  hyd::selftest_scalar_kernel<<<grid, 256, 0, (cudaStream_t)stream>>>(x, y, eta, n, out);
  return cudaGetLastError() == cudaSuccess ? HYDRO_OK : HYDRO_ECUDA;
}

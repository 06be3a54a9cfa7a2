// The two-step march: one launch advances an FP32 grid by two time steps, so the state crosses
// HBM once for two steps. Described for a gradient stencil that reaches one node; one that
// reaches two (TWO_FAR) skews the second step's rows and columns by one more, groups 3, 4 and
// 6, 7 change slots, and two groups carry what group 6 does here.
//
// A CTA of 8 row groups walks up a segment of a strip, 8 rows per pass, as march_kernel does,
// but pulls step n + 1 into registers, collides it again and pulls step n + 2, which is what it
// stores. Thread column c of a strip is grid column X0 - 3 + c: step n is collided on all
// columns, pulled on 1 .. COLS - 2, step n + 1 collided on 2 .. COLS - 3 and pulled on the
// COLS - 6 columns the strip owns. Rows are skewed alike. With s = r_begin + 8 k, pass k
//   A  collides step n of rows      s + 3 .. s + 10  (group w row s + 3 + w),
//   A' pulls step n + 1 of rows     s + 2 .. s + 9   (7: the row it collided a pass before),
//   B  collides step n + 1 of rows  s + 1 .. s + 8   (6: the row it pulled a pass before),
//   B' pulls step n + 2 of rows     s .. s + 7       (5: the row it collided in B a pass before),
// each group one row per phase; what a group carries into the next pass (7: the pre-collision h
// and phi, 6: the pulled populations, 5: the pre-collision h) waits in its own shared stash. The
// prologue pass k = -1 runs the part of this that reaches the segment's first rows. A segment is
// a multiple of 8 rows and ends at a multiple of 8 below the top of the grid (the first one may
// begin below row 0 and skips those rows), so no phase overruns the segment's end, and the last
// row of the grid is never a group's row 7.
//
// Collided rows: 12 row slots serve both steps. A needs the 8 rows it wrote and the last 2 of
// the pass before, B likewise; a phase overwrites the rows of the other step except those 2.
// Groups 0..3 write slots 0..3; groups 4, 5 and 6, 7 alternate between two pairs of slots each
// from pass to pass, which leaves B's last two rows (groups 4, 5) and A's last two (6, 7) where
// they are (slot_a, slot_b).
//
// Ghost nodes of a non-periodic face are not collided: the thread that collides the adjacent
// interior node writes their collided values too (the same node, directions mirrored behind a
// free-slip wall, or the inlet state), and its phi^{n+1} into the ghost places of the phi^{n+1}
// ring. Ghost nodes of a periodic face are the wrapped nodes, collided like any other. Every
// value is formed by the expressions of the one-step kernels: the bits are theirs.
//
// What bounds it: at 2048^2 with flow the one-step march took 152 us per step, 0.92 of the copy
// bandwidth, so only a form that moves less can be faster. This one moves 232 B of DRAM per node
// and two steps (73 us per step at the copy bandwidth) and takes 116: issue at 60% and the
// shared-memory pipe at 65%, with 19.6 warp instructions per node and step (26 of 32 columns
// useful).
// What mattered, in us per step there: collision of g and f ahead of the barrier that the slots
// need, so that both halves of a phase mix arithmetic with shared accesses, 162 -> 150; the next
// pass's node into L1 a pass ahead -> 133; 3 CTAs per SM at 80 registers instead of 4 at 64
// (216 KB of shared memory left the loads little L1, and spills) -> 121; the barrier between B' and
// the next pass's emission split into an arrival and a wait around its g and f, 123.7 -> 115.8
// (1200^2 49.0 -> 45.6, without flow 4096^2 306 -> 298, a batch of 24 294 -> 286). Not kept: the
// same for the barrier ahead of B's emission (117), and waits for the neighbour rows' groups alone
// in place of the other two (125); the next pass's populations into registers ahead of B' (125);
// 64 columns and 16 warps (140; fewer redundant columns, longer barriers), 16- and 12-row passes
// (130, 132), prefetch into L2 only (129), streaming stores (neutral), the edge march as a call (126).
#pragma once

#include "lbmice_step.cuh"

namespace lbmice {

constexpr int kTwoCols = 32;               // thread columns of a strip
constexpr int kTwoRows = 8;                // rows per pass (groups of a CTA)
constexpr int kTwoSlots = kTwoRows + 4;    // collided row slots
// CTAs per SM of the two-step march (its launch bound): 3 with flow, at 80 registers, 4 without, at
// 64 (1024^2 without flow: 26.4 us per step with 4, 40 B of spills included, 27.0 with 3).
__host__ __device__ constexpr int two_ctas(bool flow) { return flow ? 3 : 4; }

// What a launch computes: the default scheme (E4, six-fold), any stencil that reaches one node
// and either fold (E2, E4), or any stencil (reach 2; periodic grids only).
enum : int { TWO_DEFAULT = 0, TWO_NEAR = 1, TWO_FAR = 2 };
__host__ __device__ constexpr int two_reach(int v) { return v == TWO_FAR ? 2 : 1; }
// Rim of a strip or tile, collided but not stored: a pull and the stencil's reach per step, the
// first step's collisions beside them.
__host__ __device__ constexpr int two_rim(int v) { return 2 + two_reach(v); }
__host__ __device__ constexpr int two_out(int v = TWO_DEFAULT) { return kTwoCols - 2 * two_rim(v); }
__host__ __device__ constexpr int two_strips(int nx, int v = TWO_DEFAULT) {
  return (nx + two_out(v) - 1) / two_out(v);
}
// Rows below row 0 that the first segment skips: segments end at ny - 8 j.
__host__ __device__ constexpr int two_pad(int ny) { return (kTwoRows - ny % kTwoRows) % kTwoRows; }

template <bool FLOW, int VAR = TWO_DEFAULT>
struct TwoSmem {
  static constexpr int COLS = kTwoCols;
  static constexpr int SN = kTwoSlots * COLS;          // slots x columns
  static constexpr int PW = COLS + 8;                  // phi^n ring row: columns xa .. xa + PW - 1
  static constexpr int PN = 2 * kTwoRows * PW;         // phi^n ring: two blocks of a pass
  static constexpr int QN = 2 * kTwoRows * COLS;       // phi^{n+1} ring
  static constexpr int NP = FLOW ? 27 : 18;            // populations of a node
  static constexpr int E = two_reach(VAR);
  static constexpr int STASH = (10 + E * (NP + 1) + 9) * COLS;
  static constexpr size_t bytes() {
    return sizeof(float) * (PostTile::floats<FLOW>(SN) + PN + QN + STASH) + 32;
  }
  static_assert(PW == kMarchPW && kTwoRows == kMarchRows, "the phi ring blocks share the march's tensor maps");
  static_assert(PostTile::floats<FLOW>(SN) % 32 == 0 && (kTwoRows * PW * 4) % 128 == 0,
                "phi ring blocks of the two-step march not at 128-byte boundaries");
};

// Slot of the row with index i of a phase (i = 0 .. 7 the rows written in this pass, -2 and -1 the
// last two of the pass before), for an even (e = 0) or odd pass; E the stencil's reach. A's rows
// are numbered by group; B's begin with those of the E groups that pulled theirs a pass before.
__host__ __device__ constexpr int two_group_slot(int e, int w, bool b, int E) {
  constexpr int R = kTwoRows;
  const int kb = R - 3 - E;  // groups kb, kb + 1 write B's last two rows, R - 2 and R - 1 A's
  if (w >= R - 2) return (b ? !e : e) ? w + 2 : w;
  if (w == kb || w == kb + 1) return e ? R + 2 + w - kb : w;
  return w;
}
__host__ __device__ constexpr int slot_a(int e, int i, int E) {
  return i < 0 ? two_group_slot(1 - e, kTwoRows + i, false, E) : two_group_slot(e, i, false, E);
}
__host__ __device__ constexpr int slot_b(int e, int i, int E) {
  constexpr int R = kTwoRows;
  return i < 0 ? two_group_slot(1 - e, R - 1 - E + i, true, E)
               : two_group_slot(e, i < E ? R - 1 - E + i : i == E ? R - 1 : i - 1 - E, true, E);
}
// Phase row index of group w: A collides w and pulls w (the last group: -1); B collides
// two_bc(w) and pulls two_bp(w).
__host__ __device__ constexpr int two_ap(int w) { return w < kTwoRows - 1 ? w : -1; }
__host__ __device__ constexpr int two_bc(int w, int E) {
  constexpr int R = kTwoRows;
  return w == R - 1 ? E : w >= R - 1 - E ? w - (R - 1 - E) : w + 1 + E;
}
__host__ __device__ constexpr int two_bp(int w, int E) {
  return w == kTwoRows - 2 - E ? -1 : two_bc(w, E);
}

// A group's slots in one phase: the one it writes, and those of the rows below, at and above the
// row it pulls.
struct TwoSlots {
  int own, dn, at, up;
};
struct TwoTable {
  TwoSlots a[2][kTwoRows], b[2][kTwoRows];
};
constexpr TwoTable two_table(int E) {
  TwoTable t{};
  for (int e = 0; e < 2; ++e)
    for (int w = 0; w < kTwoRows; ++w) {
      const int p = two_ap(w), q = two_bp(w, E);
      t.a[e][w] = {slot_a(e, w, E), slot_a(e, p - 1, E), slot_a(e, p, E), slot_a(e, p + 1, E)};
      t.b[e][w] = {slot_b(e, two_bc(w, E), E), slot_b(e, q - 1, E), slot_b(e, q, E),
                   slot_b(e, q + 1, E)};
    }
  return t;
}
// (one symbol each: an array of the two cost the march 2%)
__constant__ TwoTable kTwoNear = two_table(1);
__constant__ TwoTable kTwoFar = two_table(2);

// Exchange a value with the thread's place in a stash: the value kept by the pass before comes
// back, this pass's stays.
__device__ __forceinline__ void swap_stash(float* place, float& v) {
  const float t = *place;
  *place = v;
  v = t;
}

// Collided values of a node into its slot, and (EDGE) those of the ghost nodes beside it at
// non-periodic faces: h is collided here (hg[a].x, which stays), g and f come collided. sx, sy:
// -1 / +1 when the node lies at a non-periodic low / high face of that axis, else 0; slots[1 + j]
// is the slot of the row j = -1, 0, +1 from the node's.
template <bool FLOW, bool EDGE>
__device__ __forceinline__ void two_emit(const Consts& C, const Coefs& K, const float2* hg,
                                         const float* fv, float rho, int sx, int sy,
                                         const int (&slots)[3], int col, const PostTile& T) {
  constexpr int COLS = kTwoCols;
  const int SN = T.SN;
  {
    const int node = slots[1] * COLS + col;
    if (!in_range(node, SN, OOB_SHARED)) return;
#pragma unroll
    for (int a = 0; a < 9; ++a) {
      T.hg[a * SN + node] = pair(collided_h(K, a, hg[a].x), hg[a].y);
      if (FLOW) T.f[a * SN + node] = fv[a];
    }
    T.B[node] = K.B;
  }
  if (!EDGE || (sx | sy) == 0) return;
  // the ghosts across x, y and the corner
#pragma unroll 1
  for (int g = 1; g < 4; ++g) {
    if (((g & 1) && !sx) || ((g & 2) && !sy)) continue;
    const int gx = (g & 1) ? sx : 0, gy = (g & 2) ? sy : 0;
    const int c = col + gx;
    if (c < 0 || c >= COLS) continue;  // beyond the strip: no pull reads it
    const int slot = gy < 0 ? slots[0] : gy > 0 ? slots[2] : slots[1];
    if (slot < 0) continue;  // beyond the rows in reach: no pull reads it
    const int node = slot * COLS + c;
    if (!in_range(node, SN, OOB_SHARED)) continue;
    const int fx = gx ? (gx < 0 ? 0 : 1) : -1, fy = gy ? (gy < 0 ? 2 : 3) : -1;
    const int kx = fx < 0 ? -1 : (fx ? C.bc[1] : C.bc[0]);
    const int ky = fy < 0 ? -1 : (fy == 3 ? C.bc[3] : C.bc[2]);
    if (kx == BC_INLET || ky == BC_INLET) {
      const int face = kx == BC_INLET ? fx : fy;
      const float ux = face == 0 ? C.uin_x[0] : face == 1 ? C.uin_x[1]
                     : face == 2 ? C.uin_x[2] : C.uin_x[3];
      const float uy = face == 0 ? C.uin_y[0] : face == 1 ? C.uin_y[1]
                     : face == 2 ? C.uin_y[2] : C.uin_y[3];
      inlet_state<FLOW>(C, ux, uy, rho, node, T);
      continue;
    }
    const bool mirx = kx == BC_FREESLIP, miry = ky == BC_FREESLIP;
#pragma unroll
    for (int a = 0; a < 9; ++a) {
      int am = mirx ? mirx_of(a) : a;
      am = miry ? miry_of(am) : am;
      T.hg[am * SN + node] = pair(collided_h(K, a, hg[a].x), hg[a].y);
      if (FLOW) T.f[am * SN + node] = fv[a];
    }
    T.B[node] = K.B;
  }
}

// The nine pull sources of one node, Eq. (d) for h, in place (hg[a].x comes in as the node's own
// h): row bases dn, at, up (slot x COLS + column) of the rows y - 1, y, y + 1.
template <bool FLOW>
__device__ __forceinline__ void two_pull(const PostTile& T, int dn, int at, int up, float2* hg,
                                         float* fn) {
#pragma unroll
  for (int a = 0; a < 9; ++a) {
    const int cy = cy_of(a);
    const int s = (cy > 0 ? dn : (cy < 0 ? up : at)) - cx_of(a);
    float2 v = T.hg[a * T.SN + s];
    v.x = fmaf(hg[a].x, T.B[s], v.x);
    hg[a] = v;
    if (FLOW) fn[a] = T.f[a * T.SN + s];
  }
}

// E4 gradient of phi through a view, with the expressions of collide_source.
template <class View>
__device__ __forceinline__ void gradient_e4(const View& V, float& gx, float& gy) {
  const float pE = V(1, 0), pW = V(-1, 0), pN = V(0, 1), pS = V(0, -1);
  const float pNE = V(1, 1), pNW = V(-1, 1), pSE = V(1, -1), pSW = V(-1, -1);
  gx = fmaf(kW1, pE - pW, __fmul_rn(kW2, (pNE - pNW) + (pSE - pSW)));
  gy = fmaf(kW1, pN - pS, __fmul_rn(kW2, (pNE - pSE) + (pNW - pSW)));
}

// The vapour and flow collision of a node whose populations (DEV: deviations) are in registers, in
// place. U and rho: the node's moments, computed here for FP32 populations.
template <bool FLOW, bool DEV>
__device__ __forceinline__ void two_collide_gf(const Consts& C, float2* hg, float* fv, float ph,
                                               float php, float& U, float& rho) {
  if (!DEV) {
    U = hg[0].y + (((hg[1].y + hg[3].y) + (hg[2].y + hg[4].y)) +
                   ((hg[5].y + hg[7].y) + (hg[6].y + hg[8].y)));
    rho = FLOW ? sum9(fv) : 1.0f;
  }
  float jx = 0.0f, jy = 0.0f;
  if (FLOW) {
    jx = sumcx9(fv);
    jy = sumcy9(fv);
  }
  Coefs K;
  coefs_gf<FLOW, DEV>(C, ph, php, U, rho, jx, jy, K);
#pragma unroll
  for (int a = 0; a < 9; ++a) {
    hg[a].y = collided_g(K, a, hg[a].y);
    if (FLOW) fv[a] = collided_f(K, a, fv[a]);
  }
}

// The phase-field collision, phi around the node in a ring view, and the output to the slots.
template <bool FLOW, bool EDGE, int VAR, bool DEV, class View>
__device__ __forceinline__ void two_collide_h(const Consts& C, const float2* hg, const float* fv,
                                              float ph, float U, float rho, const View& V, int sx,
                                              int sy, const int (&slots)[3], int col,
                                              const PostTile& T) {
  float gx, gy;
  Coefs K;
  if constexpr (VAR == TWO_DEFAULT) {
    gradient_e4(V, gx, gy);
    coefs_h<DEV, 1>(C, ph, U, gx, gy, K);
  } else {
    gradient_stencil<float>(C.stencil, V, gx, gy);
    coefs_h<DEV, 2>(C, ph, U, gx, gy, K);
  }
  two_emit<FLOW, EDGE>(C, K, hg, fv, rho, sx, sy, slots, col, T);
}

// phi around a node at column c of a ring of 2 kTwoRows rows of PW, row q.
template <int PW, int E>
struct RowRing {
  const float* s;
  int q, c;
  __device__ __forceinline__ int at(int dy) const {
    return ((q + dy) & (2 * kTwoRows - 1)) * PW + c;
  }
  __device__ __forceinline__ float operator()(int dx, int dy) const { return s[at(dy) + dx]; }
  __device__ __forceinline__ bool ok() const {
    bool k = true;
#pragma unroll
    for (int dy = -E; dy <= E; ++dy)
      k = k && in_range(at(dy) - E, 2 * kTwoRows * PW, OOB_SHARED) &&
          in_range(at(dy) + E, 2 * kTwoRows * PW, OOB_SHARED);
    return k;
  }
};

// Two steps of rows [max(r_begin, 0), r_end) of the strip whose first owned column is X0; r_end -
// r_begin is a multiple of 8.
template <bool FLOW, bool EDGE, int VAR>
__device__ __forceinline__ void two_range(const Consts& C, const StepPtrs& P, int X0, int r_begin,
                                          int r_end, float* smem) {
  using M = TwoSmem<FLOW, VAR>;
  constexpr int COLS = M::COLS, R = kTwoRows, E = M::E, RIM = two_rim(VAR);
  const PostTile post = PostTile::at<FLOW>(smem, M::SN);
  float* sphi = smem + PostTile::floats<FLOW>(M::SN);
  float* sphi1 = sphi + M::PN;
  float* stash_a = sphi1 + M::QN;                  // group 7: its h, phi
  float* stash_p = stash_a + 10 * COLS;            // group 6: populations, phi
  float* stash_b = stash_p + E * (M::NP + 1) * COLS;   // group 5: its h
  uint64_t* bar = reinterpret_cast<uint64_t*>(stash_b + 9 * COLS);
  const int col = threadIdx.x % COLS;
  const int w = threadIdx.x / COLS;
  const int X = X0 - RIM + col;
  const int xa = (X0 - RIM - E) & ~3;  // grid column of phi ring column 0 (16-byte aligned)
  const int po = X0 - RIM - E - xa;
  const long long np = (long long)C.pitch * C.ny;
  // A CTA away from the faces runs every phase on all its columns, also those of the strip's rim
  // whose values nothing reads: 192 -> 179 million warp instructions per launch at 2048^2. Their
  // populations lie inside the grid (two_cta). Their shared reads stay in the CTA's block: a pull
  // reaches one element beyond the slots, which for directions with c_x != 0 is another plane of the
  // same array, and for B the end of f (or hg) or the start of the phi ring; a stencil reaches E
  // elements beyond the phi^{n+1} ring, into the phi ring or the stash. The checked build, which
  // tests every index against its own array, skips them.
  static_assert(M::PW >= COLS + 2 * E + 3 && M::PN >= E && M::STASH >= E,
                "rim reads of the two-step march leave the shared block");
#ifdef LBMICE_CHECKED
  constexpr bool ALL = false;
#else
  constexpr bool ALL = !EDGE;
#endif
  const bool tphi = !EDGE && P.tm != nullptr;
  uint64_t* slots_free = bar + 2;  // a pass's B' has read its slots: one arrival per group
  if (threadIdx.x == 0) {
    mbar_init(bar);
    mbar_init(bar + 1);
    mbar_init(slots_free, R);
  }
  __syncthreads();
  // columns a thread collides / pulls step n, collides / pulls step n + 1 on
  const bool xper = !EDGE || C.bc[0] == BC_PERIODIC, yper = !EDGE || C.bc[2] == BC_PERIODIC;
  const auto in_x = [&](int halo) {
    return !EDGE || (xper ? X <= C.nx - 1 + halo : (X >= 0 && X < C.nx));
  };
  const auto in_y = [&](int r, int halo) {
    return !EDGE || (yper ? (r >= -halo && r <= C.ny - 1 + halo) : (r >= 0 && r < C.ny));
  };
  const bool ac = in_x(RIM), ap = in_x(RIM - 1) && col >= 1 && col < COLS - 1;
  const bool bc = in_x(1) && col >= RIM - 1 && col <= COLS - RIM;
  const bool bp = col >= RIM && col < COLS - RIM && (!EDGE || X < C.nx);
  const int mx = !EDGE ? X : (X < 0 ? X + C.nx : (X >= C.nx ? X - C.nx : X));
  const int sx = EDGE && !xper ? (X == 0 ? -1 : (X == C.nx - 1 ? 1 : 0)) : 0;
  const auto side_y = [&](int r) { return EDGE && !yper ? (r == 0 ? -1 : (r == C.ny - 1 ? 1 : 0)) : 0; };

  // phi^n block kk (rows r_begin + R kk + 2 + 2 E .. + R + 1 + 2 E) into ring half (kk + 1) & 1; grid
  // row r is ring row (r - r_begin + R - 2 - 2 E) mod 2 R
  const auto phi_block = [&](int kk) {
    float* half = sphi + ((kk + 1) & 1) * kTwoRows * M::PW;
    const int y0 = r_begin + kTwoRows * kk + 2 + 2 * E;
    if (tphi) {
      if (threadIdx.x == 0) {
        uint64_t* b = bar + ((kk + 1) & 1);
        mbar_expect(b, kTwoRows * M::PW * sizeof(float));
        tma_load_2d(half, P.tm + 5, xa, y0, b);
      }
      return;
    }
    const int rl = y0 + w;
    if (EDGE && (rl < -RIM - E || rl > C.ny - 1 + RIM + E)) return;
    float* row = half + w * M::PW + po;
    for (int c = col; c < COLS + 2 * E; c += COLS) {
      if (!in_range(row - sphi + c, M::PN, OOB_SHARED)) continue;
      const int xg = X0 - RIM - E + c;
      if (!EDGE || (xg >= 0 && xg < C.nx && rl >= 0 && rl < C.ny)) {
        cp_async_plane(row + c, P.phi_n, rl * C.pitch + xg, np);
      } else {
        int gx, gy;
        float v = -1.0f;
        if (xg > C.nx - 1 + RIM + E) {
          v = 0.0f;  // beyond the grid's halo (ragged last strip): never read
        } else if (axis_phi(xg, C.nx, C.bc[0], C.bc[1], gx) &&
                   axis_phi(rl, C.ny, C.bc[2], C.bc[3], gy)) {
          v = ldg_plane(P.phi_n, gy * C.pitch + gx, np);
        }
        row[c] = v;
      }
    }
  };

  float2 hg[9];
  float fv[9];
  // this thread's node of row r, wrapped across a periodic face
  const auto wrap_row = [&](int r) { return !EDGE ? r : (r < 0 ? r + C.ny : (r >= C.ny ? r - C.ny : r)); };
  const auto prefetch_row = [&](int r) {
    if (!ac || !in_y(r, RIM)) return;
    const int my = wrap_row(r);
    prefetch_node<FLOW>(P, my * (int)C.rstride + mx, my * C.pitch + mx);
  };
  // both halves of the ring are free: the first two blocks load at once (with a reach of two the
  // prologue's collisions need the block before its own, too), and the nodes of pass 0 come into L1
  // while the prologue runs
  constexpr int LEAD = E == 2 ? 2 : 1;  // the first block's number is -LEAD
  phi_block(-LEAD);
  phi_block(1 - LEAD);
  prefetch_row(r_begin + RIM + w);
  for (int k = -1;; ++k) {
    const int s = r_begin + kTwoRows * k, e = k & 1;
    const int rA = s + RIM + w;
    if (tphi) {
      if (LEAD == 2 && k < 0) mbar_wait(bar + 1, 0);
      mbar_wait(bar + ((k + 1) & 1), ((k + LEAD) >> 1) & 1);
    } else {
      cp_async_wait_all();
      __syncthreads();  // the other threads' rows of the block
    }

    // ---- A: collide step n of row rA; g and f before the barrier, h (which needs no more than
    //      the phi ring, either) and the output after it, when B' of the pass before has read
    //      the slots. A split barrier: a group arrives as it ends B' and waits here, with its g
    //      and f collided, for the other groups' B' but not for their g and f ----
    float ph = 0.0f, U = 0.0f, rho = 1.0f;
    const TwoSlots ta = (E == 1 ? kTwoNear : kTwoFar).a[e][w];
    const RowRing<M::PW, E> VA{sphi, (rA - r_begin + 3 * R - 2 - 2 * E) % (2 * R), col + E + po};
    const bool actA = (k >= 0 || w >= R - 4 - 2 * E) && (ALL || (ac && in_y(rA, RIM) && VA.ok()));
    if (actA) {
      const int my = wrap_row(rA);
      const int nd = my * (int)C.rstride + mx;
      load_hg_rg(C, P, nd, hg);
      if (FLOW) load_f_rg(C, P, nd, fv);
      const float php = ldg_plane(P.phi_nm1, my * C.pitch + mx, np);
      ph = VA(0, 0);
      two_collide_gf<FLOW, false>(C, hg, fv, ph, php, U, rho);
    }
    if (k >= 0) mbar_wait(slots_free, k & 1);
    if (actA) {
      const int slots[3] = {slot_a(e, w - 1, E), ta.own, w < R - 1 ? slot_a(e, w + 1, E) : -1};
      two_collide_h<FLOW, EDGE, VAR, false>(C, hg, fv, ph, U, rho, VA, sx, side_y(rA), slots, col, post);
    }
    if (w == R - 1) {  // this row is pulled in the next pass, the row of the pass before now
#pragma unroll
      for (int a = 0; a < 9; ++a) swap_stash(stash_a + a * COLS + col, hg[a].x);
      swap_stash(stash_a + 9 * COLS + col, ph);
    }
    __syncthreads();
    // block k + 1 replaces the half of block k - 1, read for the last time
    if (k + 1 > 1 - LEAD && s + kTwoRows < r_end) phi_block(k + 1);
    // the next pass's node into L1 (this pass still has three phases to run)
    if (k >= 0 && s + R < r_end) prefetch_row(rA + R);

    // ---- A': pull step n + 1 of row rP ----
    const int rP = w < R - 1 ? rA : s + RIM - 1;
    float p1 = 0.0f;
    if ((k >= 0 || (w >= R - 3 - 2 * E && w < R - 1)) && (ALL || (ap && in_y(rP, RIM - 1)))) {
      const int dn = ta.dn * COLS + col, at = ta.at * COLS + col, up = ta.up * COLS + col;
      if (in_range(dn - 1, M::SN, OOB_SHARED) && in_range(at - 1, M::SN, OOB_SHARED) &&
          in_range(up - 1, M::SN, OOB_SHARED) && in_range(dn + 1, M::SN, OOB_SHARED) &&
          in_range(at + 1, M::SN, OOB_SHARED) && in_range(up + 1, M::SN, OOB_SHARED)) {
        two_pull<FLOW>(post, dn, at, up, hg, fv);
        p1 = hg[0].x + (((hg[1].x + hg[3].x) + (hg[2].x + hg[4].x)) +
                        ((hg[5].x + hg[7].x) + (hg[6].x + hg[8].x)));
        const int q = (rP - r_begin + 2 * R) % (2 * R);
        if (in_range(q * COLS + col, M::QN, OOB_SHARED)) sphi1[q * COLS + col] = p1;
        if (EDGE) {  // the ghost places of the phi^{n+1} ring beside this node
          const int sy = side_y(rP);
          const bool ix = sx && (sx < 0 ? C.bc[0] : C.bc[1]) == BC_INLET;
          const bool iy = sy && (sy < 0 ? C.bc[2] : C.bc[3]) == BC_INLET;
          const int qy = (q + sy + 2 * R) % (2 * R);
          if (sx) sphi1[q * COLS + col + sx] = ix ? -1.0f : p1;
          if (sy) sphi1[qy * COLS + col] = iy ? -1.0f : p1;
          if (sx && sy) sphi1[qy * COLS + col + sx] = ix || iy ? -1.0f : p1;
        }
        if (bp && rP >= r_begin && rP < r_end && (!EDGE || (rP >= 0 && rP < C.ny)))
          st_plane(P.phi_mid, rP * C.pitch + X, np, p1);
      }
    }
    if (w >= R - 1 - E && w < R - 1) {  // collided in the next pass; now the row of the pass before
      float* st = stash_p + (w - (R - 1 - E)) * (M::NP + 1) * COLS + col;
#pragma unroll
      for (int a = 0; a < 9; ++a) {
        swap_stash(st + a * COLS, hg[a].x);
        swap_stash(st + (9 + a) * COLS, hg[a].y);
        if (FLOW) swap_stash(st + (18 + a) * COLS, fv[a]);
      }
      swap_stash(st + M::NP * COLS, ph);
    }

    // ---- B: collide step n + 1 of row rB (its phi^n is ph): g and f before the barrier ----
    const bool late = w >= R - 1 - E && w < R - 1;
    const int rB = late ? rP - R : rP;
    const TwoSlots tb = (E == 1 ? kTwoNear : kTwoFar).b[e][w];
    const RowRing<COLS, E> VB{sphi1, (rB - r_begin + 2 * R) % (2 * R), col};
    const bool actB = (k >= 0 || w == R - 3 - E || w == R - 2 - E) && (ALL || (bc && in_y(rB, 1) && VB.ok()));
    if (actB) {
      if (late) p1 = VB(0, 0);  // this thread's own value of the pass before
      two_collide_gf<FLOW, false>(C, hg, fv, p1, ph, U, rho);
    }
    __syncthreads();
    if (actB) {
      const int i = two_bc(w, E);
      const int slots[3] = {slot_b(e, i - 1, E), tb.own, i < R - 1 ? slot_b(e, i + 1, E) : -1};
      two_collide_h<FLOW, EDGE, VAR, false>(C, hg, fv, p1, U, rho, VB, sx, side_y(rB), slots, col, post);
    }
    if (w == R - 2 - E) {  // as A's last group
#pragma unroll
      for (int a = 0; a < 9; ++a) swap_stash(stash_b + a * COLS + col, hg[a].x);
    }
    __syncthreads();

    // ---- B': pull step n + 2 of row rO and store it ----
    const int rO = w == R - 2 - E ? s : rB;
    if (k >= 0 && bp && (!EDGE || rO >= 0)) {
      const int dn = tb.dn * COLS + col, at = tb.at * COLS + col, up = tb.up * COLS + col;
      if (in_range(dn - 1, M::SN, OOB_SHARED) && in_range(at - 1, M::SN, OOB_SHARED) &&
          in_range(up - 1, M::SN, OOB_SHARED) && in_range(dn + 1, M::SN, OOB_SHARED) &&
          in_range(at + 1, M::SN, OOB_SHARED) && in_range(up + 1, M::SN, OOB_SHARED)) {
        float hown[9];
#pragma unroll
        for (int a = 0; a < 9; ++a) hown[a] = hg[a].x;
        pull_store<FLOW, F32>(C, P, X, rO,
                              [&](int a) {
                                const int cy = cy_of(a);
                                return (cy > 0 ? dn : (cy < 0 ? up : at)) - cx_of(a);
                              },
                              post, hown);
      }
    }
    if (s + kTwoRows >= r_end) break;
    mbar_arrive_warp(slots_free, col);
  }
}

// A CTA whose phi columns and rows (four beyond what it owns) all lie inside the grid runs the
// march compiled without ghost handling.
template <bool FLOW, int VAR>
__device__ __forceinline__ void two_cta(const Consts& C, const StepPtrs& P, int strip, int seg,
                                        int H, float* smem) {
  constexpr int M = two_rim(VAR), B = M + two_reach(VAR);  // phi is read B beyond what is owned
  const int X0 = strip * two_out(VAR);
  const int r0 = seg * H - two_pad(C.ny), r1 = min(C.ny, r0 + H);
  if (X0 >= B && X0 - 2 * M + kTwoCols + B <= C.nx && r0 >= B && r1 + B <= C.ny)
    two_range<FLOW, false, VAR>(C, P, X0, r0, r1, smem);
  else
    two_range<FLOW, true, VAR>(C, P, X0, r0, r1, smem);
}

template <bool FLOW, int VAR>
__global__ void __launch_bounds__(kTwoRows* kTwoCols, two_ctas(FLOW)) two_kernel(const Consts C, const StepPtrs P) {
  extern __shared__ __align__(128) float march_smem[];
  const int strip = blockIdx.x + start_after_previous();
  two_cta<FLOW, VAR>(C, P, strip, blockIdx.y, C.two_rows, march_smem);
}

// ---- small grids: two steps of a tile per CTA ----------------------------------------------
// One CTA of W warps takes two steps of W - 6 rows of a strip at once: warp w holds row r0 - 3 + w
// in registers throughout, all of them collide step n, all but the outermost pull and collide
// step n + 1 and the inner W - 6 pull step n + 2. No prologue pass and no state carried from
// pass to pass: W/(W - 6) of the collisions for the shortest chain of dependent phases, which is
// what a grid too small to fill the GPU spends its time on.
template <bool FLOW, int W, int VAR = TWO_DEFAULT>
struct TileTwoSmem {
  static constexpr int E = two_reach(VAR);
  static constexpr int SN = W * kTwoCols, PW = kTwoCols + 2 * E, PN = (W + 2 * E) * PW, QN = W * kTwoCols;
  static constexpr size_t bytes() { return sizeof(float) * (PostTile::floats<FLOW>(SN) + PN + QN); }
};

// KEEP: step n + 1 is stored, too (the tape's recomputation of a segment's states).
template <bool FLOW, bool EDGE, int W, bool KEEP, int VAR, class S>
__device__ __forceinline__ void two_tile_range(const Consts& C, const StepPtrs& P, int X0, int r0,
                                               float* smem) {
  using M = TileTwoSmem<FLOW, W, VAR>;
  constexpr int COLS = kTwoCols, E = M::E, RIM = two_rim(VAR);
  constexpr bool DEV = Storage<S>::DEV;
  const PostTile post = PostTile::at<FLOW>(smem, M::SN);
  float* sphi = smem + PostTile::floats<FLOW>(M::SN);
  float* sphi1 = sphi + M::PN;
  const int col = threadIdx.x % COLS;
  const int w = threadIdx.x / COLS;
  const int X = X0 - RIM + col, r = r0 - RIM + w;
  const long long np = (long long)C.pitch * C.ny;
  const bool xper = !EDGE || C.bc[0] == BC_PERIODIC, yper = !EDGE || C.bc[2] == BC_PERIODIC;
  const auto inside = [&](int halo) {
    return !EDGE || ((xper ? X <= C.nx - 1 + halo : (X >= 0 && X < C.nx)) &&
                     (yper ? (r >= -halo && r <= C.ny - 1 + halo) : (r >= 0 && r < C.ny)));
  };
  const int mx = !EDGE ? X : (X < 0 ? X + C.nx : (X >= C.nx ? X - C.nx : X));
  const int my = !EDGE ? r : (r < 0 ? r + C.ny : (r >= C.ny ? r - C.ny : r));
  const int sx = EDGE && !xper ? (X == 0 ? -1 : (X == C.nx - 1 ? 1 : 0)) : 0;
  const int sy = EDGE && !yper ? (r == 0 ? -1 : (r == C.ny - 1 ? 1 : 0)) : 0;
  const int slots[3] = {w - 1, w, w + 1 < W ? w + 1 : -1};

  // ---- A: the node's loads, phi^n with a halo of E around the collided nodes into shared memory,
  //      collision ----
  float2 hg[9];
  float fv[9], ph = 0.0f, U = 0.0f, rho = 1.0f;
  const bool actA = inside(RIM);
  float php = 0.0f;
  if (actA) {
    const int nd = my * (int)C.rstride + mx;
    if constexpr (!DEV) {
      load_hg_rg(C, P, nd, hg);
      if (FLOW) load_f_rg(C, P, nd, fv);
    } else {
      deviations_hg<S>(ldg_vec_rg(C, P, 0, nd), ldg_vec_rg(C, P, 1, nd), hg);
      U = ldg_plane(P.U_n, my * C.pitch + mx, np);
      if (FLOW) {
        deviations9<S>(ldg_vec_rg(C, P, 2, nd), fv);
        rho = ldg_plane(P.rho_n, my * C.pitch + mx, np);
      }
    }
    php = ldg_plane(P.phi_nm1, my * C.pitch + mx, np);
    ph = ldg_plane(P.phi_n, my * C.pitch + mx, np);
  }
  for (int i = w; i < W + 2 * E; i += W) {
    const int rl = r0 - RIM - E + i;
    for (int c = col; c < COLS + 2 * E; c += COLS) {
      const int xg = X0 - RIM - E + c;
      float v = -1.0f;
      int gx, gy;
      if (EDGE && (xg > C.nx - 1 + RIM + E || rl > C.ny - 1 + RIM + E)) {
        v = 0.0f;  // beyond the grid's halo (ragged last tile): never read
      } else if (!EDGE) {
        v = ldg_plane(P.phi_n, rl * C.pitch + xg, np);
      } else if (axis_phi(xg, C.nx, C.bc[0], C.bc[1], gx) && axis_phi(rl, C.ny, C.bc[2], C.bc[3], gy)) {
        v = ldg_plane(P.phi_n, gy * C.pitch + gx, np);
      }
      if (in_range(i * M::PW + c, M::PN, OOB_SHARED)) sphi[i * M::PW + c] = v;
    }
  }
  if (actA) two_collide_gf<FLOW, DEV>(C, hg, fv, ph, php, U, rho);
  __syncthreads();
  if (actA) {
    const TileView V{sphi, (w + E) * M::PW + col + E, M::PW, M::PN, E};
    if (V.ok()) two_collide_h<FLOW, EDGE, VAR, DEV>(C, hg, fv, ph, U, rho, V, sx, sy, slots, col, post);
  }
  __syncthreads();

  // ---- A': pull step n + 1, collide its g and f ----
  const int dn = (w - 1) * COLS + col, at = w * COLS + col, up = (w + 1) * COLS + col;
  float p1 = 0.0f;
  const bool actP = w >= 1 && w <= W - 2 && col >= 1 && col < COLS - 1 && inside(1 + E);
  const bool own = col >= RIM && col < COLS - RIM && w >= RIM && w < W - RIM && X < C.nx && r < C.ny;
  if (actP) {
    if (in_range(dn - 1, M::SN, OOB_SHARED) && in_range(up + 1, M::SN, OOB_SHARED)) {
      if (DEV) {
#pragma unroll
        for (int a = 0; a < 9; ++a) hg[a].x = fmaf(w_of(a), ph, hg[a].x);
      }
      two_pull<FLOW>(post, dn, at, up, hg, fv);
      p1 = hg[0].x + (((hg[1].x + hg[3].x) + (hg[2].x + hg[4].x)) +
                      ((hg[5].x + hg[7].x) + (hg[6].x + hg[8].x)));
      if constexpr (DEV) {
        // the moments and the rounded deviations that a single step would have stored
        const float2 m = sum9_2(hg);
        float dh[8], dg[8];
#pragma unroll
        for (int a = 1; a < 9; ++a) {
          const float2 d = ffma2(splat(-w_of(a)), m, hg[a]);
          dh[a - 1] = d.x;
          dg[a - 1] = d.y;
        }
        deviations_hg<S>(Storage<S>::pack8(dh), Storage<S>::pack8(dg), hg);
        U = m.y;
        if (FLOW) {
          rho = sum9(fv);
          float df[8];
#pragma unroll
          for (int a = 1; a < 9; ++a) df[a - 1] = fmaf(-w_of(a), rho, fv[a]);
          deviations9<S>(Storage<S>::pack8(df), fv);
        }
      }
      sphi1[at] = p1;
      if (EDGE) {  // the ghost places beside this node
        const bool ix = sx && (sx < 0 ? C.bc[0] : C.bc[1]) == BC_INLET;
        const bool iy = sy && (sy < 0 ? C.bc[2] : C.bc[3]) == BC_INLET;
        if (sx) sphi1[at + sx] = ix ? -1.0f : p1;
        if (sy) sphi1[at + sy * COLS] = iy ? -1.0f : p1;
        if (sx && sy) sphi1[at + sy * COLS + sx] = ix || iy ? -1.0f : p1;
      }
      if (own) {
        st_plane(P.phi_mid, r * C.pitch + X, np, p1);
        if (KEEP) {
          const int nd = r * (int)C.rstride + X;
          store_hg_rg(C, P.rmid, nd, hg);
          if (FLOW) store_f_rg(C, P.rmid, nd, fv);
        }
      }
      two_collide_gf<FLOW, DEV>(C, hg, fv, p1, ph, U, rho);
    }
  }
  __syncthreads();

  // ---- B: collide step n + 1 ----
  if (w >= RIM - 1 && w <= W - RIM && col >= RIM - 1 && col <= COLS - RIM && inside(1)) {
    const TileView V{sphi1, at, COLS, M::QN, E};
    if (V.ok()) two_collide_h<FLOW, EDGE, VAR, DEV>(C, hg, fv, p1, U, rho, V, sx, sy, slots, col, post);
  }
  __syncthreads();

  // ---- B': pull step n + 2 and store it ----
  if (own) {
    float hown[9];
#pragma unroll
    for (int a = 0; a < 9; ++a) hown[a] = DEV ? fmaf(w_of(a), p1, hg[a].x) : hg[a].x;
    if (in_range(dn - 1, M::SN, OOB_SHARED) && in_range(up + 1, M::SN, OOB_SHARED))
      pull_store<FLOW, S>(C, P, X, r,
                            [&](int a) {
                              const int cy = cy_of(a);
                              return (cy > 0 ? dn : (cy < 0 ? up : at)) - cx_of(a);
                            },
                            post, hown);
  }
}

template <bool FLOW, int W, bool KEEP, int VAR, class S>
__device__ __forceinline__ void two_tile_cta(const Consts& C, const StepPtrs& P, int strip, int tile,
                                             float* smem) {
  constexpr int M = two_rim(VAR), H = M + two_reach(VAR);  // phi columns X0 - H .. X0 - M + 31 + H - M
  const int X0 = strip * two_out(VAR), r0 = tile * (W - 2 * M);
  if (X0 >= H && X0 - 2 * M + kTwoCols + H <= C.nx && r0 >= H && r0 - 2 * M + W + H <= C.ny)
    two_tile_range<FLOW, false, W, KEEP, VAR, S>(C, P, X0, r0, smem);
  else
    two_tile_range<FLOW, true, W, KEEP, VAR, S>(C, P, X0, r0, smem);
}

// Two CTAs per SM (three of 8 warps).
template <bool FLOW, int W, bool KEEP = false, int VAR = TWO_DEFAULT, class S = F32>
__global__ void __launch_bounds__(32 * W, W <= 8 ? 3 : 2)
    two_tile_kernel(const Consts C, const StepPtrs P) {
  extern __shared__ __align__(128) float march_smem[];
  two_tile_cta<FLOW, W, KEEP, VAR, S>(C, P, (int)blockIdx.x + start_after_previous(), blockIdx.y, march_smem);
}

// The two-step march over the members of a batched launch: one CTA per (strip, segment),
// numbered as in batch_march_kernel.
template <bool FLOW>
__global__ void __launch_bounds__(kTwoRows* kTwoCols, two_ctas(FLOW))
    batch_two_kernel(const __grid_constant__ BatchLaunch L) {
  extern __shared__ __align__(128) float march_smem[];
  const long long t = (int)blockIdx.x + start_after_previous();
  const int m = batch_member_of(L, t);
  const BatchDesc& d = L.d[m];
  const int local = (int)(t - L.tile_start[m]);
  const int seg = local / d.tiles_x, strip = local - seg * d.tiles_x;
  if (local < 0 || seg * d.C.two_rows - two_pad(d.C.ny) >= d.C.ny) return;
  two_cta<FLOW, TWO_DEFAULT>(d.C, d.P, strip, seg, d.C.two_rows, march_smem);
}

// The two-step tiles of the members of a batched launch, numbered tile row by tile row.
template <bool FLOW, int W>
__global__ void __launch_bounds__(32 * W, 2)
    batch_two_tile_kernel(const __grid_constant__ BatchLaunch L) {
  extern __shared__ __align__(128) float march_smem[];
  const long long t = (int)blockIdx.x + start_after_previous();
  const int m = batch_member_of(L, t);
  const BatchDesc& d = L.d[m];
  const int local = (int)(t - L.tile_start[m]);
  const int tile = local / d.tiles_x, strip = local - tile * d.tiles_x;
  if (local < 0 || tile * (W - 6) >= d.C.ny) return;
  two_tile_cta<FLOW, W, false, TWO_DEFAULT, F32>(d.C, d.P, strip, tile, march_smem);
}

}  // namespace lbmice

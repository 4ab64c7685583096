// The bulk stage kernel k_stage<R, TY> (a template instantiated per precision
// in m2c_stage_fp32.cu and m2c_stage_fp64.cu) and its launch helpers.
#pragma once
#include <cuda_runtime.h>

#include <algorithm>

#include "m2c_device.cuh"
#include "m2c_stage.h"

namespace m2c {

// ---------------------------------------------------------------------------
// Bulk stage kernel
// ---------------------------------------------------------------------------

// Shared memory of a tile: the plane being worked on and the next one (primitive
// fields, level set, material ids, with a two-cell halo); what a row hands to the
// row on its minus side (ym, the MUSCL states on the minus y faces of rows 0 ..
// TY) and on its plus side (yf, the fluxes through the plus y faces; row 0 is the
// tile's minus face); the states on both sides of the tile's two x faces (xe: cells
// -1, 0, 31, 32 of every row) and the fluxes through them (xf); the plus states of
// row -1 (yp); per thread the plus z state of
// its next cell (qz) and the last two z fluxes (fz); per row which cells equal
// those of the next row (ey), and whether its end faces count (ex).
template <typename R, int TY>
struct StageSmem {
  static constexpr int TX = 32, HX = TX + 4, HY = TY + 4, PL = HX * HY, NT = TX * TY;
  static constexpr size_t q_off = 0;
  static constexpr size_t phi_off = q_off + sizeof(R) * 2 * 5 * PL;
  static constexpr size_t ym_off = phi_off + sizeof(R) * 2 * PL;
  static constexpr size_t yf_off = ym_off + sizeof(R) * 7 * (TY + 1) * TX;
  static constexpr size_t qz_off = yf_off + sizeof(R) * 5 * (TY + 1) * TX;
  static constexpr size_t fz_off = qz_off + sizeof(R) * 7 * NT;
  static constexpr size_t xe_off = fz_off + sizeof(R) * 2 * 5 * NT;
  static constexpr size_t xf_off = xe_off + sizeof(R) * 7 * 4 * TY;
  static constexpr size_t yp_off = xf_off + sizeof(R) * 5 * 2 * TY;
  static constexpr size_t ey_off = yp_off + sizeof(R) * 7 * TX;
  static constexpr size_t id_off = ey_off + sizeof(unsigned) * (2 * TY + 4);
  static constexpr size_t bytes = (id_off + 2 * PL + 15) / 16 * 16;
};

// Shared-plane slot of the cell outside the tile whose face states lane tx of warp ty
// takes (the tile's last three warps: columns -1 and 32, row -1, row TY), and the axis
// stride so of its neighbours. A lane with no such cell to take (on false: past the two
// columns of the x warp, or a row beyond the grid, whose slots of a plane are never
// written) gets the first cell of the tile's row 0, which is always inside the grid, so
// that what it reads is defined (a material id is used as an index); its result is not.
template <int TY>
__host__ __device__ constexpr int outside_slot(int ty, int tx, bool on, int& so) {
  constexpr int TX = 32, HX = TX + 4;
  so = ty == TY - 3 ? 1 : HX;
  if (ty == TY - 3) return on ? ((tx & (TY - 1)) + 2) * HX + (tx / TY ? TX + 2 : 1) : 2 * HX + 2;
  return (ty == TY - 2 ? 1 : TY + 2) * HX + tx + 2;
}

// Shared-plane slot of halo load h of a tile (the two-cell ring without corners: four
// columns of TY rows, padded to whole warps, then four rows of 32); -1: none.
template <int TY>
__host__ __device__ constexpr int halo_slot_of(int h) {
  constexpr int TX = 32, HX = TX + 4, NHX = (4 * TY + 31) / 32 * 32;
  const int h2 = h - NHX;
  if (h < 4 * TY) {
    const int c4 = h / TY;
    return (h % TY + 2) * HX + (c4 < 2 ? c4 : TX + c4);
  }
  if (h2 >= 0 && h2 < 4 * TX) {
    const int c4 = h2 / TX;
    return (c4 < 2 ? c4 : TY + c4) * HX + h2 % TX + 2;
  }
  return -1;
}

// Compile-time integer for the material dispatch below (usable in device code).
template <int V>
struct IntC {
  static constexpr int value = V;
  __device__ constexpr operator int() const { return V; }
};

// Calls f(T, m) for material m of a cell: T its EOS type as a compile-time
// constant when the instantiation fixes the pair of material types (MT = T0 +
// 4 T1, each M2C_EOS_SG or M2C_EOS_MG), else IntC<-1> (the type is read at run
// time); m the material index, itself a compile-time constant where the two
// fixed types differ (f is then inlined once per material).
template <int MT, typename F>
__device__ __forceinline__ void by_material(int m, F&& f) {
  if constexpr (MT < 0) {
    f(IntC<-1>{}, m);
  } else if constexpr ((MT & 3) == (MT >> 2)) {
    f(IntC<(MT & 3)>{}, m);
  } else {
    if (m == 0) f(IntC<(MT & 3)>{}, IntC<0>{});
    else f(IntC<(MT >> 2)>{}, IntC<1>{});
  }
}

// Face states of a cell of material ic along one axis (cell_faces). For FP32 and a
// fixed pair of types the slopes, the face values and everything but e and c^2 are
// one code for both materials (a warp across the interface takes only the equation
// of state twice), without branches but for states that are not admissible; a zero
// slope gives the cell state itself.
template <bool GEN, int MT, typename R, typename EA>
__device__ __forceinline__ void material_faces(EA&& eos, int ic, const R Pm[5], const R P[5], const R Pp[5], bool same,
                                               FaceState<R>& QM, FaceState<R>& QP, bool& bad, int lim, R alpha) {
  if constexpr (sizeof(R) == 4 && !GEN && MT >= 0) {
    float a[5], b[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      const float s = va_slope<float>(P[v] - Pm[v], Pp[v] - P[v]), h = same ? s : 0.0f;
      a[v] = __fmaf_rn(-0.5f, h, P[v]);
      b[v] = __fmaf_rn(0.5f, h, P[v]);
    }
    const float ia = rrcp<float>(a[0]), ib = rrcp<float>(b[0]);
    float ea, ca, eb, cb;
    bool oka, okb;
    by_material<MT>(ic, [&](auto T, auto m) {
      oka = face_eos_f<decltype(T)::value>(eos(m), a[0], ia, a[4], ea, ca);
      okb = face_eos_f<decltype(T)::value>(eos(m), b[0], ib, b[4], eb, cb);
    });
    if (!(oka && okb)) {
      // first order (Reading R12)
      by_material<MT>(ic, [&](auto T, auto m) {
        oka = face_eos_f<decltype(T)::value>(eos(m), P[0], rrcp<float>(P[0]), P[4], ea, ca);
      });
      if (!oka) bad = true;
      okb = oka;
      eb = ea;
      cb = ca;
#pragma unroll
      for (int v = 0; v < 5; ++v) a[v] = b[v] = P[v];
    }
    finish_face_f(a, ea, ca, oka, QM);
    finish_face_f(b, eb, cb, okb, QP);
  } else {
    by_material<MT>(ic, [&](auto T, auto m) {
      cell_faces<R, GEN, decltype(T)::value>(eos(m), Pm, P, Pp, same, QM, QP, bad, lim, alpha);
    });
  }
}

// A tile is 32 x TY columns marching along z, one warp per row of 32 cells, one
// thread per column. Per plane and thread: the face states along z (from a register
// window), x and y (from the shared plane) of its own cell, the fluxes through its
// own plus faces with the neighbour's minus state (by shuffle along x, through
// shared memory along y), the residual and the update. The cells and faces just
// outside the tile that its fluxes need (columns -1 and 32, rows -1 and TY) are
// taken by three warps on top of their own row, the halo loads by others. The
// face states of all of them are one loop, so that the reconstruction and the
// equation of state are one piece of code (six copies of it doubled the stalls for
// instructions). Two block barriers per plane: after the minus states, and after
// the y fluxes; plane k+1 is staged during plane k, so that the update of a plane
// and the loads and face states of the next run without a barrier between them.
//
// Uniform rows. Where a cell and its two neighbours along an axis hold the same
// primitive state and material, its slopes and those of the neighbours towards it
// vanish, both fluxes of the axis are the flux of that one state, and their
// difference is exactly zero. A warp whose 32 cells and their neighbours are so
// along an axis leaves out the axis' face states and fluxes (fluid at rest ahead
// of a shock, the uniform state behind it, the inside of a bubble: most of the
// domain until the waves have crossed it); one uniform along all three copies the
// state. The results are the same bits.
//
// What bounds it: FP32 tiles the instruction issue and the latency of each warp's
// chain (about 820 instructions a cell and stage without any face state, 1700 in an
// early shock-bubble), compiled for 512 resident threads per SM (128 registers; no
// spills but 8 to 32 bytes in the MG/SG and SG/MG kernels of batches; with 1024 threads at
// 64 registers the spills went to L2, the shared memory leaving little L1, and took as
// long); FP64 tiles the FP64 pipe. Against face states
// and fluxes as items distributed over the threads (2.2 and 2.1 a thread, all states
// and fluxes through shared memory, three barriers, no uniform rows), per launch:
// 256^3 mixed 1947 -> 1617 us, 192^3 with the shock in the bubble 1028 -> 927,
// 131x67x45 120 -> 103, 48^3 38 -> 34.5; FP64 128^3 2064 -> 1277, 75x51x67 with
// mirrors 507 -> 380.
//
// GEN = false is the default scheme (TVD RK2, modified van Albada, HLLC); GEN =
// true is the general instantiation, which takes the grid's scheme options at
// run time (limiter, flux, the stages of TVD RK3) at some cost in registers.
// MT >= 0 fixes the EOS types of the two materials (SG or MG, MT = T0 + 4 T1)
// for launches whose grids all have that pair, which removes the type dispatch
// from every EOS evaluation; MT = -1 reads the types at run time.
//
// ONE (mixed path, default scheme): the launch's only grid comes as a kernel
// parameter, so that its pointers, sizes and EOS constants are constant-bank operands
// instead of loads from shared memory and registers; else the descriptor of the
// tile's grid is copied to shared memory.
template <bool ONE>
struct StageArg {
  Grid grid;
};
template <>
struct StageArg<false> {};

template <typename R, int TY, bool GEN, int MT, bool ONE>
__global__ void __launch_bounds__(32 * TY, (sizeof(R) == 8 ? 1 : 512 / (32 * TY)))
k_stage(const __grid_constant__ StageArg<ONE> arg, const Grid* __restrict__ grids,
        const long long* __restrict__ tile_begin, int ngrid, long long ntiles, int mode, int sched,
        unsigned long long* __restrict__ tile_counter) {
  constexpr int TX = 32, NT = TX * TY, HX = TX + 4, HY = TY + 4, PL = HY * HX;
  // halo cells of a plane: four columns of TY (padded to whole warps), then four rows of 32
  constexpr int NHX = (4 * TY + 31) / 32 * 32, NHALO = NHX + 4 * TX;
  constexpr int HI = (NHALO + NT - 1) / NT;
  // warps with work outside the tile: the cells of columns -1 and 32, of row -1, of row TY
  constexpr int kWarpX = TY - 3, kWarpY0 = TY - 2, kWarpY1 = TY - 1;
  static_assert(TY >= 4 && 2 * TY <= 32, "columns -1 and 32 of a tile are the lanes of one warp");
  using SM = StageSmem<R, TY>;
  constexpr int SYM = (TY + 1) * TX, SXE = 4 * TY;  // strides of the state and flux components
  extern __shared__ __align__(16) unsigned char smem[];
  R* const s_q = reinterpret_cast<R*>(smem + SM::q_off);      // [2][5][HY][HX]
  R* const s_phi = reinterpret_cast<R*>(smem + SM::phi_off);  // [2][HY][HX]
  R* const s_ym = reinterpret_cast<R*>(smem + SM::ym_off);    // [7][TY+1][32]
  R* const s_yf = reinterpret_cast<R*>(smem + SM::yf_off);    // [5][TY+1][32]
  R* const s_qz = reinterpret_cast<R*>(smem + SM::qz_off);    // [7][NT]
  R* const s_fz = reinterpret_cast<R*>(smem + SM::fz_off);    // [2][5][NT]
  R* const s_xe = reinterpret_cast<R*>(smem + SM::xe_off);    // [7][4][TY]: plus state of cell -1, minus of 0, plus of 31, minus of 32
  R* const s_xf = reinterpret_cast<R*>(smem + SM::xf_off);    // [5][2][TY]
  R* const s_yp = reinterpret_cast<R*>(smem + SM::yp_off);    // [7][32]
  unsigned* const s_ey = reinterpret_cast<unsigned*>(smem + SM::ey_off);  // [TY+3], rows -2 .. TY
  unsigned* const s_ex = s_ey + TY + 3;                                   // [TY]
  uint8_t* const s_id = smem + SM::id_off;                    // [2][HY][HX]
  // the descriptor of the tile's grid: the parameter, or copied to shared memory for each tile
  // (its fields and EOS parameters are read all through the plane loop)
  constexpr size_t kGridBytes = ONE ? 16 : sizeof(Grid);
  __shared__ __align__(16) unsigned char s_grid[kGridBytes];
  static_assert(sizeof(Grid) % 8 == 0, "grid descriptor copy");
  const Grid* Gp;
  if constexpr (ONE) Gp = &arg.grid;
  else Gp = reinterpret_cast<const Grid*>(s_grid);
  const Grid& G = *Gp;
  auto eos = [&](auto m) -> const EosP<R>& {
    if constexpr (sizeof(R) == 8) return G.eos[m];
    else return G.eosf[m];
  };
  auto eosd = [&](auto m) -> const EosDev& { return G.eos[m]; };
  __shared__ double s_dt;
  __shared__ double s_red[32];
  __shared__ long long s_tile;

  const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
  const unsigned lane = tid & 31, lt = (1u << lane) - 1u;
  // halo cell s of a plane loaded by this thread (two-cell ring without corners): its slot, -1: none
  auto halo_slot = [&](int s) { return halo_slot_of<TY>(tid + s * NT); };

  // Tiles of all grids of the launch, taken in order by a fixed stride
  // (sched 0) or from an atomic counter (sched 1).
  for (long long iter = 0;; ++iter) {
  long long tile;
  if (sched == 1) {
    if (tid == 0) s_tile = (long long)atomicAdd(tile_counter, 1ull);
    __syncthreads();
    tile = s_tile;
  } else {
    tile = blockIdx.x + iter * (long long)gridDim.x;
  }
  if (tile >= ntiles) break;
  long long t = tile;
  if constexpr (!ONE) {
    const int gidx = find_grid(tile_begin, ngrid, tile);
    const unsigned long long* src = reinterpret_cast<const unsigned long long*>(grids + gidx);
    unsigned long long* dst = reinterpret_cast<unsigned long long*>(s_grid);
    for (int i = tid; i < (int)(sizeof(Grid) / 8); i += NT) dst[i] = __ldg(src + i);
    t -= tile_begin[gidx];
    __syncthreads();
  }
  const int nx = G.nx, ny = G.ny, nz = G.nz;
  const long long N = G.N;
  const int nxy = nx * ny;
  const int bcz0 = G.bc[4], bcz1 = G.bc[5];
  const int bx = (int)(t % G.tiles_x);
  t /= G.tiles_x;
  const int by = (int)(t % G.tiles_y);
  const int bz = (int)(t / G.tiles_y);
  const int x0 = bx * TX, y0 = by * TY, k0 = bz * G.tz, k1 = min(k0 + G.tz, nz);
  const R ih = (R)G.inv_h;
  const R i6h = (R)(1.0 / (6.0 * G.h));
  const double* __restrict__ Ws = GEN ? stage_W(G, mode) : (mode == kStage2 ? G.W1 : G.W);
  const double* __restrict__ phis = GEN ? stage_phi(G, mode) : (mode == kStage2 ? G.phi1 : G.phi);
  const uint8_t* __restrict__ idg = G.id;
  Ctrl* ctrl = G.ctrl;
  const int slot = GEN ? list_slot(mode) : (mode == kStage2 ? 1 : 0);
  // material ids are frozen after the first stage of a step
  const bool ids_frozen = GEN ? (mode != kStage1 && mode != kResidual) : mode == kStage2;
  const bool final_stage = GEN ? last_stage(mode) : mode == kStage2;
  const int lim = GEN ? G.limiter : 0, flx = GEN ? G.flux : 0;
  const R alpha = GEN ? (R)G.mc_alpha : (R)0;
  const long long step = ctrl->step;

  if (tid == 0) s_dt = mode == kResidual ? 0.0 : lam_to_dt(G, ctrl->lam[step & 1]);
  __syncthreads();
  const double dt = s_dt;
  const R hdt = to_r<R>(0.5 * dt);

  const int gx = x0 + tx, gy = y0 + ty;
  const bool inside = gx < nx && gy < ny;
  // column bases (x, y mapped once per tile; a grid has fewer than 2^31 cells)
  const int own_base = map_index(gy, ny, G.bc[2], G.bc[3]) * nx + map_index(gx, nx, G.bc[0], G.bc[1]);
  int halo_base[HI];
  // general kernel: velocity components to negate for a position mirrored across a
  // symmetry side (bit 0: u, bit 1: v, bit 2: w), for the own column and the halo slots
  int own_neg = 0, halo_neg[HI];
  if constexpr (GEN) own_neg = mirrored(gx, nx, G.bc[0], G.bc[1]) | (mirrored(gy, ny, G.bc[2], G.bc[3]) << 1);
#pragma unroll
  for (int s = 0; s < HI; ++s) {
    const int slot = halo_slot(s), hx = x0 + slot % HX - 2, hy = y0 + slot / HX - 2;
    halo_base[s] = slot < 0 ? 0 : map_index(hy, ny, G.bc[2], G.bc[3]) * nx + map_index(hx, nx, G.bc[0], G.bc[1]);
    halo_neg[s] = 0;
    if constexpr (GEN) {
      if (slot >= 0) halo_neg[s] = mirrored(hx, nx, G.bc[0], G.bc[1]) | (mirrored(hy, ny, G.bc[2], G.bc[3]) << 1);
    }
  }
  auto zneg = [&](int k) { return GEN ? (mirrored(k, nz, bcz0, bcz1) << 2) : 0; };

  // failures seen by this thread in this tile: non-physical state, work-list overflow
  bool bad = false, ovf = false;
  // material at the start of the step and the stage state of cell index c
  // (neg: the velocity components to negate, general kernel only)
  auto load = [&](int c, R P[5], R& ph, int& idv, int neg) {
    const double phd = gld(phis + c);
    if (ids_frozen) idv = __ldg(idg + c) & 1;
    const double w0 = gld(Ws + c), w1 = gld(Ws + N + c), w2 = gld(Ws + 2 * N + c), w3 = gld(Ws + 3 * N + c),
                 w4 = gld(Ws + 4 * N + c);
    if constexpr (sizeof(R) == 8) {
      ph = phd;
      if (!ids_frozen) idv = lt0(phd) ? 1 : 0;
      by_material<MT>(idv, [&](auto T, auto m) {
        if (!cons_to_prim_v<R, GEN, decltype(T)::value>(eos(m), eosd(m), w0, w1, w2, w3, w4, P)) bad = true;
      });
    } else {
      // the level set and the state's first four components: one group of conversions
      const double x[5] = {phd, w0, w1, w2, w3};
      float y[5];
      d2f_group<5>(x, y);
      ph = y[0];
      if (!ids_frozen) idv = lt0(phd, y[0]) ? 1 : 0;
      P[0] = y[1];
      const float inv = rrcp<float>(y[1]);
      const double rhoe = prim_velocities_f(inv, y[2], y[3], y[4], w4, P);
      bool ok;
      by_material<MT>(idv, [&](auto T, auto m) {
        ok = prim_pressure_f<GEN, decltype(T)::value>(eos(m), eosd(m), w0, y[1], inv, rhoe, P[4]);
      });
      bad = bad || !ok || !gt0(w0, y[1]);
    }
    if constexpr (GEN) {
      if (neg & 1) P[1] = -P[1];
      if (neg & 2) P[2] = -P[2];
      if (neg & 4) P[3] = -P[3];
    }
  };
  auto plane = [&](int k) { return map_index(k, nz, bcz0, bcz1) * nxy; };

  // rows of a tile cut by the grid's edge: those inside, and the two beyond it that hold halo
  // cells (the first one's y states are needed too); the others do nothing
  const bool row_in = gy < ny, row_y = gy <= ny, row_on = gy <= ny + 1;
  const int cslot = (ty + 2) * HX + tx + 2;
  auto put = [&](int b, int slot, const R P[5], R phv, int idv) {
#pragma unroll
    for (int v = 0; v < 5; ++v) s_q[(b * 5 + v) * PL + slot] = P[v];
    s_phi[b * PL + slot] = phv;
    s_id[b * PL + slot] = (uint8_t)idv;
  };
  auto put_halo = [&](int b, int k) {
    const int pk = k * nxy;  // k is inside the grid
#pragma unroll
    for (int s = 0; s < HI; ++s) {
      const int slot = halo_slot(s);
      if (slot < 0) continue;
      R Ph[5], phh;
      int idh;
      load(pk + halo_base[s], Ph, phh, idh, halo_neg[s]);
      put(b, slot, Ph, phh, idh);
    }
  };
  // whether the cells at two slots of a shared plane hold the same primitive state (finite) and material
  auto alike = [](const R* q, const uint8_t* idp, int c0, int c1) {
    bool f = (idp[c0] == idp[c1]) & is_finite(q[4 * PL + c0]);
#pragma unroll
    for (int v = 0; v < 5; ++v) f = f & same_bits(q[v * PL + c0], q[v * PL + c1]);
    return f;
  };
  // Uniformity of a staged plane, known to all warps after the next barrier: bit x of mx, cells x and
  // x + 1 of the own row alike; mx_ends, those at the row's ends too (-2 and -1, -1 and 0, 32 and 33;
  // only looked at where all of mx are); s_ey, the cells of a row and of the next one.
  unsigned mx = 0;
  bool mx_ends = false;
  auto look_at = [&](int b) {
    const R* const q = s_q + b * 5 * PL;
    const uint8_t* const idp = s_id + b * PL;
    if (row_in) {
      mx = __ballot_sync(0xffffffffu, alike(q, idp, cslot, cslot + 1));
      mx_ends = false;
      if (mx == 0xffffffffu) {
        const int c0 = (ty + 2) * HX + (tx < 2 ? tx : (tx == 2 ? TX + 2 : 2));
        mx_ends = __all_sync(0xffffffffu, alike(q, idp, c0, c0 + 1));
      }
      if (tx == 0) s_ex[ty] = mx_ends;
    }
    const unsigned m = __ballot_sync(0xffffffffu, alike(q, idp, cslot, cslot + HX));
    if (tx == 0) s_ey[ty + 2] = m;
    if (ty >= kWarpX) {  // rows -2, -1 and TY
      const int row = ty == kWarpX ? -2 : (ty == kWarpY0 ? -1 : TY);
      const int c0 = (row + 2) * HX + tx + 2;
      const unsigned mr = __ballot_sync(0xffffffffu, alike(q, idp, c0, c0 + HX));
      if (tx == 0) s_ey[row + 2] = mr;
    }
  };
  auto put_state = [](R* o, int stride, const FaceState<R>& Q) {
    o[0] = Q.rho;
    o[stride] = Q.u;
    o[2 * stride] = Q.v;
    o[3 * stride] = Q.w;
    o[4 * stride] = Q.p;
    o[5 * stride] = Q.c;
    o[6 * stride] = Q.E;
  };
  auto get_state = [](const R* o, int stride) {
    return FaceState<R>{o[0], o[stride], o[2 * stride], o[3 * stride], o[4 * stride], o[5 * stride], o[6 * stride]};
  };

  // ---- opening of the z window: planes k0-2 .. k0+1, the flux through the tile's lower z face
  R P1[5], P2[5];
  R ph[5];
  int idm, id0, id1, id2;
  // along z: the cell of plane k is uniform, all of the row's are, qz holds the row's plus states
  bool flat_z0 = false, rowflat_z0 = false, qz_set = true, alike_z = false;
  {
    R Pb[5], Pa[5], P0[5];
    FaceState<R> QzP;
    R Fzm[5];
    int idb, ida;
    load(plane(k0 - 2) + own_base, Pb, ph[0], idb, own_neg | zneg(k0 - 2));
    load(plane(k0 - 1) + own_base, Pa, ph[1], ida, own_neg | zneg(k0 - 1));
    load(plane(k0) + own_base, P0, ph[2], id0, own_neg);
    load(plane(k0 + 1) + own_base, P1, ph[3], id1, own_neg | zneg(k0 + 1));
    FaceState<R> Qtmp, QaP, Q0M;
    material_faces<GEN, MT, R>(eos, ida, Pb, Pa, P0, idb == ida && id0 == ida, Qtmp, QaP, bad, lim, alpha);
    material_faces<GEN, MT, R>(eos, id0, Pa, P0, P1, ida == id0 && id1 == id0, Q0M, QzP, bad, lim, alpha);
    if (ida == id0) {
      num_flux<2, R, GEN>(QaP, Q0M, Fzm, flx);
    } else {
#pragma unroll
      for (int v = 0; v < 5; ++v) Fzm[v] = (R)0;
    }
    idm = ida;
    put_state(s_qz + tid, NT, QzP);
#pragma unroll
    for (int v = 0; v < 5; ++v) s_fz[(5 + v) * NT + tid] = Fzm[v];
    put(0, cslot, P0, ph[2], id0);
    put_halo(0, k0);
  }
  __syncthreads();
  look_at(0);
  __syncthreads();

  R lam_max = (R)0;

  for (int k = k0; k < k1; ++k) {
    const int pk = k * nxy;  // k is inside the grid
    const int buf = (k - k0) & 1;
    const R* const q = s_q + buf * 5 * PL;
    const R* const phip = s_phi + buf * PL;
    const uint8_t* const idp = s_id + buf * PL;
    // faces of the own cell between materials: bits 0, 1 plus x and y, bit 2 any other
    int iff;
    {
      const int xp = idp[cslot + 1] != id0, yp = idp[cslot + HX] != id0;
      iff = xp | (yp << 1) | ((idp[cslot - 1] != id0 || idp[cslot - HX] != id0 || idm != id0 || id1 != id0) ? 4 : 0);
    }

    R* const fz = s_fz + buf * 5 * NT + tid;         // flux through the upper z face
    const R* const fzm = s_fz + (buf ^ 1) * 5 * NT + tid;  // and the lower one

    // ---- to L2: the row's cells of plane k+4 (loaded two planes from now), and the old state of
    // plane k+2 where the update reads one besides the stage's; lanes 0 .. 5 and 6 .. 11, a field each
    if (row_in && tx < (mode == kStage1 || mode == kResidual ? 6 : 12)) {
      const int f = tx < 6 ? tx : tx - 6, kp = tx < 6 ? k + 4 : k + 2;
      const double* const a = f == 5 ? (tx < 6 ? phis : G.phi) : (tx < 6 ? Ws : G.W) + f * N;
      if (kp < nz && kp <= k1 + 1) prefetch_row(a, N, kp * nxy + gy * nx + x0);
    }
    // ---- plane k+1 into shared memory: own cells and the two-cell halo (no corners); own
    // column: plane k+2
    if (row_on) {
      put(buf ^ 1, cslot, P1, ph[3], id1);
      load(plane(k + 2) + own_base, P2, ph[4], id2, own_neg | zneg(k + 2));
    }
    if (k + 1 < k1) put_halo(buf ^ 1, k + 1);
    const R* const qn = s_q + (buf ^ 1) * 5 * PL + cslot;

    // ---- uniform cells and rows; face-state jobs of this warp: bit 0 the plus z state of cell k
    // where it was left out before, 1 z (cell k+1), 2 x, 3 y, 4 a cell outside the tile
    bool flat_x = false, flat_y = false, flat_z1 = false, rowflat_z1 = false, need_yp = true;
    unsigned jobs = 0;
    if (row_in) {
      // alike_z: cells k and k+1; a cell is uniform along an axis if it is like both neighbours
      bool az = is_finite(P1[4]) & (id1 == id2);
#pragma unroll
      for (int v = 0; v < 5; ++v) az = az & same_bits(P1[v], P2[v]);
      flat_z1 = alike_z & az;
      alike_z = az;
      rowflat_z1 = __all_sync(0xffffffffu, flat_z1);
      if (!(rowflat_z0 && rowflat_z1)) jobs |= qz_set ? 2u : 3u;
      qz_set = jobs != 0;
      // a row's first and last cell count as uniform where the cells outside it were looked at
      const unsigned m = mx & (mx << 1 | (mx_ends ? 1u : 0u)) & (mx_ends ? 0xffffffffu : 0x7fffffffu);
      flat_x = (m >> tx) & 1u;
      if (!mx_ends) jobs |= 4u;
    }
    if (row_y) {
      const unsigned em = s_ey[ty + 1], e0 = s_ey[ty + 2];
      flat_y = (em & e0) >> tx & 1u;
      need_yp = (em & e0 & s_ey[ty + 3]) != 0xffffffffu;
      if (need_yp || s_ey[ty] != 0xffffffffu) jobs |= 8u;
    }
    bool out_on = false, out_any = false;  // this lane's cell outside the tile counts, any of the warp's
    if (ty == kWarpX) {
      const int row = tx & (TY - 1), hi = tx / TY;
      out_on = hi < 2 && y0 + row < ny && !s_ex[row];
      out_any = __any_sync(0xffffffffu, out_on);
    } else if (ty == kWarpY0) {
      out_on = out_any = (s_ey[0] & s_ey[1] & s_ey[2]) != 0xffffffffu;
    } else if (ty == kWarpY1) {
      out_on = out_any = y0 + TY <= ny && (s_ey[TY] & s_ey[TY + 1] & s_ey[TY + 2]) != 0xffffffffu;
    }
    int so_out;  // the axis stride of its neighbours, and its slot
    const int c_out = outside_slot<TY>(ty, tx, out_on, so_out);
    if (out_any) jobs |= 16u;
    if (mode == kResidual && row_in && (jobs & 14u) == 0) {
      // no face state will test this cell: its state must be admissible (the stages of a step
      // test it in the wave-speed sum of the last one)
      R e, c2;
      by_material<MT>(id0, [&](auto T, auto m) {
        const R rho = q[cslot];
        if (!eos_e_c2<R, GEN, decltype(T)::value>(eos(m), rho, rrcp<R>(rho), q[4 * PL + cslot], e, c2)) bad = true;
      });
    }

    // ---- face states
    FaceState<R> QyP;
    R Fxp[5] = {(R)0, (R)0, (R)0, (R)0, (R)0};
#pragma unroll 1
    for (; jobs; jobs &= jobs - 1) {
      const int j = __ffs(jobs) - 1;
      R Pm[5], P[5], Pp[5];
      int ic;
      bool same;
      if (j <= 1) {
#pragma unroll
        for (int v = 0; v < 5; ++v) {
          Pm[v] = q[v * PL + cslot];
          P[v] = j ? qn[v * PL] : Pm[v];
          Pp[v] = j ? P2[v] : Pm[v];
        }
        ic = j ? id1 : id0;
        same = !j || (id0 == id1 && id2 == id1);
      } else {
        const int c0 = j == 4 ? c_out : cslot, so = j == 4 ? so_out : (j == 2 ? 1 : HX);
#pragma unroll
        for (int v = 0; v < 5; ++v) {
          Pm[v] = q[v * PL + c0 - so];
          P[v] = q[v * PL + c0];
          Pp[v] = q[v * PL + c0 + so];
        }
        ic = idp[c0];
        same = idp[c0 - so] == ic && idp[c0 + so] == ic;
      }
      FaceState<R> QM, QP;
      bool b = false;
      material_faces<GEN, MT, R>(eos, ic, Pm, P, Pp, same, QM, QP, b, lim, alpha);
      bad = bad || (b && (j < 4 || out_on));
      if (j <= 1) {
        if (j == 1) {
          R F[5];
          if (id0 == id1) {
            num_flux<2, R, GEN>(get_state(s_qz + tid, NT), QM, F, flx);
          } else {
#pragma unroll
            for (int v = 0; v < 5; ++v) F[v] = (R)0;
          }
#pragma unroll
          for (int v = 0; v < 5; ++v) fz[v * NT] = F[v];
        }
        put_state(s_qz + tid, NT, QP);
      } else if (j == 2) {
        // the states of the tile's first and last cell go to the warp that makes the fluxes
        // through the tile's x faces
        if (tx == 0) put_state(s_xe + TY + ty, SXE, QM);
        if (tx == TX - 1) put_state(s_xe + 2 * TY + ty, SXE, QP);
        FaceState<R> QR;
        QR.rho = __shfl_down_sync(0xffffffffu, QM.rho, 1);
        QR.u = __shfl_down_sync(0xffffffffu, QM.u, 1);
        QR.v = __shfl_down_sync(0xffffffffu, QM.v, 1);
        QR.w = __shfl_down_sync(0xffffffffu, QM.w, 1);
        QR.p = __shfl_down_sync(0xffffffffu, QM.p, 1);
        QR.c = __shfl_down_sync(0xffffffffu, QM.c, 1);
        QR.E = __shfl_down_sync(0xffffffffu, QM.E, 1);
        if (!(iff & 1)) num_flux<0, R, GEN>(QP, QR, Fxp, flx);
      } else if (j == 3) {
        put_state(s_ym + ty * TX + tx, SYM, QM);
        QyP = QP;
      } else if (ty == kWarpX) {
        if (out_on) {
          const int row = tx & (TY - 1);
          if (tx < TY) put_state(s_xe + row, SXE, QP);
          else put_state(s_xe + 3 * TY + row, SXE, QM);
        }
      } else if (ty == kWarpY0) {
        put_state(s_yp + tx, TX, QP);
      } else {
        put_state(s_ym + TY * TX + tx, SYM, QM);
      }
    }
    __syncthreads();

    // ---- y fluxes, the fluxes through the tile's x faces and its lower y face, the level-set residual
    R Lphi = (R)0;
    if (row_in) {
      if (need_yp) {
        R F[5];
        if (!(iff & 2)) {
          num_flux<1, R, GEN>(QyP, get_state(s_ym + (ty + 1) * TX + tx, SYM), F, flx);
        } else {
#pragma unroll
          for (int v = 0; v < 5; ++v) F[v] = (R)0;
        }
#pragma unroll
        for (int v = 0; v < 5; ++v) s_yf[v * SYM + (ty + 1) * TX + tx] = F[v];
      }
      // level-set residual -((u phi_x + v phi_y) + w phi_z), third-order upwind-biased (Sec. 4.4)
      const R u = q[PL + cslot], vv = q[2 * PL + cslot], w = q[3 * PL + cslot];
      const R* prow = phip + cslot;
      // the four values upwind of the cell, mirrored for a negative velocity (FP32: roundings written out)
      auto deriv = [&](R vel, R m2, R m1, R c, R p1, R p2) {
        if constexpr (sizeof(R) == 4) {
          return nonneg(vel) ? __fmul_rn(__fadd_rn(__fmaf_rn(-6.0f, m1, __fmaf_rn(2.0f, p1, __fmul_rn(3.0f, c))), m2), i6h)
                             : __fmul_rn(__fmaf_rn(-2.0f, m1, __fmaf_rn(-3.0f, c, __fmaf_rn(6.0f, p1, -p2))), i6h);
        } else {
          return nonneg(vel) ? ((((R)2 * p1 + (R)3 * c) - (R)6 * m1) + m2) * i6h
                             : (((-p2 + (R)6 * p1) - (R)3 * c) - (R)2 * m1) * i6h;
        }
      };
      const R Dx = deriv(u, prow[-2], prow[-1], prow[0], prow[1], prow[2]);
      const R Dy = deriv(vv, prow[-2 * HX], prow[-HX], prow[0], prow[HX], prow[2 * HX]);
      R Dz = deriv(w, ph[0], ph[1], ph[2], ph[3], ph[4]);
      if constexpr (sizeof(R) == 4 && !GEN && MT == 0) {
        // (two stiffened gases: the rounding order of this sum along z that their kernel always had)
        if (nonneg(w))
          Dz = __fmul_rn(__fadd_rn(__fmaf_rn(-6.0f, ph[1], __fmaf_rn(3.0f, ph[2], __fmul_rn(2.0f, ph[3]))), ph[0]), i6h);
      }
      if constexpr (sizeof(R) == 4) Lphi = -__fmaf_rn(w, Dz, __fmaf_rn(u, Dx, __fmul_rn(vv, Dy)));
      else Lphi = -((u * Dx + vv * Dy) + w * Dz);
      if constexpr (GEN) {
        // narrow band (Sec. 4.4): the velocity scaled by the cutoff of the cell's level set
        if (G.band_gamma > 0.0) Lphi = band_cutoff<R>((R)G.band_beta, (R)G.band_gamma, ph[2]) * Lphi;
      }
    }
    if (ty == kWarpX) {
      if (out_on) {
        const int row = tx & (TY - 1), hi = tx / TY;
        R F[5] = {(R)0, (R)0, (R)0, (R)0, (R)0};
        const int c0 = (row + 2) * HX + (hi ? TX + 1 : 1);
        if (idp[c0] == idp[c0 + 1])
          num_flux<0, R, GEN>(get_state(s_xe + 2 * hi * TY + row, SXE), get_state(s_xe + (2 * hi + 1) * TY + row, SXE),
                              F, flx);
#pragma unroll
        for (int v = 0; v < 5; ++v) s_xf[(2 * v + hi) * TY + row] = F[v];
      }
    } else if (ty == kWarpY0) {
      if (out_any) {
        R F[5] = {(R)0, (R)0, (R)0, (R)0, (R)0};
        const int c0 = HX + tx + 2;
        if (idp[c0] == idp[c0 + HX]) num_flux<1, R, GEN>(get_state(s_yp + tx, TX), get_state(s_ym + tx, SYM), F, flx);
#pragma unroll
        for (int v = 0; v < 5; ++v) s_yf[v * SYM + tx] = F[v];
      }
    }
    if (k + 1 < k1) look_at(buf ^ 1);
    R P0[5];  // (general kernel: the geometric source)
    if constexpr (GEN) {
#pragma unroll
      for (int v = 0; v < 5; ++v) P0[v] = q[v * PL + cslot];
    }
    __syncthreads();

    // ---- per cell: residual, Runge-Kutta update, work lists
    if (row_in) {
      const bool is_if = inside && iff != 0;
      // fluxes of the axes along which the cell is not uniform (the others' differences vanish)
      R res[5];
      R Fxm[5], Fym[5], Fyp[5], Fzm[5], Fzp[5];
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        Fxm[v] = __shfl_up_sync(0xffffffffu, Fxp[v], 1);
        if (tx == 0) Fxm[v] = s_xf[2 * v * TY + ty];
        if (tx == TX - 1) Fxp[v] = s_xf[(2 * v + 1) * TY + ty];
        const R* yf = s_yf + v * SYM + ty * TX + tx;
        Fxm[v] = flat_x ? (R)0 : Fxm[v];
        Fxp[v] = flat_x ? (R)0 : Fxp[v];
        Fym[v] = flat_y ? (R)0 : yf[0];
        Fyp[v] = flat_y ? (R)0 : yf[TX];
        Fzm[v] = flat_z0 ? (R)0 : fzm[v * NT];
        Fzp[v] = flat_z0 ? (R)0 : fz[v * NT];
        if constexpr (sizeof(R) == 4) {
          res[v] = __fmaf_rn(Fzm[v] - Fzp[v], ih, __fmaf_rn(Fxm[v] - Fxp[v], ih, __fmul_rn(Fym[v] - Fyp[v], ih)));
        } else {
          res[v] = ((Fxm[v] - Fxp[v]) * ih + (Fym[v] - Fyp[v]) * ih) + (Fzm[v] - Fzp[v]) * ih;
        }
      }
      // a row that changes nothing but its level set (plain copies below); for the last stage
      // its first-stage state must be the old one too
      const bool still = !GEN && __all_sync(0xffffffffu, flat_x && flat_y && flat_z0);

      const int c = pk + own_base;
      if constexpr (GEN) {
        // spherical / cylindrical forms (Sec. 3.4): S = -(alpha/r) u_r (rho, rho u, rho v,
        // rho w, rho E + p) at the cell centre r = x0 + (i + 1/2) h from the stage state,
        // added after the flux sum (interface cells get it in k_finish)
        if (G.geom != M2C_GEOM_CARTESIAN && inside && !is_if) {
          const double r = G.x0 + ((double)gx + 0.5) * G.h;
          const R a = to_r<R>((G.geom == M2C_GEOM_SPHERICAL ? 2.0 : 1.0) / r) * P0[1];
          R wv[5];
#pragma unroll
          for (int v = 0; v < 5; ++v) wv[v] = to_r<R>(gld(Ws + v * N + c));
#pragma unroll
          for (int v = 0; v < 4; ++v) res[v] = res[v] - a * wv[v];
          res[4] = res[4] - a * (wv[4] + P0[4]);
        }
      }
      bool flip = false;
      if (inside) {
        if (mode == kResidual) {
          if (!is_if) {
#pragma unroll
            for (int v = 0; v < 5; ++v) G.resR[v * N + c] = to_d<R>(res[v]);
          }
          G.resL[c] = to_d<R>(Lphi);
          G.id[c] = (uint8_t)id0;
        } else if (mode == kStage1) {
          gst(G.phi1 + c, fma(dt, to_d<R>(Lphi), gld(G.phi + c)));
          G.id[c] = (uint8_t)id0;
          if (!is_if) {
            if (still) {
#pragma unroll
              for (int v = 0; v < 5; ++v) gst(G.W1 + v * N + c, gld(G.W + v * N + c));
            } else {
#pragma unroll
              for (int v = 0; v < 5; ++v) gst(G.W1 + v * N + c, fma(dt, to_d<R>(res[v]), gld(G.W + v * N + c)));
            }
          }
        } else if (GEN && mode == kStage2of3) {
          // TVD RK3, second stage (Sec. 4.3): W2 = (3/4 W + 1/4 W1) + 1/4 dt R(W1)
          gst(G.phi2 + c, (0.75 * gld(G.phi + c) + 0.25 * gld(G.phi1 + c)) + 0.25 * dt * to_d<R>(Lphi));
          if (!is_if) {
#pragma unroll
            for (int v = 0; v < 5; ++v)
              gst(G.W2 + v * N + c,
                  (0.75 * gld(G.W + v * N + c) + 0.25 * gld(G.W1 + v * N + c)) + 0.25 * dt * to_d<R>(res[v]));
          }
        } else {
          // last stage: TVD RK2 W' = (W + (W1 + dt R(W1)))/2, or TVD RK3
          // W' = (1/3 W + 2/3 W2) + 2/3 dt R(W2). The mixed path's TVD RK2 takes
          // W' = (W + W1)/2 + (dt/2) R with the increment (dt/2) R in binary32 (R
          // itself is a binary32 result) and one rounding after the FP64 sum.
          const bool rk3 = GEN && mode == kStage3;
          constexpr bool f32inc = sizeof(R) == 4 && !GEN;
          const double pn = rk3      ? (gld(G.phi + c) / 3.0 + 2.0 / 3.0 * gld(G.phi2 + c)) +
                                      2.0 / 3.0 * dt * to_d<R>(Lphi)
                            : f32inc ? fma(0.5, gld(G.phi + c) + gld(G.phi1 + c), to_d<R>(hdt * Lphi))
                                     : 0.5 * (gld(G.phi + c) + (gld(G.phi1 + c) + dt * to_d<R>(Lphi)));
          gst(G.phi + c, pn);
          const bool neg = lt0(pn);
          flip = neg != (id0 == 1);
          // bit 2: material at the end of the step (read by the phase update)
          G.id[c] = (uint8_t)(id0 | (neg ? 4 : 0));
          if (!is_if) {
            double wn[5];
            bool kept = still;  // W1 = W: W' = W, and the stage state's wave speeds are the new state's
            if (still) {
#pragma unroll
              for (int v = 0; v < 5; ++v) {
                wn[v] = gld(G.W + v * N + c);
                kept = kept && same_bits(wn[v], gld(G.W1 + v * N + c));
              }
            }
            if (!kept) {
#pragma unroll
              for (int v = 0; v < 5; ++v) {
                wn[v] = rk3      ? (gld(G.W + v * N + c) / 3.0 + 2.0 / 3.0 * gld(G.W2 + v * N + c)) +
                                  2.0 / 3.0 * dt * to_d<R>(res[v])
                        : f32inc ? fma(0.5, gld(G.W + v * N + c) + gld(G.W1 + v * N + c), to_d<R>(hdt * res[v]))
                                 : 0.5 * (gld(G.W + v * N + c) + (gld(G.W1 + v * N + c) + dt * to_d<R>(res[v])));
                gst(G.W + v * N + c, wn[v]);
              }
            }
            if (!flip) {
              bool ok;
              R lam = (R)0;
              by_material<MT>(id0, [&](auto T, auto m) {
                // (FP32 MG: the wave speeds' p is not the stage state's to the last bit)
                if (kept && !(sizeof(R) == 4 && eos_is<decltype(T)::value>(eos(m), M2C_EOS_MG))) {
                  R P[5];
#pragma unroll
                  for (int v = 0; v < 5; ++v) P[v] = q[v * PL + cslot];
                  lam = wave_sum_p<R, GEN, decltype(T)::value>(G, eos(m), P, ok);
                } else {
                  lam = wave_sum_v<R, GEN, decltype(T)::value>(G, eos(m), eosd(m), wn, ok);
                }
              });
              bad = bad || !ok;
              lam_max = fmax(lam_max, lam);
            }
          }
        }
      }
      // ---- work lists: warp ballot, one atomic per warp (skipped when the warp has none)
      const bool fxf = inside && (iff & 1), fyf = inside && (iff & 2), fzf = inside && id1 != id0;
      const int nf = (int)fxf + (int)fyf + (int)fzf;
      if (__any_sync(0xffffffffu, is_if || nf || flip)) {
        {
          const unsigned m = __ballot_sync(0xffffffffu, is_if);
          if (m) {
            int base = 0;
            const int leader = __ffs(m) - 1;
            if ((int)lane == leader) base = atomicAdd(&ctrl->ncell[slot], __popc(m));
            base = __shfl_sync(0xffffffffu, base, leader);
            if (is_if) {
              const int s = base + __popc(m & lt);
              if (s < G.cell_cap) {
                IfCell* e = G.cells + s;
                e->cell = c;
#pragma unroll
                for (int v = 0; v < 5; ++v) {
                  e->F[0][v] = to_d<R>(Fxm[v]);
                  e->F[1][v] = to_d<R>(Fxp[v]);
                  e->F[2][v] = to_d<R>(Fym[v]);
                  e->F[3][v] = to_d<R>(Fyp[v]);
                  e->F[4][v] = to_d<R>(Fzm[v]);
                  e->F[5][v] = to_d<R>(Fzp[v]);
                }
                G.cell_slot[c] = s;
              } else {
                ovf = true;
              }
            }
          }
        }
        {
          int incl = nf;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if ((int)lane >= o) incl += y;
          }
          const int total = __shfl_sync(0xffffffffu, incl, 31);
          if (total) {
            int base = 0;
            if (lane == 31) base = atomicAdd(&ctrl->nface[slot], total);
            base = __shfl_sync(0xffffffffu, base, 31);
            int s = base + incl - nf;
            const bool fl[3] = {fxf, fyf, fzf};
#pragma unroll
            for (int d = 0; d < 3; ++d) {
              if (fl[d]) {
                if (s < G.face_cap) {
                  G.faces[s].cell = c;
                  G.faces[s].dir = d;
                } else {
                  ovf = true;
                }
                ++s;
              }
            }
          }
        }
        if (final_stage) {
          const unsigned m = __ballot_sync(0xffffffffu, flip);
          if (m) {
            int base = 0;
            const int leader = __ffs(m) - 1;
            if ((int)lane == leader) base = atomicAdd(&ctrl->nflip, __popc(m));
            base = __shfl_sync(0xffffffffu, base, leader);
            if (flip) {
              const int s = base + __popc(m & lt);
              if (s < G.flip_cap) G.flips[s] = c;
              else ovf = true;
            }
          }
        }
      }
    }

    // ---- shift the z window
#pragma unroll
    for (int v = 0; v < 5; ++v) P1[v] = P2[v];
    flat_z0 = flat_z1;
    rowflat_z0 = rowflat_z1;
    ph[0] = ph[1]; ph[1] = ph[2]; ph[2] = ph[3]; ph[3] = ph[4];
    idm = id0; id0 = id1; id1 = id2;
  }
  // failures are latched once per tile, with the thread's column at the tile's first plane
  if (bad) latch_error(ctrl, M2C_ENONPHYS, cell_of(G, gx, gy, k0));
  if (ovf) latch_error(ctrl, M2C_EOVERFLOW, cell_of(G, gx, gy, k0));
  if (final_stage) block_max_to(to_d<R>(lam_max), &ctrl->lam[(step + 1) & 1], s_red);
  __syncthreads();  // the next tile reuses the shared memory
  }
}

// The shared-memory opt-in is a per-device attribute of the kernel: it is set
// once on every device the calling threads make current.
template <typename R, int TY, bool GEN, int MT, bool ONE>
void stage_smem_setup() {
  static bool done[kMaxDevices] = {};
  const int dev = current_device();
  if (done[dev]) return;
  cudaFuncSetAttribute(k_stage<R, TY, GEN, MT, ONE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)StageSmem<R, TY>::bytes);
  done[dev] = true;
}

template <typename R, int TY, bool GEN, int MT, bool ONE>
cudaError_t launch_stage_k(const Grid* grids, const long long* tiles, int ngrid, long long ntiles, int mode,
                           const LaunchPlan& lp, cudaStream_t s) {
  stage_smem_setup<R, TY, GEN, MT, ONE>();  // (done by the context's set-up, outside captures)
  long long nb = ntiles;
  if (lp.blocks_per_sm > 0) nb = std::min<long long>(ntiles, (long long)lp.blocks_per_sm * sm_count());
  if (nb < 1) nb = 1;
  if (lp.sched == 1) {
    cudaError_t e = cudaMemsetAsync(lp.counter, 0, sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
  }
  StageArg<ONE> arg;
  if constexpr (ONE) arg.grid = *lp.one;
  k_stage<R, TY, GEN, MT, ONE><<<(unsigned)nb, 32 * TY, StageSmem<R, TY>::bytes, s>>>(arg, grids, tiles, ngrid, ntiles,
                                                                                    mode, lp.sched, lp.counter);
  return cudaGetLastError();
}

template <typename R, int TY, bool GEN, int MT = -1>
cudaError_t launch_stage_t(const Grid* grids, const long long* tiles, int ngrid, long long ntiles, int mode,
                           const LaunchPlan& lp, cudaStream_t s) {
  // (FP64: one kernel for grids alone and in batches, whose results are the same bits)
  if constexpr (sizeof(R) == 4 && !GEN && MT >= 0) {
    if (lp.one) return launch_stage_k<R, TY, GEN, MT, true>(grids, tiles, ngrid, ntiles, mode, lp, s);
  }
  return launch_stage_k<R, TY, GEN, MT, false>(grids, tiles, ngrid, ntiles, mode, lp, s);
}

template <typename R, int TY, bool GEN, int MT = -1>
void stage_smem_setup_t() {
  if constexpr (sizeof(R) == 4 && !GEN && MT >= 0) stage_smem_setup<R, TY, GEN, MT, true>();
  stage_smem_setup<R, TY, GEN, MT, false>();
}

// The launch for the material pair of the plan: instantiations with fixed EOS
// types for the four SG / MG pairs, else the run-time types.
template <typename R, int TY>
cudaError_t launch_stage_pair(const Grid* grids, const long long* tiles, int ngrid, long long ntiles, int mode,
                              const LaunchPlan& lp, cudaStream_t s) {
  switch (lp.mats) {
    case M2C_EOS_SG + 4 * M2C_EOS_SG:
      return launch_stage_t<R, TY, false, M2C_EOS_SG + 4 * M2C_EOS_SG>(grids, tiles, ngrid, ntiles, mode, lp, s);
    case M2C_EOS_MG + 4 * M2C_EOS_SG:
      return launch_stage_t<R, TY, false, M2C_EOS_MG + 4 * M2C_EOS_SG>(grids, tiles, ngrid, ntiles, mode, lp, s);
    case M2C_EOS_SG + 4 * M2C_EOS_MG:
      return launch_stage_t<R, TY, false, M2C_EOS_SG + 4 * M2C_EOS_MG>(grids, tiles, ngrid, ntiles, mode, lp, s);
    case M2C_EOS_MG + 4 * M2C_EOS_MG:
      return launch_stage_t<R, TY, false, M2C_EOS_MG + 4 * M2C_EOS_MG>(grids, tiles, ngrid, ntiles, mode, lp, s);
    default:
      return launch_stage_t<R, TY, false>(grids, tiles, ngrid, ntiles, mode, lp, s);
  }
}

template <typename R, int TY>
void stage_smem_setup_pairs() {
  stage_smem_setup_t<R, TY, false, M2C_EOS_SG + 4 * M2C_EOS_SG>();
  stage_smem_setup_t<R, TY, false, M2C_EOS_MG + 4 * M2C_EOS_SG>();
  stage_smem_setup_t<R, TY, false, M2C_EOS_SG + 4 * M2C_EOS_MG>();
  stage_smem_setup_t<R, TY, false, M2C_EOS_MG + 4 * M2C_EOS_MG>();
  stage_smem_setup_t<R, TY, false>();
}

}  // namespace m2c

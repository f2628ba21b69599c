// lbcad_march.cuh -- the hybrid step as two kernels that march up z through shared-memory tiles.
//
//   k_march_fields (a1-a4): per site the stencils of Q and psi, H, mu and the stress sigma, and
//     with the lagged Euler step also the whole update of Q and the flux divergence of psi; leaves
//     sigma, mu, the divergence and psi in a scratch of 12 values per site (six arrays of pairs);
//   k_march_lb (a3, a5, a4 of psi, a6): the force F = div sigma and lap mu from that scratch, the pull of
//     the populations, the collision, psi, and the conserved sums.
//
// A block owns a TX x TY column of the lattice and marches up z.  The stencils run as carries
// (FieldsCarry, ForceCarry, LapCarry): a new plane's nine points finish the site of the plane
// below and leave their share of the next, so a plane is read from shared memory once per stencil
// and nothing is computed twice.  Planes arrive by cp.async one plane ahead, one barrier per
// plane.  The stress never has to be known on a halo of the tile in shared memory, which is what
// the split buys: one kernel for the whole step computes sigma on 1.38 sites per output site (tile
// halo, partly filled warps), opens every run of planes with three sigma planes and no output,
// and holds both halves' registers.  The scratch costs 2 x 48 bytes per site of traffic in FP32.
//
// Measured (FP32 with the a6 sums, one kernel for the step -> this file): 64^3 52 -> 34.0 us a step, 128^3 234 -> 193,
// 256^3 1640 -> 1360; the FP64 step is twice as fast.  At 128^3 k_march_fields takes 85 us, bound by instruction
// issue at 12 warps an SM (its stencils' registers) with the shared-memory pipe busy most of that time;
// k_march_lb 104 us, 216 bytes a site at two thirds of the copy rate.  FP64 is bound by the FP64 pipe.
//
// The grid is persistent: blocks take work items (a tile column over a slab of planes) in turn, and one
// launch covers up to kPackMany instances of a batch.
//
// The end of the file holds the order-parameter half of the sync-coupled and Heun steps, as tiled
// z-marching kernels on the same tiles and work split.
#pragma once

#include <type_traits>

#include "lbcad_kernels.cuh"

namespace lbcad {

// Periodic plane index for p in [-n, 2n): the planes a work item touches lie in
// [-1, nz + 1] and every edge is >= 4, so one add or subtract suffices (no division).
__device__ __forceinline__ int wrap_plane(int p, int n) { return p < 0 ? p + n : (p >= n ? p - n : p); }

__device__ __forceinline__ int wrapmod(int v, int n) {
  v %= n;
  return v < 0 ? v + n : v;
}

template <typename T>
__device__ __forceinline__ Vec2<T> lds2(const T* p) {
  if constexpr (sizeof(T) == 4) {
    const float2 v = *reinterpret_cast<const float2*>(p);
    return Vec2<T>{v.x, v.y};
  } else {
    const double2 v = *reinterpret_cast<const double2*>(p);
    return Vec2<T>{v.x, v.y};
  }
}

// An aligned pair from global memory through the read-only path.
template <typename T>
__device__ __forceinline__ Vec2<T> ldg2(const T* p) {
  if constexpr (sizeof(T) == 4) {
    const float2 v = __ldg(reinterpret_cast<const float2*>(p));
    return Vec2<T>{v.x, v.y};
  } else {
    const double2 v = __ldg(reinterpret_cast<const double2*>(p));
    return Vec2<T>{v.x, v.y};
  }
}

// A store of an output value to global memory, cached in L2 only: the next kernel reads it
// back through L2, and the loads of this one keep L1 to themselves.
template <typename T>
__device__ __forceinline__ void st_out(T* p, T v) {
  __stcg(p, v);
}
template <typename T>
__device__ __forceinline__ void st_pair(T* p, T a, T b) {
  if constexpr (sizeof(T) == 4) __stcg(reinterpret_cast<float2*>(p), make_float2(a, b));
  else __stcg(reinterpret_cast<double2*>(p), make_double2(a, b));
}

__device__ __forceinline__ void cp_async4(void* smem_dst, const void* gsrc) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async8(void* smem_dst, const void* gsrc) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gsrc) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_commit_wait_all() {
  asm volatile("cp.async.commit_group;\ncp.async.wait_all;\n" ::: "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
// Waits until at most the N latest groups are still on their way.
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }
template <typename T>
__device__ __forceinline__ void cp_async_elem(T* dst, const T* src) {
  if constexpr (sizeof(T) == 4) cp_async4(dst, src); else cp_async8(dst, src);
}
// Component i of a field of n sites from a pointer into component 0: one wide multiply-add (a table of component
// pointers in the launch's arguments costs a constant load each, through the same queue as the shared-memory
// accesses).
template <typename T>
__device__ __forceinline__ T* comp(T* p, int i, unsigned n) {
  return reinterpret_cast<T*>(reinterpret_cast<uintptr_t>(p) + (unsigned long long)n * (unsigned)(i * (int)sizeof(T)));
}

// Pair s of an array of pairs.
template <typename T>
__device__ __forceinline__ T* pair_at(T* base, unsigned s) {
  struct alignas(2 * sizeof(T)) P { T v[2]; };
  return reinterpret_cast<T*>(reinterpret_cast<P*>(base) + s);
}
template <typename T>
__device__ __forceinline__ void cp_async_pair(T* dst, const T* src) {
  if constexpr (sizeof(T) == 4) cp_async8(dst, src); else cp_async16(dst, src);
}

// Programmatic dependent launch (MarchWork::early): every kernel of a step lets the next one start its blocks
// when its own have all come to their last item, and waits for the kernels before it to finish, memory
// included, before it touches anything they write or read.  So a kernel's start-up runs under the tail
// of the one before.
__device__ __forceinline__ void let_next_kernel_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_previous_kernels() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// A TX x TY tile with a halo of 1, and the sites of it each thread loads.
template <int TX_, int TY_>
struct Tile {
  static constexpr int TX = TX_, TY = TY_, NT = TX * TY;
  static constexpr int SW = TX + 2, SH = TY + 2, SP = SW * SH;
  static constexpr int LD = (SP + NT - 1) / NT;
};

// Shared-memory planes of a tile.  Q and psi: the field pairs (Q_xx, Q_xy), (Q_xz, Q_yy), (Q_yz, psi), pair j
// of site k at elements 2 (j SP + k).  Velocity: (u_x, u_y) of site k at 2 k, u_z at 2 SP + k.
template <int SP>
__device__ __forceinline__ int qidx(int f, int k) {
  return (f >> 1) * 2 * SP + 2 * k + (f & 1);
}

// Neighbour reads of one tile site: Q/psi pairs and velocity.
template <typename T, class G>
struct TileAcc {
  const T* qpl[3];
  const T* upl[3];
  int sc;
  __device__ __forceinline__ int at(int cx, int cy) const { return sc + cy * G::SW + cx; }
  __device__ __forceinline__ Vec2<T> pair(int j, int cx, int cy, int cz) const {
    return lds2(qpl[cz + 1] + 2 * (j * G::SP + at(cx, cy)));
  }
  __device__ __forceinline__ T psi(int cx, int cy, int cz) const { return qpl[cz + 1][qidx<G::SP>(5, at(cx, cy))]; }
  // pair j at the neighbour below or above the site along axis a
  __device__ __forceinline__ Vec2<T> pair_upwind(int j, int a, bool from_below) const {
    const T* pl = a == 2 ? (from_below ? qpl[0] : qpl[2]) : qpl[1];
    const int d = a == 2 ? 0 : (a == 0 ? 1 : G::SW);
    return lds2(pl + 2 * (j * G::SP + (from_below ? sc - d : sc + d)));
  }
  __device__ __forceinline__ Vel3<T> u3(int cx, int cy, int cz) const {
    const int k = at(cx, cy);
    return Vel3<T>{lds2(upl[cz + 1] + 2 * k), upl[cz + 1][2 * G::SP + k]};
  }
};

// Global offsets are unsigned site numbers (a box has at most 2^31 sites) added to a field's base pointer: the
// 64-bit address is one multiply-add of the offset and a base that depends on the launch's arguments only.
// In-plane offsets of this thread's load sites of a tile:
template <class G>
__device__ __forceinline__ void tile_offsets(const MarchItem& tl, int nx, int ny, unsigned off[G::LD]) {
#pragma unroll
  for (int r = 0; r < G::LD; ++r) {
    const int k = (int)threadIdx.x + r * G::NT;
    off[r] = k < G::SP ? (unsigned)(wrapmod(tl.y0 + k / G::SW - 1, ny) * nx + wrapmod(tl.x0 + k % G::SW - 1, nx)) : 0u;
  }
}

// The scratch plane of lattice plane z (in [0, nz)): plane I.sz0 comes first (see MarchDesc).
template <typename T>
__device__ __forceinline__ int scratch_plane(const MarchDesc<T>& I, int z) {
  const int k = z - I.sz0;
  return k < 0 ? k + I.nz : k;
}

// Resident blocks per SM a kernel is built for, given its threads and the registers a thread wants.
__host__ __device__ constexpr int blocks_for(int threads, int regs) {
  return 65536 / (threads * regs) > 0 ? 65536 / (threads * regs) : 1;
}

// ---------------------------------------------------------------- fields
constexpr int kMarchOp = 0, kMarchH = 1, kMarchPred = 2;

template <typename T, class G, int MODE>
struct FieldsSmem {
  static constexpr int NSLOT = 4;  // planes p-2 (faces below), p-1, p, and the arriving one
  static constexpr int QSL = 6 * G::SP, USL = MODE == kMarchOp ? 3 * G::SP : 0;
  static constexpr size_t bytes = (size_t)NSLOT * (QSL + USL) * sizeof(T);
};

// kMarchOp: sigma, mu, the flux divergence and psi of every site into the scratch pairs and the new Q
// (Euler with the velocity of the previous step).  kMarchH: sigma and mu into the pairs, H into its
// scratch (sync coupling, Heun).  kMarchPred: H and mu of the Heun predicted state qp into Hp.
template <typename T, int MI, int TX, int TY, int MODE>
__global__ void __launch_bounds__(TX * TY, sizeof(T) == 4 ? blocks_for(TX * TY, TX * TY > 128 ? 128 : 168) : 1)
    k_march_fields(const __grid_constant__ InstPack<T, MI> P, const MarchItem* __restrict__ items, int nitems) {
  constexpr bool OP = MODE == kMarchOp, WH = MODE == kMarchH;
  using G = Tile<TX, TY>;
  using M = FieldsSmem<T, G, MODE>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* sQ = reinterpret_cast<T*>(smem_raw);
  T* sU = sQ + M::NSLOT * M::QSL;
  const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
  bool waited = false;
  for (int item = blockIdx.x; item < nitems; item += gridDim.x) {
    const MarchItem tl = items[item];
    const int zb = tl.zb, ze = tl.ze;
    const MarchDesc<T>& I = P.d[MI == 1 ? 0 : tl.inst];
    const int nx = I.nx, ny = I.ny, nz = I.nz;
    const unsigned plane = I.plane;
    const Coef<T>& cf = I.c;
    unsigned off[G::LD];
    tile_offsets<G>(tl, nx, ny, off);
    auto issue = [&](int p) {
      const unsigned gz = (unsigned)wrap_plane(p, nz) * plane;
      T* dq = sQ + ((p + 4) & 3) * M::QSL;
#pragma unroll
      for (int r = 0; r < G::LD; ++r) {
        const int k = tid + r * G::NT;
        if (k < G::SP) {
          const unsigned o = gz + off[r];
#pragma unroll
          for (int f = 0; f < 5; ++f) cp_async_elem(dq + qidx<G::SP>(f, k), (MODE == kMarchPred ? I.qp[f] : I.q_in[f]) + o);
          cp_async_elem(dq + qidx<G::SP>(5, k), (MODE == kMarchPred ? I.qp[5] : I.psi_in) + o);
          if constexpr (OP) {
            T* du = sU + ((p + 4) & 3) * M::USL;
#pragma unroll
            for (int a = 0; a < 3; ++a) cp_async_elem(du + (a < 2 ? 2 * k + a : 2 * G::SP + k), I.u_in[a] + o);
          }
        }
      }
    };
    if (!waited) wait_for_previous_kernels();
    waited = true;
    if (item + (int)gridDim.x >= nitems) let_next_kernel_start();
    __syncthreads();  // the previous item is done with the tiles
    issue(zb - 1);
    issue(zb);
    issue(zb + 1);
    cp_async_commit_wait_all();
    __syncthreads();
    const bool inside = tl.x0 + tx < nx && tl.y0 + ty < ny;
    const int sc = (ty + 1) * G::SW + (tx + 1);
    const unsigned soff = (unsigned)((tl.y0 + ty) * nx + (tl.x0 + tx));
    FieldsCarry<T> car;
#pragma unroll 1
    for (int p = zb - 1; p <= ze; ++p) {
      if (p > zb && p < ze) issue(p + 1);
      if (inside) {
        T q0[5], p0, dq[3][5], lapq[5], dp[3], lapp, hp[6];
        const T* np = sQ + ((p + 4) & 3) * M::QSL;
        car.advance([&](int j, int cx, int cy) { return lds2(np + 2 * (j * G::SP + sc + cy * G::SW + cx)); }, q0, p0, dq,
                    lapq, dp, lapp, hp);
        if (p > zb) {
          const int z = p - 1;
          const unsigned s = (unsigned)z * plane + soff;
          T H[5], sig[9], mu;
          local_fields<T>(cf, q0, p0, dq, lapq, dp, lapp, hp, H, mu, sig);
          if constexpr (MODE == kMarchPred) {
#pragma unroll
            for (int k = 0; k < 5; ++k) st_out(I.Hp[k] + s, H[k]);
            st_out(I.Hp[5] + s, mu);
          } else {
            const unsigned ss = (unsigned)scratch_plane(I, z) * plane + soff;
#pragma unroll
            for (int j = 0; j < 4; ++j) st_pair(pair_at(I.S[j], ss), sig[pair_c0(j)], sig[pair_c1(j)]);
            st_pair(pair_at(I.S[4], ss), sig[8], mu);
            T div = T(0);
            if constexpr (OP) {
              TileAcc<T, G> acc;
              acc.sc = sc;
#pragma unroll
              for (int j = 0; j < 3; ++j) {
                acc.qpl[j] = sQ + ((z + 3 + j) & 3) * M::QSL;
                acc.upl[j] = sU + ((z + 3 + j) & 3) * M::USL;
              }
              T Wg[3][3], u0[3], uf[6], pf[6], inc[5];
              Vec2<T> qu[3][3];
              gather_velocity<T>(acc, Wg, u0, uf);
              gather_upwind<T>(acc, u0, qu, pf);
              q_increment<T>(cf, Wg, q0, qu, u0, H, inc);
#pragma unroll
              for (int k = 0; k < 5; ++k) st_out(I.q_out[k] + s, q0[k] + inc[k]);
              div = flux_divergence(p0, pf, u0, uf);
            }
            if constexpr (WH) {
#pragma unroll
              for (int k = 0; k < 5; ++k) st_out(I.H[k] + s, H[k]);
            }
            if constexpr (OP) st_pair(pair_at(I.S[5], ss), div, p0);
          }
        }
      }
      if (p > zb) {
        cp_async_commit_wait_all();
        __syncthreads();
      }
    }
  }
}

// ---------------------------------------------------------------- LB
// Copies the populations g_i(x - c_i) of velocity set V to this thread's places in shared memory (population i
// at i STRIDE): zo, pyo and pxo hold the offsets of the planes z-1, z, z+1, the rows y-1, y, y+1 and the
// columns x-1, x, x+1.
template <typename T, class V, int STRIDE>
__device__ __forceinline__ void pull_populations(const MarchDesc<T>& I, const unsigned zo[3], const unsigned pyo[3],
                                                 const unsigned pxo[3], T* dst) {
#pragma unroll
  for (int i = 0; i < V::Q; ++i) {
    const unsigned o = zo[1 - V::c(i, 2)] + pyo[1 - V::c(i, 1)] + pxo[1 - V::c(i, 0)];
    cp_async_elem(dst + i * STRIDE, comp(I.g_in[0], i, I.N) + o);
  }
}

// The scratch pairs of one plane in shared memory (pair j of tile site k at 2 (j SP + k)): the stress pairs (sig_pair) with
// mu in pair 4, and pair 5 = (flux divergence, psi).  As pairs, a warp's read of one takes two wavefronts; read
// from quads it took four.
template <typename T, class G>
struct PairPlane {
  const T* pl;
  int sc;
  __device__ __forceinline__ Vec2<T> spair(int j, int cx, int cy) const {
    return lds2(pl + 2 * (j * G::SP + sc + cy * G::SW + cx));
  }
  // component c (= 3a + b) of the stress
  __device__ __forceinline__ T comp(int c, int cx, int cy) const {
    const Vec2<T> v = spair(sig_pair(c), cx, cy);
    return sig_lane(c) ? v.y : v.x;
  }
  // the antisymmetric part sigma^A = (sigma - sigma^T)/2 (the force of the Eq. 9-11 form)
  __device__ __forceinline__ T anti(int c, int cx, int cy) const {
    const int r = c / 3, k = c - 3 * r;
    if (r == k) return T(0);
    return mul_rn(T(0.5), sub2(comp(c, cx, cy), comp(3 * k + r, cx, cy)));
  }
  __device__ __forceinline__ Vec2<T> apair(int j, int cx, int cy) const {
    if (j == 4) return Vec2<T>{T(0), T(0)};
    return Vec2<T>{anti(pair_c0(j), cx, cy), anti(pair_c1(j), cx, cy)};
  }
};

// The a6 sums within a block.  Each thread adds its sites' twelve shares in T: FP64 arithmetic is
// slow on this part.  In FP32 the additions are error-free (two_sum_add): every sum is kept as
// an unevaluated pair (s, c) whose exact value is s + c, each addition split into its rounded
// result and its exact rounding error, the errors gathered in c.  The pair carries about twice
// FP32's precision (the only loss is the rounding of c itself, second order in the unit
// roundoff), and FP64 takes over at the end of each run of items as (double)s + (double)c.  So
// the sums of the FP32 state come out as its FP64 sums, up to the FP32 rounding of each site's own
// share.
template <typename T>
struct ObsAcc {
  Vec2<T> s[6], c[6];  // values 2q, 2q+1
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int q = 0; q < 6; ++q) s[q] = c[q] = v2(T(0), T(0));
  }
  __device__ __forceinline__ void add(const T v[12]) {
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      const Vec2<T> x{v[2 * q], v[2 * q + 1]};
      if constexpr (sizeof(T) == 4) {  // two_sum_add on two lanes
        const Vec2<T> t = add2(s[q], x), bp = sub2(t, s[q]);
        c[q] = add2(c[q], add2(sub2(s[q], sub2(t, bp)), sub2(x, bp)));
        s[q] = t;
      } else {
        s[q] = add2(s[q], x);
      }
    }
  }
};

// red[k + 12 m] (k < 12, m < M) summed over m into red[k] by a fixed pairing tree (all threads;
// barriers between the levels).  FP64 additions are long-latency on this part, so the sums run
// as trees of depth log2(M) rather than as chains of length M; the order is fixed, so the
// result does not depend on timing.
__device__ __forceinline__ void obs_tree12(double* red, int M) {
  for (int len = M; len > 1;) {
    const int half = (len + 1) >> 1;
    for (int t = threadIdx.x; t < 12 * (len - half); t += blockDim.x) red[t] += red[t + 12 * half];
    __syncthreads();
    len = half;
  }
}

// End of the kernel (all threads): the block counts each of its runs' slots on the run's instance; the block
// whose count completes an instance sums that instance's slots into ob.latest: each of the
// twelve values over fixed strided subsets of the slots, sixteen loads of a thread in flight together and added
// pairwise (an FP64 addition takes 64 cycles here, so a chain over the slots took longer than the loads), then over the
// subsets by a fixed tree, so the result does not depend on which block finishes last.
// No spin waits.  red: shared scratch of at least 12 * (blockDim.x / 12) doubles.
// mass0(inst) = N rho0 with shifted populations, else 0.  ONE: the launch holds one instance, so every block has one
// slot and the slot maps need not be read (each read is a trip to L2 on the critical path of a small box).
template <bool ONE, class MS>
__device__ __forceinline__ void obs_block_end(const FusedObs& ob, int nrun, double* red, const MS& mass0) {
  __shared__ int last;
  const int tid = threadIdx.x;
  if (tid < 12) __threadfence();  // the slot stores of this block's runs, before the counting
  __syncthreads();
  for (int j = 0; j < nrun; ++j) {
    const int inst = ONE ? 0 : ob.slot_inst[blockIdx.x * ob.maxrun + j];
    if (tid == 0) last = atomicAdd(&ob.cnt[inst], 1u) == (ONE ? (unsigned)ob.total : (unsigned)ob.nslot[inst]) - 1u;
    __syncthreads();
    if (last) {
      __threadfence();
      const int per = blockDim.x / 12;
      const int lo = ONE ? 0 : ob.slot_lo[inst], hi = ONE ? ob.total : ob.slot_hi[inst];
      if (tid < 12 * per) {
        const int k = tid % 12, l = tid / 12;
        double v = 0.0;
        for (int s0 = lo + l; s0 < hi; s0 += 16 * per) {
          double x[16];
#pragma unroll
          for (int e = 0; e < 16; ++e) {
            const int sl = s0 + e * per;
            x[e] = sl < hi && (ONE || __ldg(ob.slot_inst + sl) == inst) ? __ldcg(ob.slots + sl * 12 + k) : 0.0;
          }
#pragma unroll
          for (int h = 8; h > 0; h >>= 1)
#pragma unroll
            for (int e = 0; e < h; ++e) x[e] += x[e + h];
          v += x[0];
        }
        red[l * 12 + k] = v;
      }
      __syncthreads();
      obs_tree12(red, per);
      if (tid < 12) ob.latest[inst * 12 + tid] = red[tid] + (tid == 0 ? mass0(inst) : 0.0);
      if (tid == 0) ob.cnt[inst] = 0u;
    }
    __syncthreads();
  }
}

// End of a run: the block's twelve FP64 sums from its threads' accumulators to the run's
// slot, through shared memory (the plane ring, free by then).  Thread t adds value t % 12 of a
// fixed strided subset of the threads, then the subsets are added by a fixed tree.
template <typename T, int NT>
struct ObsReduce {
  static constexpr int STR = NT + 1, SUB = NT / 12;
  static constexpr size_t dred_off = ((size_t)24 * STR * sizeof(T) + 15) / 16 * 16;
  static constexpr size_t bytes = dred_off + (size_t)12 * SUB * sizeof(double);
  __device__ __forceinline__ static void run(const ObsAcc<T>& a, unsigned char* smem, const FusedObs& ob, int slot) {
    T* red = reinterpret_cast<T*>(smem);
    double* dred = reinterpret_cast<double*>(smem + dred_off);
    const int tid = threadIdx.x;
    __syncthreads();  // the ring is free
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      red[2 * q * STR + tid] = a.s[q].x;
      red[(2 * q + 1) * STR + tid] = a.s[q].y;
      if constexpr (sizeof(T) == 4) {
        red[(12 + 2 * q) * STR + tid] = a.c[q].x;
        red[(13 + 2 * q) * STR + tid] = a.c[q].y;
      }
    }
    __syncthreads();
    if (tid < 12 * SUB) {
      const int k = tid % 12;
      T s = T(0), c = T(0);
#pragma unroll 4
      for (int e = tid / 12; e < NT; e += SUB) {
        two_sum_add(s, c, red[k * STR + e]);
        if constexpr (sizeof(T) == 4) c += red[(12 + k) * STR + e];
      }
      dred[tid] = (double)s + (double)c;
    }
    __syncthreads();
    obs_tree12(dred, SUB);
    if (tid < 12) ob.slots[slot * 12 + tid] = dred[tid];
    __syncthreads();
  }
};

template <typename T, class G, int Q, int MODE>
struct LbSmem {
  static constexpr int NSLOT = 3;  // planes p-1, p and the arriving one
  static constexpr int NP = MODE == kFusedLbOnly ? 5 : 6;  // without psi and its divergence
  static constexpr int SL = 2 * NP * G::SP;
  static constexpr size_t ring = (size_t)NSLOT * SL * sizeof(T);
  static constexpr int PULL = Q * G::NT;  // pulled populations of one plane; two planes
  static constexpr size_t bytes = ring + (size_t)2 * PULL * sizeof(T);
  static_assert(MODE != kFusedSums || ring >= ObsReduce<T, G::NT>::bytes, "the ring is the scratch of the a6 sums");
};

// FORM 0: F = div sigma, BGK + Guo (Eqs. 6-8).  FORM 1: FA = div sigma^A and the equilibrium carrying
// sigma^S (Eqs. 9-11).  MODE kFusedPlain: with the update of psi; kFusedSums: and the a6 sums;
// kFusedLbOnly: populations and velocity only (sync coupling, Heun).
template <typename T, bool SHIFT, int MI, int TX, int TY, class V, int FORM, int MODE>
__global__ void __launch_bounds__(TX * TY, sizeof(T) == 4 ? blocks_for(TX * TY, 128) : 1)
    k_march_lb(const __grid_constant__ InstPack<T, MI> P, const MarchItem* __restrict__ items, int nitems, FusedObs ob) {
  constexpr bool OBS = MODE == kFusedSums;
  using G = Tile<TX, TY>;
  using M = LbSmem<T, G, V::Q, MODE>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* sS = reinterpret_cast<T*>(smem_raw);
  const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
  bool waited = false;
  ObsAcc<T> sums;
  int run = 0, run_inst = -1;
  if constexpr (OBS) sums.clear();
  for (int item = blockIdx.x; item < nitems; item += gridDim.x) {
    const MarchItem tl = items[item];
    const int zb = tl.zb, ze = tl.ze;
    const MarchDesc<T>& I = P.d[MI == 1 ? 0 : tl.inst];
    if constexpr (OBS && MI > 1) {
      if (run_inst >= 0 && tl.inst != run_inst) {
        ObsReduce<T, G::NT>::run(sums, smem_raw, ob, ob.slot0 + blockIdx.x * ob.maxrun + run);
        sums.clear();
        ++run;
      }
      run_inst = tl.inst;
    }
    const int nx = I.nx, ny = I.ny, nz = I.nz;
    const unsigned plane = I.plane;
    const Coef<T>& cf = I.c;
    unsigned off[G::LD];
    tile_offsets<G>(tl, nx, ny, off);
    auto slot = [&](int p) { return sS + ((p + 3) % 3) * M::SL; };
    auto issue = [&](int p) {
      const unsigned gz = (unsigned)scratch_plane(I, wrap_plane(p, nz)) * plane;
      T* d = slot(p);
#pragma unroll
      for (int r = 0; r < G::LD; ++r) {
        const int k = tid + r * G::NT;
        if (k < G::SP) {
          const unsigned o = gz + off[r];
#pragma unroll
          for (int j = 0; j < M::NP; ++j) cp_async_pair(d + 2 * (j * G::SP + k), pair_at(I.S[j], o));
        }
      }
    };
    const int x = tl.x0 + tx, y = tl.y0 + ty;
    const bool inside = x < nx && y < ny;
    const int sc = (ty + 1) * G::SW + (tx + 1);
    const unsigned soff = (unsigned)(y * nx + x);
    const unsigned pxo[3] = {(unsigned)(x ? x - 1 : nx - 1), (unsigned)x, (unsigned)(x + 1 < nx ? x + 1 : 0)};
    const unsigned pyo[3] = {(unsigned)((y ? y - 1 : ny - 1) * nx), (unsigned)(y * nx),
                             (unsigned)((y + 1 < ny ? y + 1 : 0) * nx)};
    // the pulled populations of a plane are copied to each thread's own places while the plane before is worked
    // on, and waited for just before they are used, not with the planes at the barrier
    T* const pulled = sS + M::NSLOT * M::SL + tid;
    auto pull = [&](int z) {
      const unsigned zo[3] = {(unsigned)wrap_plane(z - 1, nz) * plane, (unsigned)z * plane,
                              (unsigned)wrap_plane(z + 1, nz) * plane};
      pull_populations<T, V, G::NT>(I, zo, pyo, pxo, pulled + (z & 1) * M::PULL);
    };
    if (!waited) wait_for_previous_kernels();
    waited = true;
    if (item + (int)gridDim.x >= nitems) let_next_kernel_start();
    __syncthreads();  // the previous item is done with the tiles
    issue(zb - 1);
    issue(zb);
    issue(zb + 1);
    cp_async_commit();
    if (inside) pull(zb);
    cp_async_commit();
    cp_async_wait<1>();
    Vec2<T> trx = v2(T(0), T(0)), trY = v2(T(0), T(0));
    if constexpr (OBS) {
      if (inside) {
        trx = ldg2(I.trig + 2 * x);
        trY = ldg2(I.trig + 2 * (nx + y));
      }
    }
    __syncthreads();
    ForceCarry<T> force;
    LapCarry<T> lapm;
#pragma unroll 1
    for (int p = zb - 1; p <= ze; ++p) {
      if (p > zb && p < ze) issue(p + 1);
      cp_async_commit();
      if (inside) {
        const int z = p - 1;
        Vec2<T> trz = v2(T(0), T(0));
        if (OBS && p > zb) trz = ldg2(I.trig + 2 * (nx + ny + z));
        T F[3], lapmu = T(0);
        const PairPlane<T, G> np{slot(p), sc};
        if constexpr (FORM == 0) force.advance([&](int j, int cx, int cy) { return np.spair(j, cx, cy); }, F);
        else force.advance([&](int j, int cx, int cy) { return np.apair(j, cx, cy); }, F);
        if constexpr (MODE != kFusedLbOnly) lapmu = lapm.advance([&](int cx, int cy) { return np.spair(4, cx, cy).y; });
        if (p > zb) {
          const PairPlane<T, G> cp{slot(z), sc};
          T g[V::Q], u[3], mom[4];
          cp_async_wait<1>();  // the populations of plane z; the scratch of plane p + 1 may still be arriving
#pragma unroll
          for (int i = 0; i < V::Q; ++i) g[i] = pulled[(z & 1) * M::PULL + i * G::NT];
          if (p < ze) pull(p);
          cp_async_commit();
          if constexpr (FORM == 0) {
            lb_collide<T, SHIFT, V>(cf, F, g, u, OBS ? mom : nullptr);
          } else {
            T sg[9];
#pragma unroll
            for (int c = 0; c < 9; ++c) sg[c] = cp.comp(c, 0, 0);
            lb_collide_stress<T, SHIFT, V>(cf, F, sg, g, u, OBS ? mom : nullptr);
          }
          const unsigned s = (unsigned)z * plane + soff;
          T* const go = I.g_out[0] + s;
          T* const uo = I.u_out[0] + s;
#pragma unroll
          for (int i = 0; i < V::Q; ++i) st_out(comp(go, i, I.N), g[i]);
#pragma unroll
          for (int a = 0; a < 3; ++a) st_out(comp(uo, a, I.N), u[a]);
          if constexpr (MODE == kFusedForce) {
#pragma unroll
            for (int a = 0; a < 3; ++a) st_out(I.F[a] + s, F[a]);
          }
          if constexpr (MODE != kFusedLbOnly) {
            const Vec2<T> dp = cp.spair(5, 0, 0);  // flux divergence, psi
            const T pn = dp.y + fma(cf.M, lapmu, -dp.x);
            st_out(I.psi_out + s, pn);
            if constexpr (OBS) {
              // mass, psi and momentum of the new state, and phi_c with its centroid moments
              const T pc = T(0.5) * (T(1) + pn);
              const T v[12] = {mom[0], pn, mom[1], mom[2], mom[3], mul_rn(pc, trx.x), mul_rn(pc, trY.x),
                               mul_rn(pc, trz.x), mul_rn(pc, trx.y), mul_rn(pc, trY.y), mul_rn(pc, trz.y), pc};
              sums.add(v);
            }
          }
        }
      }
      // the next issue overwrites plane p-1: from p = zb on, every warp is done with it first
      if (p >= zb) {
        if (p > zb && inside) cp_async_wait<1>();  // the scratch of plane p + 1; the populations of plane p may still be arriving
        else cp_async_wait<0>();
        __syncthreads();
      }
    }
    cp_async_wait<0>();
  }
  if constexpr (OBS) {
    ObsReduce<T, G::NT>::run(sums, smem_raw, ob, ob.slot0 + blockIdx.x * ob.maxrun + run);
    obs_block_end<MI == 1>(ob, run + 1, reinterpret_cast<double*>(smem_raw), [&](int inst) { return P.d[MI == 1 ? 0 : inst].mass0; });
  }
}

// ---------------------------------------------------------------- tiled order-parameter half
// The order-parameter half of a sync-coupled or Heun step (after step_lb), as z-marching kernels on the
// tiles and work split of the step: rings of planes with a halo of 1 in shared memory, filled by
// cp.async one plane ahead, one barrier per plane, and the shared per-site functions on them.
//   k_op_tiled<STAGE>: STAGE 0 the update Q + R(Q) (Euler, sync), 1 the Heun predictor
//     (rq = R(Q), qp = Q + rq), 2 the Heun corrector Q + (rq + R(qp))/2, R from gather_op and
//     op_update with u of this step (sync) or of the previous one, H and mu of the scratch
//     (k_march_fields: kMarchH at t, kMarchPred at the predicted state).
// Ring slots: planes z-1 .. z+2 (the last one arriving).  The values a site reads only at
// itself (H, and in the corrector R(Q) at t and Q, psi at t) arrive the same way, one plane
// ahead, into two slots by plane parity: read from global memory after the stencils, their
// latency stood between the update and the plane barrier.
// lap mu is carried up the planes (nine reads a plane instead of nineteen): 96^3 sync 59.6 -> 58.7 us a step,
// 128^3 Heun 365 -> 361.
template <typename T, class G>
struct OpSmem {
  static constexpr int NSLOT = 4;
  static constexpr int QSLOT = 6 * G::SP, USLOT = 3 * G::SP, MSLOT = G::SP;
  __host__ __device__ static constexpr int NSITE(int stage) { return stage == 2 ? 17 : 5; }  // H, rq, Q, psi
  static constexpr size_t site_off = ((size_t)NSLOT * (QSLOT + USLOT + MSLOT) * sizeof(T) + 15) / 16 * 16;
  __host__ __device__ static constexpr size_t bytes(int stage) {
    return site_off + (size_t)2 * NSITE(stage) * G::NT * sizeof(T);
  }
};

template <typename T, int MI, int TX, int TY, int STAGE>
__global__ void __launch_bounds__(TX * TY, sizeof(T) == 8 ? 2 : blocks_for(TX * TY, 128))
    k_op_tiled(const __grid_constant__ InstPack<T, MI> P, const MarchItem* __restrict__ items, int nitems, int sync) {
  using G = Tile<TX, TY>;
  using M = OpSmem<T, G>;
  constexpr int NSV = M::NSITE(STAGE);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* sQ = reinterpret_cast<T*>(smem_raw);
  T* sU = sQ + M::NSLOT * M::QSLOT;
  T* sM = sU + M::NSLOT * M::USLOT;
  T* sI = reinterpret_cast<T*>(smem_raw + M::site_off);  // site-local values [2][NSV][NT]
  const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
  bool waited = false;
  for (int item = blockIdx.x; item < nitems; item += gridDim.x) {
    const MarchItem tl = items[item];
    const int zb = tl.zb, ze = tl.ze;
    const MarchDesc<T>& I = P.d[MI == 1 ? 0 : tl.inst];
    const int nx = I.nx, ny = I.ny, nz = I.nz;
    const unsigned plane = I.plane;
    const T* const* const us = sync ? I.u_out : I.u_in;
    // mu: planar at the predicted state (corrector), lane 1 of scratch pair 4 otherwise
    const T* msrc = STAGE == 2 ? I.Hp[5] : I.S[4] + 1;
    constexpr int MST = STAGE == 2 ? 1 : 2;
    unsigned off[G::LD];
    tile_offsets<G>(tl, nx, ny, off);
    auto issue = [&](int p) {
      const unsigned gz = (unsigned)wrap_plane(p, nz) * plane;
      const int sl = (p + 4) & 3;
#pragma unroll
      for (int r = 0; r < G::LD; ++r) {
        const int k = tid + r * G::NT;
        if (k < G::SP) {
          const unsigned gs = gz + off[r];
          T* dq = sQ + sl * M::QSLOT;
#pragma unroll
          for (int f = 0; f < 5; ++f) cp_async_elem(dq + qidx<G::SP>(f, k), (STAGE == 2 ? I.qp[f] : I.q_in[f]) + gs);
          cp_async_elem(dq + qidx<G::SP>(5, k), (STAGE == 2 ? I.qp[5] : I.psi_in) + gs);
          T* du = sU + sl * M::USLOT;
#pragma unroll
          for (int a = 0; a < 3; ++a) cp_async_elem(du + (a < 2 ? 2 * k + a : 2 * G::SP + k), us[a] + gs);
          cp_async_elem(sM + sl * M::MSLOT + k, msrc + (size_t)MST * gs);
        }
      }
    };
    const bool inside = tl.x0 + tx < nx && tl.y0 + ty < ny;
    const unsigned soff = (unsigned)((tl.y0 + ty) * nx + (tl.x0 + tx));
    auto issue_site = [&](int p) {
      if (!inside) return;
      const unsigned gs = (unsigned)p * plane + soff;
      T* d = sI + (p & 1) * NSV * G::NT + tid;
#pragma unroll
      for (int k = 0; k < 5; ++k) cp_async_elem(d + k * G::NT, (STAGE == 2 ? I.Hp[k] : I.H[k]) + gs);
      if constexpr (STAGE == 2) {
#pragma unroll
        for (int k = 0; k < 6; ++k) cp_async_elem(d + (5 + k) * G::NT, I.rq[k] + gs);
#pragma unroll
        for (int k = 0; k < 5; ++k) cp_async_elem(d + (11 + k) * G::NT, I.q_in[k] + gs);
        cp_async_elem(d + 16 * G::NT, I.psi_in + gs);
      }
    };
    if (!waited) wait_for_previous_kernels();
    waited = true;
    if (item + (int)gridDim.x >= nitems) let_next_kernel_start();
    __syncthreads();  // the previous item is done with the tiles
    issue(zb - 1);
    issue(zb);
    issue(zb + 1);
    issue_site(zb);
    cp_async_commit_wait_all();
    __syncthreads();
    const int sc = (ty + 1) * G::SW + (tx + 1);
    LapCarry<T> lapm;
    auto lap_mu = [&](int p) {
      const T* m = sM + ((p + 4) & 3) * M::MSLOT + sc;
      return lapm.advance([&](int cx, int cy) { return m[cy * G::SW + cx]; });
    };
    if (inside) {
      lap_mu(zb - 1);
      lap_mu(zb);
    }
#pragma unroll 1
    for (int z = zb; z < ze; ++z) {
      issue(z + 2);
      if (z + 1 < ze) issue_site(z + 1);
      if (inside) {
        const T* si = sI + (z & 1) * NSV * G::NT + tid;
        TileAcc<T, G> acc;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          const int sl = (z + 3 + j) & 3;
          acc.qpl[j] = sQ + sl * M::QSLOT;
          acc.upl[j] = sU + sl * M::USLOT;
        }
        acc.sc = sc;
        const T lapmu = lap_mu(z + 1);
        T Wg[3][3], q0[5], p0, pf[6], u0[3], uf[6];
        Vec2<T> qu[3][3];
        gather_advection<T>(acc, Wg, q0, qu, p0, pf, u0, uf);
        const unsigned s = (unsigned)z * plane + soff;
        T Hs[5];
#pragma unroll
        for (int k = 0; k < 5; ++k) Hs[k] = si[k * G::NT];
        T qn[5], pn;
        op_update<T, STAGE != 0>(I.c, lapmu, Wg, q0, qu, p0, pf, u0, uf, Hs, qn, pn);
        if constexpr (STAGE == 0) {
#pragma unroll
          for (int k = 0; k < 5; ++k) st_out(I.q_out[k] + s, qn[k]);
          st_out(I.psi_out + s, pn);
        } else if constexpr (STAGE == 1) {
#pragma unroll
          for (int k = 0; k < 5; ++k) {
            I.rq[k][s] = qn[k];
            I.qp[k][s] = q0[k] + qn[k];
          }
          I.rq[5][s] = pn;
          I.qp[5][s] = p0 + pn;
        } else {
#pragma unroll
          for (int k = 0; k < 5; ++k)
            st_out(I.q_out[k] + s, si[(11 + k) * G::NT] + T(0.5) * (si[(5 + k) * G::NT] + qn[k]));
          st_out(I.psi_out + s, si[16 * G::NT] + T(0.5) * (si[10 * G::NT] + pn));
        }
      }
      cp_async_commit_wait_all();
      __syncthreads();
    }
  }
}

// ---------------------------------------------------------------- launchers
// Allows a kernel `smem` bytes of dynamic shared memory and adds its blocks per SM (an attribute of the
// function on the current device, idempotent).
template <class K>
cudaError_t prepare_kernel(K kernel, int threads, size_t smem, int* per_sm) {
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, kernel, threads, smem);
}

// One tile shape of one variant (velocity set V, LB form FORM): FX x FY for the fields kernels, LX x LY for the others.
template <typename T, bool SHIFT, class V, int FORM, int FX, int FY, int LX, int LY>
struct MarchShape {
  using FG = Tile<FX, FY>;
  using G = Tile<LX, LY>;
  using OS = OpSmem<T, G>;
  static constexpr bool kDefaultLb = std::is_same<V, VelD3Q19>::value && FORM == 0;
  template <int MODE>
  static constexpr size_t fields_smem() { return FieldsSmem<T, FG, MODE>::bytes; }
  template <int MODE>
  static constexpr size_t lb_smem() { return LbSmem<T, G, V::Q, MODE>::bytes; }

  template <int MI>
  static cudaError_t prepare_mi(bool split, bool heun, FusedCfg* c) {
    cudaError_t e;
    if (!split) {
      // both LB kernels run on the grid of the one with the sums (the a6 slots are laid out for it)
      int plain = 0;
      e = prepare_kernel(k_march_fields<T, MI, FX, FY, kMarchOp>, FG::NT, fields_smem<kMarchOp>(), &c->fields_per_sm);
      if (e == cudaSuccess)
        e = prepare_kernel(k_march_lb<T, SHIFT, MI, LX, LY, V, FORM, kFusedPlain>, G::NT, lb_smem<kFusedPlain>(), &plain);
      if (e == cudaSuccess)
        e = prepare_kernel(k_march_lb<T, SHIFT, MI, LX, LY, V, FORM, kFusedSums>, G::NT, lb_smem<kFusedSums>(),
                           &c->lb_per_sm);
      return e;
    }
    e = prepare_kernel(k_march_fields<T, MI, FX, FY, kMarchH>, FG::NT, fields_smem<kMarchH>(), &c->fields_per_sm);
    if (e == cudaSuccess)
      e = prepare_kernel(k_march_lb<T, SHIFT, MI, LX, LY, V, FORM, kFusedLbOnly>, G::NT, lb_smem<kFusedLbOnly>(),
                         &c->lb_per_sm);
    if (!heun) {
      if (e == cudaSuccess) e = prepare_kernel(k_op_tiled<T, MI, LX, LY, 0>, G::NT, OS::bytes(0), &c->op_per_sm[0]);
      return e;
    }
    if (e == cudaSuccess) e = prepare_kernel(k_op_tiled<T, MI, LX, LY, 1>, G::NT, OS::bytes(1), &c->op_per_sm[0]);
    if (e == cudaSuccess)
      e = prepare_kernel(k_march_fields<T, MI, FX, FY, kMarchPred>, FG::NT, fields_smem<kMarchPred>(), &c->pred_per_sm);
    if (e == cudaSuccess) e = prepare_kernel(k_op_tiled<T, MI, LX, LY, 2>, G::NT, OS::bytes(2), &c->op_per_sm[1]);
    return e;
  }
  static cudaError_t prepare(bool many, bool split, bool heun, FusedCfg* c) {
    c->fx = FX;
    c->fy = FY;
    c->lx = LX;
    c->ly = LY;
    const cudaError_t e = prepare_mi<1>(split, heun, c);  // (a batch can leave one instance for its last launch)
    return many && e == cudaSuccess ? prepare_mi<kPackMany>(split, heun, c) : e;
  }

  template <class... P, class... A>
  static void launch(void (*kernel)(P...), const MarchWork& w, int threads, size_t smem, cudaStream_t s, const A&... args) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)w.grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = w.early ? 1 : 0;
    (void)cudaLaunchKernelEx(&cfg, kernel, P(args)...);  // the caller reads the error
  }
  template <int MI, int MODE>
  static void fields(const InstPack<T, MI>& P, const MarchWork& w, cudaStream_t s) {
    launch(k_march_fields<T, MI, FX, FY, MODE>, w, FG::NT, fields_smem<MODE>(), s, P, w.items, w.nitems);
  }
  template <int MI, int MODE>
  static void lb(const InstPack<T, MI>& P, const MarchWork& w, const FusedObs& ob, cudaStream_t s) {
    launch(k_march_lb<T, SHIFT, MI, LX, LY, V, FORM, MODE>, w, G::NT, lb_smem<MODE>(), s, P, w.items, w.nitems, ob);
  }
  template <int MI, int STAGE>
  static void op(const InstPack<T, MI>& P, const MarchWork& w, bool sync, cudaStream_t s) {
    launch(k_op_tiled<T, MI, LX, LY, STAGE>, w, G::NT, OS::bytes(STAGE), s, P, w.items, w.nitems, sync ? 1 : 0);
  }

  template <int MI>
  static InstPack<T, MI> pack(const StepWork& w, const MarchDesc<T>* d) {
    InstPack<T, MI> P{};
    for (int i = 0; i < w.ninst && i < MI; ++i) {
      P.d[i] = d[i];
      P.d[i].sz0 = w.sz0;
    }
    return P;
  }
  template <int MI>
  static cudaError_t step_mi(const StepWork& w, const MarchDesc<T>* d, const FusedObs& ob, bool obs, cudaStream_t s) {
    const InstPack<T, MI> P = pack<MI>(w, d);
    fields<MI, kMarchOp>(P, w.fields, s);
    if (obs) lb<MI, kFusedSums>(P, w.lb, ob, s);
    else lb<MI, kFusedPlain>(P, w.lb, ob, s);
    return cudaGetLastError();
  }
  static cudaError_t step(const StepWork& w, const MarchDesc<T>* d, const FusedObs& ob, bool obs, cudaStream_t s) {
    return w.ninst > 1 ? step_mi<kPackMany>(w, d, ob, obs, s) : step_mi<1>(w, d, ob, obs, s);
  }
  template <int MI>
  static cudaError_t split_mi(const StepWork& w, bool heun, bool sync, const MarchDesc<T>* d, cudaStream_t s) {
    const InstPack<T, MI> P = pack<MI>(w, d);
    fields<MI, kMarchH>(P, w.fields, s);
    lb<MI, kFusedLbOnly>(P, w.lb, FusedObs{}, s);
    if (!heun) {
      op<MI, 0>(P, w.op[0], sync, s);
      return cudaGetLastError();
    }
    op<MI, 1>(P, w.op[0], sync, s);
    fields<MI, kMarchPred>(P, w.pred, s);
    op<MI, 2>(P, w.op[1], sync, s);
    return cudaGetLastError();
  }
  // One replayed step of the adjoint: the Euler step without the sums, leaving its force too.
  static cudaError_t prepare_replay() {
    int n = 0;
    return prepare_kernel(k_march_lb<T, SHIFT, 1, LX, LY, V, FORM, kFusedForce>, G::NT, lb_smem<kFusedForce>(), &n);
  }
  static cudaError_t replay(const StepWork& w, const MarchDesc<T>* d, cudaStream_t s) {
    const InstPack<T, 1> P = pack<1>(w, d);
    fields<1, kMarchOp>(P, w.fields, s);
    lb<1, kFusedForce>(P, w.lb, FusedObs{}, s);
    return cudaGetLastError();
  }
  static cudaError_t split(const StepWork& w, bool heun, bool sync, const MarchDesc<T>* d, cudaStream_t s) {
    return w.ninst > 1 ? split_mi<kPackMany>(w, heun, sync, d, s) : split_mi<1>(w, heun, sync, d, s);
  }
};

// Tile shapes: f(shape) for candidate k of variant (V, FORM).  0 and 3 come for every variant,
// the others in FP32 for the Euler step of D3Q19 with the body force; FP64 has 0 only.
template <typename T, bool SHIFT, class V, int FORM, class F>
cudaError_t with_shape(int k, bool split, const F& f) {
  if (k < 0 || k >= LaunchFused<T, SHIFT>::num_configs()) return cudaErrorInvalidValue;
  if constexpr (sizeof(T) == 8) {
    if (k == 0) return f(MarchShape<T, SHIFT, V, FORM, 32, 8, 32, 8>{});
  } else {
    if (k == 0) return f(MarchShape<T, SHIFT, V, FORM, 32, 4, 32, 8>{});
    if (k == 3) return f(MarchShape<T, SHIFT, V, FORM, 16, 8, 16, 16>{});
    if constexpr (std::is_same<V, VelD3Q19>::value && FORM == 0) {
      if (split) return cudaErrorNotSupported;
      if (k == 1) return f(MarchShape<T, SHIFT, V, FORM, 32, 4, 32, 4>{});
      if (k == 2) return f(MarchShape<T, SHIFT, V, FORM, 64, 2, 64, 4>{});
      if (k == 4) return f(MarchShape<T, SHIFT, V, FORM, 32, 8, 32, 8>{});
      if (k == 5) return f(MarchShape<T, SHIFT, V, FORM, 16, 8, 16, 8>{});
      if (k == 6) return f(MarchShape<T, SHIFT, V, FORM, 8, 8, 8, 8>{});
    }
  }
  return cudaErrorNotSupported;
}

// variant = (velocity set D3Q15 ? 1 : 0) + 2 * (Eq. 9-11 form ? 1 : 0)
template <typename T, bool SHIFT, class F>
cudaError_t with_variant(int variant, int k, bool split, const F& f) {
  switch (variant) {
    case 0: return with_shape<T, SHIFT, VelD3Q19, 0>(k, split, f);
    case 1: return with_shape<T, SHIFT, VelD3Q15, 0>(k, split, f);
    case 2: return with_shape<T, SHIFT, VelD3Q19, 1>(k, split, f);
    case 3: return with_shape<T, SHIFT, VelD3Q15, 1>(k, split, f);
  }
  return cudaErrorInvalidValue;
}

template <typename T, bool SHIFT>
int LaunchFused<T, SHIFT>::num_configs() {
  return sizeof(T) == 4 ? 7 : 1;
}

template <typename T, bool SHIFT>
cudaError_t LaunchFused<T, SHIFT>::prepare(int variant, int k, bool many, bool split, bool heun, FusedCfg* cfg) {
  return with_variant<T, SHIFT>(variant, k, split, [&](auto sh) { return decltype(sh)::prepare(many, split, heun, cfg); });
}

template <typename T, bool SHIFT>
cudaError_t LaunchFused<T, SHIFT>::step(int variant, int k, const StepWork& w, const MarchDesc<T>* d, const FusedObs& ob,
                                        bool obs, cudaStream_t s) {
  return with_variant<T, SHIFT>(variant, k, false, [&](auto sh) { return decltype(sh)::step(w, d, ob, obs, s); });
}

// (The adjoint differentiates the Euler step of D3Q19 with the body force: variant 0.)
template <typename T, bool SHIFT>
cudaError_t LaunchFused<T, SHIFT>::prepare_replay(int k) {
  return with_variant<T, SHIFT>(0, k, false, [&](auto sh) {
    if constexpr (decltype(sh)::kDefaultLb) return decltype(sh)::prepare_replay();
    else return cudaErrorNotSupported;
  });
}

template <typename T, bool SHIFT>
cudaError_t LaunchFused<T, SHIFT>::replay(int k, const StepWork& w, const MarchDesc<T>* d, cudaStream_t s) {
  return with_variant<T, SHIFT>(0, k, false, [&](auto sh) {
    if constexpr (decltype(sh)::kDefaultLb) return decltype(sh)::replay(w, d, s);
    else return cudaErrorNotSupported;
  });
}

template <typename T, bool SHIFT>
cudaError_t LaunchFused<T, SHIFT>::split_step(int variant, int k, const StepWork& w, bool heun, bool sync,
                                              const MarchDesc<T>* d, cudaStream_t s) {
  return with_variant<T, SHIFT>(variant, k, true, [&](auto sh) { return decltype(sh)::split(w, heun, sync, d, s); });
}

}  // namespace lbcad

// hs_common.cuh -- device-side building blocks shared by the libhsolve kernels:
// the stencil descriptor, deterministic block reductions, and the bounded
// grid "reduce-barrier" used by the persistent solver kernels.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace hs {

// ---------------------------------------------------------------------------
// Debug builds (-DHS_DEBUG): every global index the tile engines compute is
// checked against the vector length before it is used; a bad index is
// recorded (1 + index, first one wins) in a word of this translation unit and
// the access is skipped -- no trap, no assert, the kernel runs on.  The host
// launchers read and clear the word after each solve (hs_dbg_take) and return
// HS_ERR_BOUNDS.  In release builds HS_IN_BOUNDS is constant true.
// ---------------------------------------------------------------------------
#ifdef HS_DEBUG
static __device__ unsigned long long hs_dbg_word;
__device__ __forceinline__ bool hs_in_bounds(long long idx, long long n) {
  if (idx >= 0 && idx < n) return true;
  atomicCAS(&hs_dbg_word, 0ull, 1ull + (unsigned long long)idx);
  return false;
}
#define HS_IN_BOUNDS(idx, n) hs_in_bounds((long long)(idx), (long long)(n))
#else
#define HS_IN_BOUNDS(idx, n) true
#endif

// Operator kinds as compiled into kernels.
// OP_BOX27: the HPCG 27-point system (diagonal 27, -1 on the 26 neighbours of
// the 3x3x3 box), applied through separable box sums (3-D only).
// FP64 only, applied through a neighbour sum on the integer pipes (hs_fx.cuh):
// OP_ISO, an OP_SYM operator with one coupling for all neighbours (equal
// spacings, or HPCG's 7-point matrix); OP_WSYM and OP_WNON, OP_SYM and
// OP_NONSYM operators whose couplings lie within a factor of 64.
enum OpKind : int { OP_SYM = 0, OP_NONSYM = 1, OP_VARK = 2, OP_BOX27 = 3, OP_ISO = 4, OP_WSYM = 5, OP_WNON = 6 };
__host__ __device__ constexpr bool fx_op(int opk) { return opk >= OP_ISO; }

// Device status word values (mirrors hs_status where they overlap).
enum DevStatus : int {
  DS_RUNNING = 0,
  DS_CONVERGED = 1,
  DS_MAXIT = 2,
  DS_BREAKDOWN = -3,
  DS_NONFINITE = -4,
  DS_TIMEOUT = -5,
};

// Stencil coefficients.  A row reads
//   y_i = d c + xl W + xu E + yl S + yu N + zl B + zu T
// (W/E = i -+ 1, S/N = j -+ 1, B/T = k -+ 1, out-of-grid values are zero).
// OP_SYM keeps xl == xu etc. so that pairs can be summed first.  OP_VARK
// reads per-cell coefficients: D[i] on the diagonal and the lower-face
// couplings ax/ay/az (positive), the upper faces taken from the neighbour's
// lower face:  y_i = D_i c - ax_i W - ax_{i+1} E - ay_i S - ay_{i+nx} N
//                         - az_i B - az_{i+nx ny} T.
//
// FxW: the couplings of an OP_WSYM / OP_WNON operator relative to the upper x
// one, in the order xl, xu, yl, yu, zl, zu: as doubles w, and as fixed-point
// significand and exponent, w = c 2^(x - 60), 2^60 <= c < 2^61 in limbs of 31
// bits (ch, cl); rc = the rounding constant of a product (see fx_scale).
struct FxW {
  double w[6];
  int ch[6], cl[6];
  unsigned rc[6];
  int x[6];
};

template <typename T>
struct CoefFx {};
template <>
struct CoefFx<double> {
  FxW fx;
};

template <typename T>
struct Coef : CoefFx<T> {
  T d, xl, xu, yl, yu, zl, zu;
  const T* D;
  const T* ax;
  const T* ay;
  const T* az;
};

struct Geom {
  int nx, ny, nz;      // nz = 1 for 2-D, ny = nz = 1 for 1-D
  long long N;
  long long plane;     // nx * ny
};

// ---------------------------------------------------------------------------
// Exact binary32 -> binary64 widening with integer operations.  On this GPU
// the F2F.F64.F32 conversion instruction issues on the FP64 pipe (measured at
// about the FP64 FMA rate), so the FP64-accumulated dot products of FP32
// vectors build the binary64 bit pattern from the binary32 fields instead:
// exponent rebiased by 1023 - 127 = 896, fraction shifted left by 29.  Normal
// numbers, zeros, infinities and NaNs are widened exactly; binary32
// subnormals (magnitude below 2^-126) are flushed to zero.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double widen(double d) { return d; }
__device__ __forceinline__ double widen(float f) {
  const unsigned u = __float_as_uint(f), a = u & 0x7fffffffu;
  unsigned hi = (a >> 3) + 0x38000000u;
  if (a >= 0x7f800000u) hi += 0x38000000u;   // infinity, NaN
  const bool none = a < 0x00800000u;         // zero, subnormal
  hi = none ? 0u : hi;
  const unsigned lo = none ? 0u : u << 29;
  return __hiloint2double((int)(hi | (u & 0x80000000u)), (int)lo);
}

// ---------------------------------------------------------------------------
// Deterministic reductions.  Every sum below is taken in a fixed order that
// depends only on the launch shape, never on timing, so repeated solves give
// bit-identical scalars.
// ---------------------------------------------------------------------------

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Block-wide sums of NS values; result valid in every thread.  `sh` must hold
// at least 32 * NS doubles.  Contains __syncthreads(): call from all threads.
template <int NS>
__device__ __forceinline__ void block_sum(double (&v)[NS], double* sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nwarp = (blockDim.x + 31) >> 5;
#pragma unroll
  for (int s = 0; s < NS; s++) v[s] = warp_sum(v[s]);
  __syncthreads();
  if (lane == 0) {
#pragma unroll
    for (int s = 0; s < NS; s++) sh[s * 32 + warp] = v[s];
  }
  __syncthreads();
#pragma unroll
  for (int s = 0; s < NS; s++) {
    double t = (lane < nwarp) ? sh[s * 32 + lane] : 0.0;
    v[s] = warp_sum(t);
  }
  __syncthreads();
}

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void red_release(unsigned* p, unsigned v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned atom_acq_rel(unsigned* p, unsigned v) {
  unsigned r;
  asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(r) : "l"(p), "r"(v) : "memory");
  return r;
}
__device__ __forceinline__ void st_release(unsigned* p, unsigned v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void st_relaxed(unsigned* p, unsigned v) {
  asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ int ld_acquire_int(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Control block at the start of every solver workspace (zeroed by the host
// before each solve).
struct Ctrl {
  unsigned count;        // arrivals at the team's barriers (only grows; LastTeam: at this one)
  unsigned gen;          // barrier generation (LastTeam, BiTeam)
  int status;            // DevStatus
  int iters;             // iterations completed
  int restarts;          // BiCGStab restarts
  int pad0;
  unsigned long long timeout_ns;
  double scal[16];       // reduced scalars of the last barrier (LastTeam, BiTeam)
  double rel_res;        // last relative residual
  double aux[7];
};

static_assert(sizeof(Ctrl) <= 512, "Ctrl must fit its 512-byte slot");

// A team is the set of blocks that solve one system together: rank and size
// within the team, and the team's own control block and partial-sum slots.
// A standalone solve uses the whole grid as one team; the batched solver runs
// many teams (one per large system, single-block teams for small ones) in
// one cooperative launch.  A shared word of the block counts the grid team's
// barriers since its control block was initialised (a register a thread would
// cost the FP32 kernels a block per SM).
constexpr int RED_MAX = 3;                 // scalars per reduction
constexpr int RED_SLOTS = 2 * RED_MAX;     // partial sums per block (two barriers' worth)

struct Team {
  int rank;
  int size;
  Ctrl* ctrl;
  double* partials;   // RED_SLOTS * size doubles (LastTeam: NS * size)
  __device__ __forceinline__ long long tid() const { return (long long)rank * blockDim.x + threadIdx.x; }
  __device__ __forceinline__ long long stride() const { return (long long)size * blockDim.x; }
  __device__ __forceinline__ bool lead() const { return rank == 0 && threadIdx.x == 0; }
};

__device__ __forceinline__ unsigned& team_epoch() {
  __shared__ unsigned epoch;
  return epoch;
}
// Before the first barrier of a grid team; the block barriers of a
// reduction's block_sum come in between.
__device__ __forceinline__ void team_begin() {
  if (threadIdx.x == 0) team_epoch() = 0u;
}

// Team reduce-barrier.  Every block of the team contributes NS partial sums
// (block-reduced, valid in every thread) and arrives on a counter that only
// grows.  All partials are summed in rank order, so the result does not depend
// on arrival order and is the same in every block:
//   every form: each block waits for the whole team and sums them itself.
//     Three trips to L2 lie on the critical path (arrive, see the count, read
//     the partials), but size^2 NS values are read;
//   last form: the last block to arrive sums them, publishes the sums and
//     releases the others: six trips, size NS values.
// us per barrier, every / last form: one scalar 152 blocks 2.5 / 4.6, 304 3.7 /
// 5.4, 608 (the largest grid with one) 6.3 / 6.5; two 304 4.7 / 6.0, 456 6.7 /
// 6.4, 608 8.5 / 7.3; three 304 5.7 / 7.3, 456 8.5 / 7.7, 608 10.9 / 8.7.  So
// Team is always the every form, and BiTeam, for BiCGStab with its two and
// three scalars in every iteration, takes the last form beyond 400 blocks (FP32
// at 2048^2 168 us per iteration instead of 178); one kernel holds both there.
// A block one barrier ahead writes the other half of the slots; it cannot be
// two ahead.  Returns false if the wait ran out (ctrl->status is then
// DS_TIMEOUT) or another block flagged an error; the caller must then stop
// working on this team's solve.
//
// All blocks of the team must be co-resident (cooperative launch), and every
// thread has called team_begin before the block barrier of the first
// block_sum.  `sh` needs 32 * NS doubles of shared memory.  Inlined, and the
// sums passed through copies: by reference to a call the sums' owner, a sink
// with all its coefficients, lives in local memory, where every node reads them
// again (FP32 BiCGStab at 2048^2 187 us per iteration, so 168; FP64 CG-NB at
// 1024^2 61 and 51).
template <int NS, bool BOTH>
__device__ __forceinline__ bool team_reduce_impl(const Team& tm, const double (&mine)[NS], double (&out)[NS],
                                                 double* sh) {
  static_assert(NS <= RED_MAX, "partial-sum slots");
  __shared__ int s_ok;   // 0: gave up, 1: released, 2: the last block, which sums for all
  const int tid = threadIdx.x;
  Ctrl* ctrl = tm.ctrl;
  const unsigned epoch = team_epoch();
  const bool every = !BOTH || NS == 1 || tm.size <= 400;
  double* slots = tm.partials + (size_t)(epoch & 1u) * RED_MAX * tm.size;
  if (tid == 0) {
#pragma unroll
    for (int s = 0; s < NS; s++) slots[(size_t)tm.rank * NS + s] = mine[s];
    const unsigned full = (epoch + 1u) * (unsigned)tm.size;   // compared modulo 2^32
    int ok = 1;
    if (every) red_release(&ctrl->count, 1u);
    else if (atom_acq_rel(&ctrl->count, 1u) + 1u == full) ok = 2;
    if (ok == 1) {
      const unsigned* word = every ? &ctrl->count : &ctrl->gen;
      const unsigned target = every ? full : epoch + 1u;
      unsigned long long t0 = 0;
      unsigned spins = 0;
      while ((int)(ld_acquire(word) - target) < 0) {
        if (++spins > 64) {
          __nanosleep(100);
          if ((spins & 255) == 0) {
            if (t0 == 0) t0 = global_ns();
            if (ld_acquire_int(&ctrl->status) < 0) { ok = 0; break; }
            if (global_ns() - t0 > ctrl->timeout_ns) {
              atomicCAS(&ctrl->status, 0, (int)DS_TIMEOUT);
              ok = 0;
              break;
            }
          }
        }
      }
    }
    s_ok = ok;
  }
  __syncthreads();
  const int ok = s_ok;
  if (!ok) return false;
  if (tid == 0) team_epoch() = epoch + 1u;
  if (!every && ok == 1) {
#pragma unroll
    for (int s = 0; s < NS; s++) out[s] = __ldcg(&ctrl->scal[s]);
    return true;
  }
#pragma unroll
  for (int s = 0; s < NS; s++) out[s] = 0.0;
  for (int b = tid; b < tm.size; b += blockDim.x) {
#pragma unroll
    for (int s = 0; s < NS; s++) out[s] += __ldcg(&slots[(size_t)b * NS + s]);
  }
  block_sum<NS>(out, sh);
  if (!every && tid == 0) {
#pragma unroll
    for (int s = 0; s < NS; s++) ctrl->scal[s] = out[s];
    st_release(&ctrl->gen, epoch + 1u);
  }
  return true;
}
template <int NS, bool BOTH>
__device__ __forceinline__ bool team_reduce_copies(const Team tm, const double (&mine)[NS], double (&out)[NS],
                                                   double* sh) {
  double m[NS], r[NS];
#pragma unroll
  for (int s = 0; s < NS; s++) m[s] = mine[s];
  const bool ok = team_reduce_impl<NS, BOTH>(tm, m, r, sh);
#pragma unroll
  for (int s = 0; s < NS; s++) out[s] = r[s];
  return ok;
}
template <int NS>
__device__ __forceinline__ bool team_reduce(const Team& tm, const double (&mine)[NS], double (&out)[NS], double* sh) {
  return team_reduce_copies<NS, false>(tm, mine, out, sh);
}
struct BiTeam : Team {};
template <int NS>
__device__ __forceinline__ bool team_reduce(const BiTeam& tm, const double (&mine)[NS], double (&out)[NS],
                                            double* sh) {
  return team_reduce_copies<NS, true>(tm, mine, out, sh);
}

// LastTeam: the last block to arrive sums the partials in rank order, publishes
// the sums and releases the others.  Six trips to L2 instead of three, but
// fewer registers: for the batch kernels, which spill already (48 systems of 16
// to 24 nodes a side, 40 iterations: 4.10 ms against 4.64 with team_reduce
// above; up to 128 a side: 27.1 against 27.7), and for Gauss-Seidel, which has
// a barrier per residual check and not per sweep (256^3, 20 pipelined sweeps:
// 436 us each against 444; the 27-point form 4.27 ms against 4.50).  Its slots:
// NS * size partials.
struct LastTeam : Team {};

template <int NS>
__device__ bool team_reduce(const LastTeam& tm, const double (&mine)[NS], double (&out)[NS], double* sh) {
  __shared__ int s_last;
  __shared__ int s_ok;
  Ctrl* ctrl = tm.ctrl;
  double* partials = tm.partials;
  const int tid = threadIdx.x;
  if (tid == 0) {
    unsigned g = ld_acquire(&ctrl->gen);
#pragma unroll
    for (int s = 0; s < NS; s++) partials[(size_t)tm.rank * NS + s] = mine[s];
    __threadfence();
    unsigned arrived = atomicAdd(&ctrl->count, 1u);
    s_last = (arrived == (unsigned)tm.size - 1);
    s_ok = 1;
    if (!s_last) {
      unsigned long long t0 = global_ns();
      unsigned spins = 0;
      while (ld_acquire(&ctrl->gen) == g) {
        if (++spins > 64) {
          __nanosleep(100);
          if ((spins & 255) == 0) {
            if (ld_acquire_int(&ctrl->status) < 0) { s_ok = 0; break; }
            if (global_ns() - t0 > ctrl->timeout_ns) {
              atomicCAS(&ctrl->status, 0, (int)DS_TIMEOUT);
              s_ok = 0;
              break;
            }
          }
        }
      }
    }
  }
  __syncthreads();
  if (s_last) {
    __threadfence();
    double acc[NS];
#pragma unroll
    for (int s = 0; s < NS; s++) acc[s] = 0.0;
    for (int b = tid; b < tm.size; b += blockDim.x) {
#pragma unroll
      for (int s = 0; s < NS; s++) acc[s] += __ldcg(&partials[(size_t)b * NS + s]);
    }
    block_sum<NS>(acc, sh);
    if (tid == 0) {
#pragma unroll
      for (int s = 0; s < NS; s++) ctrl->scal[s] = acc[s];
      ctrl->count = 0;
      __threadfence();
      unsigned g = ctrl->gen;
      st_release(&ctrl->gen, g + 1);
    }
#pragma unroll
    for (int s = 0; s < NS; s++) out[s] = acc[s];
    __syncthreads();
    return ld_acquire_int(&ctrl->status) >= 0;
  }
  int ok = s_ok;
  __syncthreads();
  if (!ok) return false;
#pragma unroll
  for (int s = 0; s < NS; s++) out[s] = __ldcg(&ctrl->scal[s]);
  __syncthreads();
  return true;
}

// A plain barrier (no data).  The block barrier first: one thread arrives for
// the block, which must not be before the other warps' work is done
// (team_reduce's callers come from block_sum, which ends with one).
template <class TM>
__device__ __forceinline__ bool team_sync(const TM& tm, double* sh) {
  __syncthreads();
  double z[1] = {0.0}, o[1];
  return team_reduce<1>(tm, z, o, sh);
}

template <class TM = Team>
__device__ __forceinline__ TM grid_team(Ctrl* ctrl, double* partials) {
  TM t;
  t.rank = blockIdx.x;
  t.size = gridDim.x;
  t.ctrl = ctrl;
  t.partials = partials;
  return t;
}
// Whole-grid forms of LastTeam (Gauss-Seidel).
template <int NS>
__device__ __forceinline__ bool grid_reduce(Ctrl* ctrl, double* partials, const double (&mine)[NS],
                                            double (&out)[NS], double* sh) {
  return team_reduce<NS>(grid_team<LastTeam>(ctrl, partials), mine, out, sh);
}
__device__ __forceinline__ bool grid_sync(Ctrl* ctrl, double* partials, double* sh) {
  return team_sync(grid_team<LastTeam>(ctrl, partials), sh);
}

}  // namespace hs

// Warp-strip SGS sweep with bulk-copy staging (FP32 recurrence), and the FP64 defect correction
// that turns two such sweeps into an FP64-accurate application of the preconditioner.
//
// The sweeps apply P^-1 = ((D+L) D^-1 (D+U))^-1 of eq. (sgs-precon) (section 4.4) in the
// transfer-block form of kernels_sweep.cu:
//   forward  y_c = D_c^-1 r_c + G_W y_W + G_S y_S            (y_S: the wake-cut mirror on row 0
//                                                             of the upper wake),
//   backward z_c = y_c + H_E z_E + H_N z_N (+ G_S z_mirror on row 0 of the lower wake).
// Rows are cut into strips of 8, one warp each, four lanes per cell (one per component): lane
// 4 r + q holds component q of row r.  Step s of a strip takes cell i = s - r of row r, so that a
// step needs only what the step before left: the cell's own previous vector (the west / east
// neighbour) and the neighbour row's (south / north).
//
// What bounds it: the latency of one step, not bandwidth (about 5 % of the DRAM rate).  A step is
// a store of the previous result to shared memory, two 16-byte loads of it (own vector and
// neighbour row) and a chain of eight FMAs; at 1024x256 the chain is walked 2 x 1,032 times.
// Measured per step on one SM, operands in shared memory: one lane per cell (32 rows, shuffles,
// nine 16-byte operand loads per lane) 96 cycles and 124 with its 16-byte result store; two lanes
// per cell 108; four lanes with eight shuffles 85; four lanes exchanging through shared memory 67.
// The operand and result instructions of a step queue ahead of the next step's exchange in the
// same in-order pipe, so fewer of them per lane is what shortens the step.
//
// A strip's operands are laid out in the order its warp consumes them (strip-major, step by step,
// zero where a step has no cell).  A second warp per strip moves them: stages of eight steps by
// cp.async.bulk into a ring in shared memory, and the results back by one bulk store per stage, so
// that the computing warp issues no global access at all; a third warp watches for what a stage
// needs.  Two strips share a CTA (each strip's computing warp has a scheduler of its own; one strip
// per CTA is 1-3 % faster alone and takes twice the SMs).
//
// The strips of a sweep form one thread-block cluster.  Strip b follows strip b-1 (forward; b+1
// backward) through the neighbour's boundary row: each stage of the neighbour's out row is stored
// straight into this strip's edge buffer (remote stores inside the cluster), which holds a
// sentinel bit pattern until the value lands.  No fence or flag is needed: each 32-bit word arrives
// whole, and the sentinel (a NaN payload that no arithmetic produces) marks the words not yet
// written.  Every wait is bounded; on timeout the kernel sets the error word, waits (bounded) for its
// own copies in flight, and still meets the cluster's barriers, so that no strip waits forever.
//
// One sweep pair in an FP64 cycle (from the end of the kernel before), strips of 32 rows with a lane per cell
// that staged and stored for themselves against these: 64x16 17.7 -> 12 us, 128x32 30.8 -> 22, 256x64 62.5 -> 42,
// 512x128 82, 1024x256 246 -> 162; about 43 ns a step (about 80 before) and 1.1 us from strip to strip.
// A tree instead of the chain of eight FMAs (FP64 contexts could take it) gains 1 %: the step waits for its
// shared-memory instructions.
#include <atomic>
#include <cstdint>
#include <type_traits>

#include "fasw_fp64.cuh"
#include "fasw_internal.cuh"
#include "fasw_sweep.cuh"

namespace fasw {

namespace {

constexpr unsigned WS_SENT = 0xFFFFFFFFu;  // "not yet written": a NaN payload no FP32 operation returns
constexpr unsigned WS_ALL = 0xFFFFFFFFu;   // every lane of a warp
constexpr int WS_STEP_BYTES = 16 * WS_F4_STEP, WS_VEC_BYTES = 16 * WS_ROWS;  // one step's blocks / vectors
constexpr int WS_HEAD = 512;               // barriers and the two strips' give-up words
constexpr int WS_STAGES = 5, WS_SHALLOW = 3;  // ring depth; of kind 10
constexpr int WS_TAIL = 16;                // zero entries after the edge buffer's last step

__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool mbar_test(uint64_t* bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// global -> shared bulk copy (16-byte aligned addresses, size a multiple of 16)
__device__ __forceinline__ void bulk_copy(void* dst, const void* src, unsigned bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_addr(dst)),
               "l"(src), "r"(bytes), "r"(smem_addr(bar))
               : "memory");
}

// shared -> global bulk copy (same rules), and the wait until its source may be overwritten
__device__ __forceinline__ void bulk_store(void* dst, const void* src, unsigned bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_addr(src)),
               "r"(bytes)
               : "memory");
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}

// address of the same shared-memory variable in CTA `rank` of this cluster
__device__ __forceinline__ unsigned cluster_addr(const void* p, unsigned rank) {
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr(p)), "r"(rank));
  return r;
}

__device__ __forceinline__ float4 lds4(unsigned a) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(a)
               : "memory");
  return v;
}

__device__ __forceinline__ float lds1(unsigned a) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}

__device__ __forceinline__ void sts1(unsigned a, float v) {
  asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}

// predicated in the instruction itself (no branch around it)
__device__ __forceinline__ void sts1_if(bool pred, unsigned a, float v) {
  asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %2, 0;\n @p st.shared.f32 [%0], %1;\n}\n" ::"r"(a), "f"(v),
               "r"((unsigned)pred)
               : "memory");
}

__device__ __forceinline__ void sts4(unsigned a, float4 v) {
  asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}

__device__ __forceinline__ void st_cluster4(unsigned a, float4 v) {
  asm volatile("st.relaxed.cluster.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.x), "f"(v.y),
               "f"(v.z), "f"(v.w)
               : "memory");
}

__device__ __forceinline__ void mbar_arrive_if(bool pred, uint64_t* bar) {
  asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %1, 0;\n @p mbarrier.arrive.shared::cta.b64 _, [%0];\n}\n" ::"r"(
                   smem_addr(bar)),
               "r"((unsigned)pred)
               : "memory");
}

__device__ __forceinline__ uint4 ld_cluster4(unsigned a) {
  uint4 v;
  asm volatile("ld.relaxed.cluster.shared::cta.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "r"(a)
               : "memory");
  return v;
}

__device__ __forceinline__ unsigned ld_acquire(unsigned a) {
  unsigned v;
  asm volatile("ld.acquire.cta.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}

__device__ __forceinline__ unsigned ld_relaxed(unsigned a) {
  unsigned v;
  asm volatile("ld.relaxed.cta.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}

__device__ __forceinline__ void st_release(unsigned a, unsigned v) {
  asm volatile("st.release.cta.shared::cta.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

__device__ __forceinline__ bool unwritten(uint4 v) {
  return v.x == WS_SENT || v.y == WS_SENT || v.z == WS_SENT || v.w == WS_SENT;
}

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

// Shared memory of one strip (byte addresses): the barriers of its ring, the ring (blocks, right
// hand sides, results), the exchange vectors of the last step, the edge buffers of the two passes
// (one buffer, cleared between them, on grids too long for two); and, shared by the CTA, the wake
// cut's vectors and coupling blocks (strip 0 only).
struct WsSmem {
  uint64_t *full, *empty;    // per ring slot: operands landed; slot consumed, its results complete
  // counters: ring uses whose operands and edge entries have landed; passes whose first right-hand
  // sides are in place
  unsigned char *ready, *primed;
  volatile int* gave_up;     // a warp of this strip gave up
  unsigned char *F, *C, *H;  // NS stages of blocks / right-hand sides / results
  unsigned char* X;          // [row][component] of the last step
  unsigned char *Ef, *Eb;    // Mp + WS_TAIL vectors: the neighbour's out row by its step (t >= Mp: zero)
  unsigned char *cutv, *cutG;
};

template <int NS, bool TWO>
__host__ __device__ constexpr size_t ws_strip_bytes(int Mp) {
  return (size_t)NS * WS_U * (WS_STEP_BYTES + 2 * WS_VEC_BYTES) + WS_VEC_BYTES +
         (TWO ? 2 : 1) * (size_t)(Mp + WS_TAIL) * 16;
}

template <int NS, bool TWO>
__host__ __device__ constexpr size_t ws_cta_bytes(int Mp, int nw) {
  return WS_HEAD + 2 * ws_strip_bytes<NS, TWO>(Mp) + 80 * (size_t)(nw > 0 ? nw : 1);
}

template <int NS, bool TWO>
__device__ __forceinline__ WsSmem ws_carve(unsigned char* base, int w, int Mp, int nw) {
  static_assert(32 * NS + 32 <= WS_HEAD, "the barriers fit the head");
  WsSmem S;
  S.full = reinterpret_cast<uint64_t*>(base) + w * 2 * NS;
  S.empty = S.full + NS;
  S.ready = base + WS_HEAD - 8 + 4 * w;
  S.primed = S.ready - 16;
  S.gave_up = reinterpret_cast<volatile int*>(base + WS_HEAD - 16) + w;
  S.F = base + WS_HEAD + w * ws_strip_bytes<NS, TWO>(Mp);
  S.C = S.F + NS * WS_U * WS_STEP_BYTES;
  S.H = S.C + NS * WS_U * WS_VEC_BYTES;
  S.X = S.H + NS * WS_U * WS_VEC_BYTES;
  S.Ef = S.X + WS_VEC_BYTES;
  S.Eb = TWO ? S.Ef + (size_t)(Mp + WS_TAIL) * 16 : S.Ef;
  S.cutv = base + WS_HEAD + 2 * ws_strip_bytes<NS, TWO>(Mp);
  S.cutG = S.cutv + 16 * (size_t)(nw > 0 ? nw : 1);
  return S;
}

}  // namespace

int ws_strips(int nj) { return (nj + WS_ROWS - 1) / WS_ROWS; }

namespace {

// Ring bookkeeping: stage ch of a pass that starts at ring count `base` (0 forward, the number of
// stages backward) is ring use n = base + ch: slot n % NS, phase n / NS.
template <int NS>
__device__ __forceinline__ bool ws_landed(uint64_t* bar, unsigned n) {
  return mbar_test(&bar[n % NS], (n / NS) & 1u);
}

__device__ __forceinline__ void ws_give_up(const WsSmem& S, int* err) {
  atomicExch(err, 1);
  *S.gave_up = 1;
}

// What the copying warp of a strip moves: blocks and right-hand sides in, results out.
struct WsGlobal {
  const unsigned char *F, *B, *C;  // forward / backward blocks, forward right-hand sides
  unsigned char *Y, *Z;            // forward result (the backward right-hand sides), backward result
  int nch;                         // stages of a pass
};

// Fills the slot of ring use n (the copying lane): the blocks (ws_fill_blocks, which also announces
// the bytes of both) and the right-hand sides (ws_fill_rhs).  The right-hand sides of the first NS
// backward stages are not fetched: they are the last forward stages' results, still in shared memory.
template <int NS>
__device__ __forceinline__ bool ws_fetched(const WsGlobal& G, unsigned n) {
  return n < (unsigned)G.nch || n - G.nch >= NS;
}

template <int NS>
__device__ __forceinline__ void ws_fill_blocks(const WsSmem& S, const WsGlobal& G, unsigned n) {
  constexpr unsigned FB = WS_U * WS_STEP_BYTES, CB = WS_U * WS_VEC_BYTES;
  const unsigned sl = n % NS;
  const bool fwd = n < (unsigned)G.nch;
  mbar_expect_tx(&S.full[sl], ws_fetched<NS>(G, n) ? FB + CB : FB);
  bulk_copy(S.F + sl * FB, (fwd ? G.F : G.B) + (size_t)(fwd ? n : n - G.nch) * FB, FB, &S.full[sl]);
}

template <int NS>
__device__ __forceinline__ void ws_fill_rhs(const WsSmem& S, const WsGlobal& G, unsigned n) {
  constexpr unsigned CB = WS_U * WS_VEC_BYTES;
  const unsigned sl = n % NS;
  const bool fwd = n < (unsigned)G.nch;
  if (ws_fetched<NS>(G, n))
    bulk_copy(S.C + sl * CB, (fwd ? G.C : G.Y) + (size_t)(fwd ? n : n - G.nch) * CB, CB, &S.full[sl]);
}

// The helper warps' loops are warp-uniform (a vote decides whether any lane still waits), so that a
// warp leaves them converged; each ends when the strip gives up, or after WS_LONG rounds (helpers
// outwait the computing warp and the edge entries, whose limit is the caller's).
constexpr long long WS_LONG = 1LL << 26;

template <class Ready>
__device__ __forceinline__ bool ws_wait(const WsSmem& S, Ready ready) {
  long long spins = 0;
  while (!__all_sync(WS_ALL, ready()))
    if (__any_sync(WS_ALL, *S.gave_up || ++spins > WS_LONG)) return false;
  return true;
}

// One pass of the copying warp: a consumed slot's boundary row goes to the strip this one feeds
// (feeds: the cluster address of its edge buffer, 0: none), its results to global memory, then the
// slot is filled again (backward stages too: their blocks are on their way while the forward pass
// ends).  A slot's operands were only read by the computing warp, its results written by it before
// it arrived on `empty`.  Returns false if the strip gave up, after waiting (bounded: its copies
// depend on no other CTA) for the copies in flight into this CTA's shared memory.
template <bool FWD, int NS>
__device__ __forceinline__ bool ws_copies(const WsSmem& S, const WsGlobal& G, unsigned feeds) {
  constexpr unsigned CB = WS_U * WS_VEC_BYTES;
  const int lane = threadIdx.x & 31;
  const unsigned nch = G.nch, all = 2 * nch, base = FWD ? 0 : nch, end = base + nch;
  if (FWD) {
    if (lane == 0)
      for (unsigned n = 0; n < NS && n < all; ++n) ws_fill_rhs<NS>(S, G, n);  // the blocks are on their way
  } else {
    // results of stage nch - 1 - k: right-hand sides of ring use nch + k
    for (int k = min(NS, G.nch) - 1; k >= 0; --k) {
      const unsigned from = smem_addr(S.H) + ((nch - 1 - k) % NS) * CB, to = smem_addr(S.C) + ((nch + k) % NS) * CB;
      for (unsigned x = 16 * lane; x < CB; x += 512) sts4(to + x, lds4(from + x));
    }
  }
  __syncwarp();
  if (lane == 0) st_release(smem_addr(S.primed), FWD ? 1 : 2);
  for (unsigned n = base; n < end; ++n) {
    if (!ws_wait(S, [&] { return ws_landed<NS>(S.empty, n); })) {
      for (unsigned k = n; k < n + NS && k < all; ++k) {
        long long m = 0;
        while (!ws_landed<NS>(S.full, k) && ++m <= WS_LONG) {
        }
      }
      asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
      __syncwarp();
      return false;
    }
    const unsigned d = n - base;
    const unsigned char* H = S.H + (n % NS) * CB;
    if (feeds && lane < WS_U)  // the out row at step d WS_U + lane
      st_cluster4(feeds + 16 * (d * WS_U + lane),
                  lds4(smem_addr(H) + (FWD ? WS_U - 1 - lane : lane) * WS_VEC_BYTES + (FWD ? 16 * (WS_ROWS - 1) : 0)));
    if (lane == 0) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the results just acquired
      bulk_store((FWD ? G.Y : G.Z) + (size_t)(FWD ? nch - 1 - d : d) * CB, H, CB);
      if (n + NS < all) {
        if (n == nch)  // from here on y comes back from global memory: its stores have completed
          asm volatile("cp.async.bulk.wait_group 1;\n\tfence.proxy.async.global;" ::: "memory");
        asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
        ws_fill_blocks<NS>(S, G, n + NS);
        ws_fill_rhs<NS>(S, G, n + NS);
      }
    }
    __syncwarp();
  }
  if (!FWD) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
  __syncwarp();
  return true;
}

// One pass of the watching warp: a stage is ready when its operands have landed and, where a
// neighbour feeds this strip, its edge entries (lane k: entry s0 + 7 + k): none of their words holds
// the sentinel.
template <int NS>
__device__ __forceinline__ bool ws_watch(const WsSmem& S, int nch, unsigned base, bool fed, const unsigned char* Eb,
                                         int* err, long long limit) {
  const int lane = threadIdx.x & 31;
  const unsigned E = smem_addr(Eb) + 16 * (WS_ROWS - 1 + (lane & (WS_U - 1)));
  if (!ws_wait(S, [&] { return ld_acquire(smem_addr(S.primed)) > (base ? 1u : 0u); })) return false;
  for (int ch = 0; ch < nch; ++ch) {
    if (!ws_wait(S, [&] { return ws_landed<NS>(S.full, base + ch); })) return false;
    long long spins = 0;
    while (fed && __any_sync(WS_ALL, unwritten(ld_cluster4(E + 16 * WS_U * ch)))) {
      ++spins;
      const bool stop = spins > limit || ((spins & 255) == 0 && (*S.gave_up || *((volatile int*)err) != 0));
      if (__any_sync(WS_ALL, stop)) {
        if (lane == 0) ws_give_up(S, err);
        __syncwarp();
        return false;
      }
    }
    __syncwarp();
    if (lane == 0) st_release(smem_addr(S.ready), base + ch + 1);
  }
  return true;
}

// One pass (forward: FWD, else backward) of one strip by its computing warp.  Returns false on a
// timeout.  Row r at step s holds cell i = s - r (forward) or Mp - 1 - s - r (backward); the edge
// row needs the neighbour's out row of the same column, which the neighbour computed at its step
// s + 7: edge entry s + 7 (entries Mp ... are zero).  On row 0 of the upper wake the entry is the
// mirror cell's vector, stored there by this strip's own row 0 when it passed that cell.
//
// A taken branch costs this warp about 35 cycles and each test or vote as much as half a step, so
// a stage is straight-line code: eight unrolled steps, one wait, asked for two steps ahead, and one
// loop branch; everything else is the other warps' work.
template <bool FWD, int NS>
__device__ __forceinline__ bool ws_pass(const LevelDev& L, const WsSmem& S, int b, int Mp, unsigned base, int* err,
                                        long long limit) {
  constexpr unsigned FB = WS_U * WS_STEP_BYTES, CB = WS_U * WS_VEC_BYTES;
  const int lane = threadIdx.x & 31, r = lane >> 2, q = lane & 3;
  const int ni = L.ni, nw = L.nw, nch = Mp / WS_U;
  const bool edge_row = r == (FWD ? 0 : WS_ROWS - 1);
  const unsigned x_own = smem_addr(S.X) + 16 * r, x_put = smem_addr(S.X) + 4 * lane;
  const unsigned E = smem_addr(FWD ? S.Ef : S.Eb), ready = smem_addr(S.ready);
  const unsigned fa = smem_addr(S.F) + 16 * lane, ca = smem_addr(S.C) + 4 * lane, ha = smem_addr(S.H) + 4 * lane;
  const unsigned cutv = smem_addr(S.cutv), cutG = smem_addr(S.cutG) + 16 * q;
  // the row below (forward) / above (backward); the edge row's moves on by an entry a step
  const unsigned nb0 = edge_row ? E + 16 * (WS_ROWS - 1) : FWD ? x_own - 16 : x_own + 16;
  const unsigned nb_step = edge_row ? 16 : 0;

  auto wait_stage = [&](unsigned n) -> bool {  // the rare path: the stage has not landed yet
    long long spins = 0;
    while (!__all_sync(WS_ALL, ld_acquire(ready) > n)) {
      ++spins;
      const bool stop = spins > limit || ((spins & 255) == 0 && *S.gave_up);
      if (__any_sync(WS_ALL, stop)) {
        if (lane == 0) ws_give_up(S, err);
        __syncwarp();
        return false;
      }
    }
    return true;
  };
  // Operands of one step: this lane's row of the two blocks and its right-hand side component,
  // loaded one step ahead of their use (across stages too).
  float4 A[2], B[2];
  float c[2];
  auto load = [&](int z, unsigned sl, int u) {
    c[z] = lds1(ca + sl * CB + u * WS_VEC_BYTES);  // first: the sum starts with it
    A[z] = lds4(fa + sl * FB + u * WS_STEP_BYTES);
    B[z] = lds4(fa + sl * FB + u * WS_STEP_BYTES + WS_STEP_BYTES / 2);
  };
  float y = 0.f;            // this lane's component at the previous step
  unsigned sl = base % NS;  // ring slot
  bool ok = true;
  // Stages ch0 .. ch1 - 1.  Padded positions (no cell) carry zero blocks and vectors, so they
  // compute zero and need no test.  Only the wake-cut coupling of row 0 (strip 0) is special; stages
  // that hold no cut cell run without it (CUT false).
  auto stages = [&](int ch0, int ch1, auto cut_tag) {
    constexpr bool CUT = decltype(cut_tag)::value;
#pragma unroll 1
    for (int ch = ch0; ch < ch1; ++ch) {
      const int s = ch * WS_U;
      const unsigned nb = nb0 + ch * WS_U * nb_step, h = ha + sl * CB;
      const unsigned nsl = sl + 1 == NS ? 0 : sl + 1;
      const unsigned next = base + min(ch + 1, nch - 1);  // the last stage waits for itself
      unsigned landed = 0;
#pragma unroll
      for (int u = 0; u < WS_U; ++u) {
        sts1(x_put, y);
        __syncwarp();
        const float4 x = lds4(x_own), w = lds4(nb + u * nb_step);
        if (u > 0) sts1(h + (FWD ? WS_U - u : u - 1) * WS_VEC_BYTES, y);  // the previous step's result
        if (u == WS_U - 2) landed = ld_relaxed(ready);
        // one decision for the warp: each lane reads the counter for itself, and wait_stage's votes take every lane
        if (u == WS_U - 1 && __builtin_expect(!__all_sync(WS_ALL, landed > next), 0) && !wait_stage(next)) {
          ok = false;
          return;
        }
        if (u == WS_U - 1) asm volatile("fence.acq_rel.cta;" ::: "memory");  // the counter was read relaxed
        load((u + 1) & 1, u + 1 < WS_U ? sl : nsl, (u + 1) % WS_U);
        // the west / east part first: its vector is this row's own
        float a = c[u & 1];
        a = fmaf(A[u & 1].x, x.x, a);
        a = fmaf(A[u & 1].y, x.y, a);
        a = fmaf(A[u & 1].z, x.z, a);
        a = fmaf(A[u & 1].w, x.w, a);
        a = fmaf(B[u & 1].x, w.x, a);
        a = fmaf(B[u & 1].y, w.y, a);
        a = fmaf(B[u & 1].z, w.z, a);
        a = fmaf(B[u & 1].w, w.w, a);
        if constexpr (CUT) {
          const int i = FWD ? s + u : Mp - 1 - s - u, m = ni - 1 - i;  // row 0's cell and its mirror
          if (FWD) {  // lower wake: read by its mirror as that cell's edge entry
            sts1_if(r == 0 && i < nw, E + 16 * (unsigned)(m + WS_ROWS - 1) + 4 * q, a);
          } else {
            const int ic = min(max(i, 0), nw - 1);
            const float4 g = lds4(cutG + 64 * ic), v = lds4(cutv + 16 * ic);
            const float t = fmaf(g.w, v.w, fmaf(g.z, v.z, fmaf(g.x, v.x, __fmul_rn(g.y, v.y))));
            if (r == 0 && i >= 0 && i < nw) a = __fadd_rn(a, t);                              // lower wake
            sts1_if(r == 0 && i < ni && m < nw, cutv + 16 * (unsigned)max(m, 0) + 4 * q, a);  // read by its mirror
          }
        }
        y = a;
      }
      sts1(h + (FWD ? 0 : WS_U - 1) * WS_VEC_BYTES, y);
      // the slot's operands are consumed and its results complete: over to the copying warp
      __syncwarp();
      mbar_arrive_if(lane == 0, &S.empty[sl]);
      sl = nsl;
    }
  };
  if (!wait_stage(base)) return false;
  load(0, sl, 0);
  // stages with a cut cell of row 0 whose coupling is its own: forward the lower wake (the first
  // nw columns); backward the upper wake (whose vectors are kept) and the lower one
  const bool cut = b == 0 && nw > 0;
  const int lo = cut ? min((nw + WS_U - 1) / WS_U, nch) : 0;               // stages 0 .. lo - 1: columns < nw
  const int hi = cut ? min((Mp - (ni - nw) + WS_U - 1) / WS_U, nch) : 0;   // backward: columns >= ni - nw
  const int mid = cut && !FWD ? min(max(hi, (Mp - nw) / WS_U), nch) : nch;  // backward, from here: columns < nw
  stages(0, FWD ? lo : hi, std::true_type{});
  if (ok) stages(FWD ? lo : hi, mid, std::false_type{});
  if (ok) stages(mid, nch, std::true_type{});
  return ok;
}

__device__ __forceinline__ void ws_clear(unsigned char* E, int Mp, bool fed, int t0, int dt) {
  const float sent = __uint_as_float(WS_SENT);
  for (int t = t0; t < Mp + WS_TAIL; t += dt) {
    const float v = t < Mp && fed ? sent : 0.f;
    reinterpret_cast<float4*>(E)[t] = make_float4(v, v, v, v);
  }
}

// One launch: forward then backward pass of every strip.  Warps 0 and 1 of a CTA compute strips
// 2 blockIdx and 2 blockIdx + 1, on schedulers 0 and 1; their helpers (copying: warps 2, 3; watching:
// 6, 7) are the warps of schedulers 2 and 3, so that no helper takes an issue slot of a computing
// warp, and warps 4 and 5 only meet the barriers.  Every thread meets the cluster barriers (set-up,
// two between the passes where they share an edge buffer, at the end) whatever happened in its
// passes, so that a strip that gave up leaves no other one waiting on a barrier; the last barrier
// also keeps every CTA's shared memory alive until the neighbours' remote stores into it have
// completed.
constexpr int WS_THREADS = 256;

template <int NS, bool TWO>
__global__ void __launch_bounds__(WS_THREADS)
    k_sweep_ws(LevelDev L, const float4* Fb, const float4* Bb, const float4* C, float4* Y, const float* cutG, float4* Z,
               int* err, long long limit) {
  extern __shared__ __align__(128) unsigned char ws_raw[];
  const int nw = L.nw, Mp = ws_steps(L.ni, L.nj), nst = (L.nj + WS_ROWS - 1) / WS_ROWS;
  const int warp = threadIdx.x >> 5, w = warp & 1, b = 2 * blockIdx.x + w, lane = threadIdx.x & 31;
  const bool compute = warp < 2, copier = (warp & ~1) == 2, watcher = (warp & ~1) == 6;
  const bool below = b > 0, above = b < nst - 1;  // neighbour strips
  const WsSmem S = ws_carve<NS, TWO>(ws_raw, w, Mp, nw);
  // Set-up while the kernel before still runs: this CTA's shared memory, the cluster's first barrier, and
  // the first blocks.  The blocks are k_sgs_prep's, which is never the kernel before (the right-hand
  // side's kernel is), and a kernel lets its successor start only once its own predecessors have
  // completed (pdl_entry), so they are complete here (a sweep pair 1 us less).
  if (copier && lane == 0) {
    for (int k = 0; k < NS; ++k) {
      mbar_init(&S.full[k], 1);
      mbar_init(&S.empty[k], 1);
    }
    *S.gave_up = 0;
    st_release(smem_addr(S.ready), 0);
    st_release(smem_addr(S.primed), 0);
    asm volatile("fence.mbarrier_init.release.cluster;\n\tfence.proxy.async.shared::cta;" ::: "memory");
  }
  const int part = (warp >> 1) * 32 + lane;  // of the threads of this strip
  ws_clear(S.Ef, Mp, below, part, WS_THREADS / 2);
  if (TWO) ws_clear(S.Eb, Mp, above, part, WS_THREADS / 2);
  const size_t blk = (size_t)b * Mp * WS_STEP_BYTES, vec = (size_t)b * Mp * WS_VEC_BYTES;
  const WsGlobal G{reinterpret_cast<const unsigned char*>(Fb) + blk, reinterpret_cast<const unsigned char*>(Bb) + blk,
                   reinterpret_cast<const unsigned char*>(C) + vec,  reinterpret_cast<unsigned char*>(Y) + vec,
                   reinterpret_cast<unsigned char*>(Z) + vec,        Mp / WS_U};
  if (b < nst && copier && lane == 0) {  // see above: written two launches ago or earlier
    for (unsigned n = 0; n < NS && n < 2u * G.nch; ++n) ws_fill_blocks<NS>(S, G, n);
  }
  if (b == 0)
    for (int x = part; x < 16 * nw; x += WS_THREADS / 2) reinterpret_cast<float*>(S.cutG)[x] = cutG[x];
  // every strip's edge buffer holds its sentinels before any neighbour stores into it
  cluster_arrive();
  cluster_wait();
  pdl_entry();
  bool ok = b < nst;
  const WsSmem other = ws_carve<NS, TWO>(ws_raw, w ^ 1, Mp, nw);
  if (compute) {
    ok = ok && ws_pass<true, NS>(L, S, b, Mp, 0, err, limit);
  } else if (copier) {
    ok = ok && ws_copies<true, NS>(S, G, above ? cluster_addr(other.Ef, (unsigned)(b + 1) >> 1) : 0u);
  } else if (watcher) {
    ok = ok && ws_watch<NS>(S, G.nch, 0, below, S.Ef, err, limit);
  }
  __syncwarp();
  if (!TWO) {  // every strip has read its edge buffer to the end; cleared before a neighbour stores into it again
    cluster_arrive();
    cluster_wait();
    ws_clear(S.Eb, Mp, above, part, WS_THREADS / 2);
    cluster_arrive();
    cluster_wait();
  }
  if (compute) {
    if (ok) ws_pass<false, NS>(L, S, b, Mp, G.nch, err, limit);
  } else if (copier) {
    if (ok) ws_copies<false, NS>(S, G, below ? cluster_addr(other.Eb, (unsigned)(b - 1) >> 1) : 0u);
  } else if (watcher) {
    if (ok) ws_watch<NS>(S, G.nch, G.nch, above, S.Eb, err, limit);
  }
  __syncwarp();
  cluster_arrive();
  cluster_wait();
}

// ---------------------------------------------------------------- the kernels around the sweep
// The FP64 kernels of one application, written per row q of their block products: a thread
// takes one cell and all four rows (SPLIT false: the loads of a warp coalesce along the cells, for
// levels whose time is their memory traffic), or one cell and one row (SPLIT true: a quarter of
// the FP64 chain per thread, for the small levels whose time is that chain).  Every row is summed
// in the same order either way.

template <bool SPLIT>
__device__ __forceinline__ bool ws_thread(const LevelDev& L, int& c, int& q0, int& q1) {
  const int g = blockIdx.x * blockDim.x + threadIdx.x;
  if (SPLIT) {
    c = g >> 2;
    q0 = g & 3;
    q1 = q0 + 1;
  } else {
    c = g;
    q0 = 0;
    q1 = 4;
  }
  return c < L.n;
}

// row q of D^-1 r
template <typename T>
__device__ __forceinline__ double rhs_row(const LevelDev& L, const T* tb, const double* rhs, int c, int q) {
  const int n = L.n;
  double a = 0.0;
#pragma unroll
  for (int t = 0; t < 4; ++t) a += to64(tb[(size_t)(4 * q + t) * n + c]) * rhs[(size_t)t * n + c];
  return a;
}

// D^-1 r of a given right-hand side (the stages' own comes from the residual kernel): FP32, skewed, and
// in FP64 contexts FP64 in R for the defect.
template <typename T, bool SPLIT>
__global__ void k_ws_rhs(LevelDev L, const T* tb, const double* rhs, float4* C, double* R) {
  pdl_entry();
  int c, q0, q1;
  if (!ws_thread<SPLIT>(L, c, q0, q1)) return;
  const int ni = L.ni, i = c % ni, j = c / ni;
  const int b = j / WS_ROWS, jl = j % WS_ROWS, Mp = ws_steps(ni, L.nj);
  float* out = reinterpret_cast<float*>(C + ((size_t)b * Mp + (i + jl)) * WS_ROWS + jl);
  for (int q = q0; q < q1; ++q) {
    const double a = rhs_row(L, tb, rhs, c, q);
    out[q] = d2f(a);
    if (R) R[(size_t)q * L.n + c] = a;
  }
}

// ---------------------------------------------------------------- FP64 defect correction
// t = (I + U~) z: the vector the backward sweep would have started from to reach z,
//   t_c = z_c - H_E z_E - H_N z_N (- G_S z_mirror on row 0 of the lower wake),
// z = z0 (+ dz: SECOND, the second correction's).
// One thread per cell, t and d in a launch each (grids above WS_SPLIT_CELLS).
template <bool SECOND>
__device__ __forceinline__ void load_z(const float4* z0, const float4* dz, size_t pos, double x[4]) {
  ws_load64(z0, pos, x);
  if constexpr (SECOND) {
    double d[4];
    ws_load64(dz, pos, d);
#pragma unroll
    for (int q = 0; q < 4; ++q) x[q] += d[q];
  }
}

template <bool SECOND>
__global__ void k_ws_defect_t(LevelDev L, const double* tb, const float4* z0, const float4* dz, double* t) {
  pdl_entry();
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= L.n) return;
  const int ni = L.ni, nj = L.nj, n = L.n, i = c % ni, j = c / ni, Mp = ws_steps(ni, nj);
  double x[4];
  load_z<SECOND>(z0, dz, ws_bpos(i, j, Mp), x);
  double acc[4] = {x[0], x[1], x[2], x[3]};
  auto sub = [&](int blk, int in, int jn) {
    load_z<SECOND>(z0, dz, ws_bpos(in, jn, Mp), x);
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int k = 0; k < 4; ++k) acc[q] -= tb[(size_t)(blk * 16 + 4 * q + k) * n + c] * x[k];
  };
  if (i < ni - 1) sub(3, i + 1, j);
  if (j < nj - 1) sub(4, i, j + 1);
  if (j == 0 && L.nw > 0 && i < L.nw && ni - 1 - i > i) sub(2, ni - 1 - i, 0);
#pragma unroll
  for (int q = 0; q < 4; ++q) t[(size_t)q * n + c] = acc[q];
}

// d = D^-1 r - (I + L~) t = D^-1 r - t_c + G_W t_W + G_S t_S (t_S: the mirror on row 0 of the
// upper wake, none elsewhere on row 0), written as the next forward right-hand side (FP32).
__device__ __forceinline__ double defect_d_row(const LevelDev& L, const double* tb, const double* R, const double* t,
                                               int c, int q) {
  const int ni = L.ni, n = L.n, i = c % ni, j = c / ni;
  double a = R[(size_t)q * n + c] - t[(size_t)q * n + c];
  auto add = [&](int blk, int cn) {
#pragma unroll
    for (int k = 0; k < 4; ++k) a += tb[(size_t)(blk * 16 + 4 * q + k) * n + c] * t[(size_t)k * n + cn];
  };
  if (i > 0) add(1, c - 1);
  if (j > 0) add(2, c - ni);
  else if (L.nw > 0 && i >= ni - L.nw && ni - 1 - i < i) add(2, ni - 1 - i);
  return a;
}

__global__ void k_ws_defect_d(LevelDev L, const double* tb, const double* R, const double* t, float4* C) {
  pdl_entry();
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= L.n) return;
  float* out = reinterpret_cast<float*>(C + ws_fpos(c % L.ni, c / L.ni, ws_steps(L.ni, L.nj)));
#pragma unroll
  for (int q = 0; q < 4; ++q) out[q] = d2f(defect_d_row(L, tb, R, t, c, q));
}

// Both in one launch (grids up to WS_SPLIT_CELLS): a block forms t of its 8 x 4 cells and of the row below
// and the column to their west in shared memory, a row of the products per thread, then d of its cells.
// tb and R were written two launches ago or earlier, so they are fetched before the wait for the sweep (a
// kernel lets its successor start only once its own predecessors have completed).  t's rows of the halo
// are three eighths more work: 64x16 4.7 -> 3.0 us against a launch each, 256x64 7.1 -> 6.4; with blocks of
// 32 x 8 cells (a sixth more) 512x128 takes 27 us against 20.6, 1024x256 76 against 53.
constexpr int WD_X = 8, WD_Y = 4, WD_THREADS = 192;
template <bool SECOND>
__global__ void __launch_bounds__(WD_THREADS) k_ws_defect(LevelDev L, const double* tb, const double* R, const float4* z0,
                                                          const float4* dz, float4* C) {
  constexpr int OWN = WD_X * WD_Y, ALL = OWN + WD_X + WD_Y;
  static_assert(4 * ALL <= WD_THREADS, "a row of the products per thread");
  __shared__ double ts[4][ALL];
  const int ni = L.ni, nj = L.nj, n = L.n, nw = L.nw, Mp = ws_steps(ni, nj);
  const int i0 = blockIdx.x * WD_X, j0 = blockIdx.y * WD_Y;
  // cell h of the block: its own, the row below (row 0: the mirrors on the upper wake), the column to the west
  auto cell = [&](int h, int& i, int& j) {
    if (h < OWN) {
      i = i0 + h % WD_X;
      j = j0 + h / WD_X;
    } else if (h < OWN + WD_X) {
      i = i0 + h - OWN;
      j = j0 - 1;
      if (j < 0) {
        if (i >= ni || i < ni - nw || ni - 1 - i >= i) return false;
        i = ni - 1 - i;
        j = 0;
      }
    } else {
      i = i0 - 1;
      j = j0 + h - OWN - WD_X;
    }
    return i >= 0 && i < ni && j < nj;
  };
  auto entry = [&](int blk, int q, int k, int c) { return tb[(size_t)(blk * 16 + 4 * q + k) * n + c]; };
  double E[4], N[4], W[4], S[4], r = 0.0;
  const int x = threadIdx.x, ht = x % ALL, qt = x / ALL, hd = x % OWN, qd = x / OWN;
  int it, jt, id, jd;
  const bool has_t = x < 4 * ALL && cell(ht, it, jt), has_d = x < 4 * OWN && cell(hd, id, jd);
  if (has_t) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      E[k] = entry(3, qt, k, jt * ni + it);
      N[k] = entry(4, qt, k, jt * ni + it);
    }
  }
  if (has_d) {
    r = R[(size_t)qd * n + jd * ni + id];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      W[k] = entry(1, qd, k, jd * ni + id);
      S[k] = entry(2, qd, k, jd * ni + id);
    }
  }
  pdl_entry();
  if (has_t) {
    const int i = it, j = jt, q = qt;
    double v[4];
    double a = f2d(reinterpret_cast<const float*>(z0 + ws_bpos(i, j, Mp))[q]);
    if (SECOND) a += f2d(reinterpret_cast<const float*>(dz + ws_bpos(i, j, Mp))[q]);
    if (i < ni - 1) {
      load_z<SECOND>(z0, dz, ws_bpos(i + 1, j, Mp), v);
#pragma unroll
      for (int k = 0; k < 4; ++k) a -= E[k] * v[k];
    }
    if (j < nj - 1) {
      load_z<SECOND>(z0, dz, ws_bpos(i, j + 1, Mp), v);
#pragma unroll
      for (int k = 0; k < 4; ++k) a -= N[k] * v[k];
    }
    if (j == 0 && nw > 0 && i < nw && ni - 1 - i > i) {
      load_z<SECOND>(z0, dz, ws_bpos(ni - 1 - i, 0, Mp), v);
#pragma unroll
      for (int k = 0; k < 4; ++k) a -= entry(2, q, k, i) * v[k];
    }
    ts[q][ht] = a;
  }
  __syncthreads();
  if (has_d) {
    const int h = hd, q = qd, i = id, j = jd, lx = h % WD_X, ly = h / WD_X;
    double a = r - ts[q][h];
    if (i > 0) {
      const int w = lx > 0 ? h - 1 : OWN + WD_X + ly;
#pragma unroll
      for (int k = 0; k < 4; ++k) a += W[k] * ts[k][w];
    }
    if (j > 0 || (nw > 0 && i >= ni - nw && ni - 1 - i < i)) {
      const int s = ly > 0 ? h - WD_X : OWN + lx;
#pragma unroll
      for (int k = 0; k < 4; ++k) a += S[k] * ts[k][s];
    }
    reinterpret_cast<float*>(C + ws_fpos(i, j, Mp))[q] = d2f(a);
  }
}

// Blocks 1-4 of tb in FP32 in the layout of the sweep, as k_sgs_prep writes them (a row per thread).
__global__ void k_ws_skew(LevelDev L) {
  pdl_entry();
  const int x = blockIdx.x * blockDim.x + threadIdx.x, c = x >> 2, r = x & 3;
  if (c >= L.n) return;
  const int ni = L.ni, n = L.n, i = c % ni, j = c / ni, Mp = ws_steps(ni, L.nj);
  auto row = [&](int blk) {
    const double* b = L.tb + (size_t)(16 * blk + 4 * r) * n + c;
    return make_float4(d2f(b[0]), d2f(b[n]), d2f(b[2 * (size_t)n]), d2f(b[3 * (size_t)n]));
  };
  const int jl = j % WS_ROWS;
  const size_t strip = (size_t)(j / WS_ROWS) * Mp;
  float4* f = reinterpret_cast<float4*>(L.wsF) + (strip + i + jl) * WS_F4_STEP + 4 * jl + r;
  float4* b = reinterpret_cast<float4*>(L.wsB) + (strip + Mp - 1 - i - jl) * WS_F4_STEP + 4 * jl + r;
  const bool cut = L.nw > 0 && (i < L.nw || i >= ni - L.nw);
  const float4 s = row(2);
  f[0] = row(1);
  f[WS_F4_STEP / 2] = j > 0 || (cut && ni - 1 - i < i) ? s : make_float4(0.f, 0.f, 0.f, 0.f);
  if (j == 0 && cut && ni - 1 - i > i) reinterpret_cast<float4*>(L.wsCut)[4 * i + r] = s;
  b[0] = row(3);
  b[WS_F4_STEP / 2] = row(4);
}

// z = z0 (+ dz + dz2): the stage update u = u0 - alpha z (scaled by dt* for ARK), or z to the level's
// sweep vector (FP64 contexts: yz64; mixed: yz32).
__global__ void k_ws_finish(LevelDev L, const float4* z0, const float4* dz, const float4* dz2, int do_update, int aw,
                            double alpha, int mixed) {
  pdl_entry();
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= L.n) return;
  const int n = L.n, i = c % L.ni, j = c / L.ni;
  const size_t zp = ws_bpos(i, j, ws_steps(L.ni, L.nj));
  double z[4];
  ws_load64(z0, zp, z);
  for (const float4* more : {dz, dz2}) {
    if (!more) break;
    double d[4];
    ws_load64(more, zp, d);
#pragma unroll
    for (int q = 0; q < 4; ++q) z[q] += d[q];
  }
  if (do_update) {
    const double sc = aw ? alpha : alpha * L.dts[c];
    const size_t g = (size_t)(j + 2) * L.P + (i + 2);
#pragma unroll
    for (int q = 0; q < 4; ++q) L.u[q * (size_t)L.Gn + g] = fma(-sc, z[q], L.u0[q * (size_t)n + c]);
  } else if (mixed) {
#pragma unroll
    for (int q = 0; q < 4; ++q) L.yz32[q * (size_t)n + c] = d2f(z[q]);
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q) L.yz64[q * (size_t)n + c] = z[q];
  }
}

// ---------------------------------------------------------------- the exact preconditioner
// Block Gauss-Seidel iterations on the full first-order operator A = D + L + U (the "exact"
// preconditioner of section 5.4's tables is A^-1): x <- x + P^-1 (r - A x), each P^-1 one
// warp-strip sweep pair, converging to A^-1 r.  x accumulates in FP64 (cell-major, 4 per cell).

// x = (init ? 0 : x) + z0 (+ dz), z0 / dz skewed in the backward order
__global__ void k_ws_accum(LevelDev L, const float4* z0, const float4* dz, double* x, int init) {
  pdl_entry();
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= L.n) return;
  const int i = c % L.ni, j = c / L.ni;
  const size_t zp = ws_bpos(i, j, ws_steps(L.ni, L.nj));
  double v[4];
  ws_load64(z0, zp, v);
  if (dz) {
    double d[4];
    ws_load64(dz, zp, d);
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] += d[q];
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) x[4 * (size_t)c + q] = (init ? 0.0 : x[4 * (size_t)c + q]) + v[q];
}

// D^-1 (r - A x) = D^-1 r - x + G_W x_W + G_S x_S + H_E x_E + H_N x_N (+ G_S x_mirror on row 0 of
// the wake cut, either side), as the next sweep's right-hand side (skewed, FP32)
template <typename T>
__global__ void k_ws_exact_defect(LevelDev L, const T* tb, const double* rhs, const double* x, float4* C) {
  pdl_entry();
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= L.n) return;
  const int ni = L.ni, nj = L.nj, n = L.n, i = c % ni, j = c / ni;
  double r[4], acc[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) r[k] = rhs[(size_t)k * n + c];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    double a = -x[4 * (size_t)c + q];
#pragma unroll
    for (int k = 0; k < 4; ++k) a += to64(tb[(size_t)(4 * q + k) * n + c]) * r[k];
    acc[q] = a;
  }
  auto add = [&](int blk, int cn) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int k = 0; k < 4; ++k) acc[q] += to64(tb[(size_t)(blk * 16 + 4 * q + k) * n + c]) * x[4 * (size_t)cn + k];
  };
  if (i > 0) add(1, c - 1);
  if (j > 0) add(2, c - ni);
  else if (L.nw > 0 && (i < L.nw || i >= ni - L.nw)) add(2, ni - 1 - i);
  if (i < ni - 1) add(3, c + 1);
  if (j < nj - 1) add(4, c + ni);
  const int b = j / WS_ROWS, jl = j % WS_ROWS, Mp = ws_steps(ni, L.nj);
  C[((size_t)b * Mp + (i + jl)) * WS_ROWS + jl] = make_float4(d2f(acc[0]), d2f(acc[1]), d2f(acc[2]), d2f(acc[3]));
}

// the stage update (or the result vector) from the accumulated x
__global__ void k_ws_finish_x(LevelDev L, const double* x, int do_update, int aw, double alpha, int mixed) {
  pdl_entry();
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= L.n) return;
  const int n = L.n, i = c % L.ni, j = c / L.ni;
  if (do_update) {
    const double sc = aw ? alpha : alpha * L.dts[c];
    const size_t g = (size_t)(j + 2) * L.P + (i + 2);
#pragma unroll
    for (int q = 0; q < 4; ++q) L.u[q * (size_t)L.Gn + g] = L.u0[q * (size_t)n + c] - sc * x[4 * (size_t)c + q];
  } else if (mixed) {
#pragma unroll
    for (int q = 0; q < 4; ++q) L.yz32[q * (size_t)n + c] = float(x[4 * (size_t)c + q]);
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q) L.yz64[q * (size_t)n + c] = x[4 * (size_t)c + q];
  }
}

constexpr size_t kWsSmemMax = 227 * 1024;
constexpr int kWsPortable = 8, kWsCluster = 16;  // CTAs of a cluster: portable, and the most sm_103 allows

// The kernel's per-device attributes, set once on each device (idempotent if two host threads race
// on the first launch).
template <int NS, bool TWO>
void ws_attributes() {
  static std::atomic<unsigned long long> done{0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64 || (done.load() & (1ull << dev))) return;
  if (cudaFuncSetAttribute(k_sweep_ws<NS, TWO>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWsSmemMax) ==
          cudaSuccess &&
      cudaFuncSetAttribute(k_sweep_ws<NS, TWO>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess)
    done.fetch_or(1ull << dev);
}

// The strips of one sweep wait on one another, so they are launched as one thread-block cluster
// (two strips per CTA): the hardware schedules a cluster's CTAs together, so every strip is
// resident whatever else runs beside it (concurrent cases of a batch included).
template <int NS, bool TWO>
cudaLaunchConfig_t ws_config(const LevelDev& L, cudaLaunchAttribute* at, cudaStream_t st) {
  const int nb = (ws_strips(L.nj) + 1) / 2;
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = !t_ordered;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = nb;
  at[1].val.clusterDim.y = 1;
  at[1].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(nb);
  cfg.blockDim = dim3(WS_THREADS);
  cfg.dynamicSmemBytes = ws_cta_bytes<NS, TWO>(ws_steps(L.ni, L.nj), L.nw);
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  return cfg;
}

template <int NS, bool TWO>
cudaError_t ws_sweep_launch(const LevelDev& L, float4* zout, int* err, long long limit, cudaStream_t st) {
  ws_attributes<NS, TWO>();
  cudaLaunchAttribute at[2];
  const cudaLaunchConfig_t cfg = ws_config<NS, TWO>(L, at, st);
  return cudaLaunchKernelEx(&cfg, k_sweep_ws<NS, TWO>, L, reinterpret_cast<const float4*>(L.wsF),
                            reinterpret_cast<const float4*>(L.wsB), reinterpret_cast<const float4*>(L.wsC),
                            reinterpret_cast<float4*>(L.wsY), static_cast<const float*>(L.wsCut), zout, err, limit);
}

// The forms in order of speed: an edge buffer per pass (1024x256 pair 162 us; with one, cleared between
// the passes, 3 % more), a ring of five stages (three: 1-3 % slower).
struct WsForm {
  int stages;
  bool two;
  size_t (*bytes)(int Mp, int nw);
  cudaLaunchConfig_t (*config)(const LevelDev&, cudaLaunchAttribute*, cudaStream_t);
  void (*attributes)();
  const void* kernel;
  cudaError_t (*launch)(const LevelDev&, float4*, int*, long long, cudaStream_t);
};

template <int NS, bool TWO>
WsForm form_of() {
  return {NS,
          TWO,
          [](int Mp, int nw) { return ws_cta_bytes<NS, TWO>(Mp, nw); },
          ws_config<NS, TWO>,
          ws_attributes<NS, TWO>,
          reinterpret_cast<const void*>(k_sweep_ws<NS, TWO>),
          ws_sweep_launch<NS, TWO>};
}

const WsForm kWsForms[] = {form_of<WS_STAGES, true>(), form_of<WS_STAGES, false>(), form_of<WS_SHALLOW, true>(),
                           form_of<WS_SHALLOW, false>()};

// whether the device can hold the cluster of this form's launch
bool ws_cluster_fits(const WsForm& f, int ni, int nj, int nw) {
  LevelDev L = {};
  L.ni = ni;
  L.nj = nj;
  L.nw = nw;
  f.attributes();
  cudaLaunchAttribute at[2];
  const cudaLaunchConfig_t cfg = f.config(L, at, nullptr);
  int n = 0;
  const cudaError_t e = cudaOccupancyMaxActiveClusters(&n, f.kernel, &cfg);
  if (e != cudaSuccess) cudaGetLastError();  // not this call's error: the level takes another form
  return e == cudaSuccess && n >= 1;
}

}  // namespace

// One cluster per sweep: at most 16 CTAs of two strips, a ring and an edge buffer that fit in shared
// memory, and (beyond the portable 8 CTAs) a device that can hold such a cluster.  The question is asked for
// the very form that is launched: at 1024x256 the deepest takes 176 KB a CTA and 16 SMs, the shallowest 103 KB
// and 8.
int ws_form(int ni, int nj, int nw, bool deep, long long cluster_bytes) {
  const int nb = (ws_strips(nj) + 1) / 2;
  if (nb > kWsCluster) return -1;
  for (int k = 0; k < 4; ++k) {
    const WsForm& f = kWsForms[k];
    const size_t bytes = f.bytes(ws_steps(ni, nj), nw);
    if ((f.stages > WS_SHALLOW && !deep) || bytes > kWsSmemMax) continue;
    if (nb <= kWsPortable || (cluster_bytes > 0 ? (long long)bytes <= cluster_bytes : ws_cluster_fits(f, ni, nj, nw)))
      return k;
  }
  return -1;
}

void ws_form_shape(int ni, int nj, int nw, int form, int* stages, int* edges, long long* bytes) {
  *stages = form < 0 ? 0 : kWsForms[form].stages;
  *edges = form < 0 ? 0 : kWsForms[form].two ? 2 : 1;
  *bytes = form < 0 ? 0 : (long long)kWsForms[form].bytes(ws_steps(ni, nj), nw);
}

int launch_ws_sweep(const LevelDev& L, int mixed, int refine, int do_update, int aw, double alpha, const double* rhs,
                    int* err, long long limit, cudaStream_t st, int exact_iters, bool deep, WsPending* pending) {
  const WsForm& form = kWsForms[L.wsForm[deep]];
  auto sweep = [&](float4* zout) { return form.launch(L, zout, err, limit, st); };
  const int g = (L.n + 127) / 128;
  float4* z0 = reinterpret_cast<float4*>(L.wsZ);
  float4* dz = z0 + ws_vec_floats(L.ni, L.nj) / 4;
  float4* dz2 = dz + ws_vec_floats(L.ni, L.nj) / 4;
  int launches = 0;
  const bool split = L.n <= WS_SPLIT_CELLS;
  const int g4 = (4 * L.n + 127) / 128;  // one thread per cell and row
  float4* wC = reinterpret_cast<float4*>(L.wsC);
  const double* tb64 = static_cast<const double*>(L.tb);
  double* noR = nullptr;
  if (rhs) {
    if (mixed) {
      const float* tb32 = reinterpret_cast<const float*>(L.tb);
      if (split)
        launch_pdl(k_ws_rhs<float, true>, g4, 128, 0, st, L, tb32, rhs, wC, noR);
      else
        launch_pdl(k_ws_rhs<float, false>, g, 128, 0, st, L, tb32, rhs, wC, noR);
    } else if (split) {
      launch_pdl(k_ws_rhs<double, true>, g4, 128, 0, st, L, tb64, rhs, wC, L.wsR);
    } else {
      launch_pdl(k_ws_rhs<double, false>, g, 128, 0, st, L, tb64, rhs, wC, L.wsR);
    }
    ++launches;
  }
  sweep(z0);
  ++launches;
  const bool corr = refine > 0 && !mixed;
  if (!corr || refine < 2) dz2 = nullptr;
  const float4 *z0c = z0, *none = nullptr;
  auto correct = [&](auto second, float4* out) {
    constexpr bool SECOND = decltype(second)::value;
    const float4* dzc = SECOND ? dz : none;
    const double *wT = L.wsT, *wR = L.wsR;
    if (split) {
      launch_pdl(k_ws_defect<SECOND>, dim3((L.ni + WD_X - 1) / WD_X, (L.nj + WD_Y - 1) / WD_Y), WD_THREADS, 0, st, L,
                 tb64, wR, z0c, dzc, wC);
    } else {
      launch_pdl(k_ws_defect_t<SECOND>, g, 128, 0, st, L, tb64, z0c, dzc, L.wsT);
      launch_pdl(k_ws_defect_d, g, 128, 0, st, L, tb64, wR, wT, wC);
      ++launches;
    }
    sweep(out);
    launches += 2;
  };
  if (corr) correct(std::false_type{}, dz);
  if (dz2) correct(std::true_type{}, dz2);
  if (exact_iters > 0) {
    launch_pdl(k_ws_accum, g, 128, 0, st, L, static_cast<const float4*>(z0),
               corr ? static_cast<const float4*>(dz) : nullptr, L.wsX, 1);
    ++launches;
    for (int it = 0; it < exact_iters; ++it) {
      if (mixed)
        launch_pdl(k_ws_exact_defect<float>, g, 128, 0, st, L, reinterpret_cast<const float*>(L.tb), rhs,
                   static_cast<const double*>(L.wsX), reinterpret_cast<float4*>(L.wsC));
      else
        launch_pdl(k_ws_exact_defect<double>, g, 128, 0, st, L, static_cast<const double*>(L.tb), rhs,
                   static_cast<const double*>(L.wsX), reinterpret_cast<float4*>(L.wsC));
      sweep(z0);
      launch_pdl(k_ws_accum, g, 128, 0, st, L, static_cast<const float4*>(z0), nullptr, L.wsX, 0);
      launches += 3;
    }
    launch_pdl(k_ws_finish_x, g, 128, 0, st, L, static_cast<const double*>(L.wsX), do_update, aw, alpha, mixed);
    return launches + 1;
  }
  if (pending) {
    *pending = WsPending{z0, corr ? dz : nullptr, dz2, alpha, aw};
    return launches;
  }
  launch_pdl(k_ws_finish, g, 128, 0, st, L, z0c, corr ? static_cast<const float4*>(dz) : none,
             static_cast<const float4*>(dz2), do_update, aw, alpha, mixed);
  return launches + 1;
}

void launch_ws_skew(const LevelDev& L, cudaStream_t st) {
  launch_pdl(k_ws_skew, (4 * L.n + 127) / 128, 128, 0, st, L);
}

size_t ws_floats(int ni, int nj) { return (size_t)ws_strips(nj) * ws_steps(ni, nj) * WS_F4_STEP * 4; }
size_t ws_vec_floats(int ni, int nj) { return (size_t)ws_strips(nj) * ws_steps(ni, nj) * WS_ROWS * 4; }

}  // namespace fasw

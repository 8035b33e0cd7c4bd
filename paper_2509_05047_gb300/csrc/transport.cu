// transport.cu -- fused emission -> Woodcock transport -> detection -> LUT
// weight -> LOR/TOF binning kernel (Sec. 2.2.1-2.2.3 of the paper; the
// simulator itself is the project's own design).
//
// A history is a small state machine:
//
//   EMIT -> STEP <-> {COMPTON, RAYLEIGH} -> ESCAPE -> (photon B) STEP ...
//        -> ESCAPE -> COINC -> next history
//
// Each warp owns a pool of kSlotsPerWarp photon slots whose state lives in
// shared memory (the fields only emission, detection and coincidence touch
// live in an L2-resident global buffer instead, which leaves room for 32
// warps per SM).  Every loop iteration the warp picks the section that the
// most slots wait for (weighting sections by their cost was measured slower,
// since it runs sections on fewer lanes), packs up to 32 slots in that state
// onto its 32 lanes, and runs the section once.  With three times as many
// slots as lanes the chosen section nearly fills the warp, where one history
// per lane left most lanes idle (the states of 32 histories spread over six
// sections).  The code holds a single copy of each section, and one
// rejection-sampling try runs per iteration.  Pools stay per warp, so warps
// never wait on each other: pools shared by two warps (barrier-coupled)
// measured slower on this issue-bound loop.
//
// Random numbers: a history's sub-streams (0: emission + TOF blur, 1: photon
// A, 2: photon B) are read through the slot's copy of the stream's last
// Philox block; a section that reads more words than are left draws one more
// block (emission draws its two blocks itself).  The words consumed, and
// their order, are those of the per-history definition, so results do not
// depend on the schedule, the slot or the lane.
//
// A history adds one fixed-point weight to the int64 accumulator or nothing
// (Sec. 2.2.3: weighted or discarded, never duplicated); lanes of a warp
// that hit the same bin combine their weights before one atomic.
#include "psc_internal.h"

namespace psc {

enum : int {
  kEmit = 0, kStep = 1, kCompton = 2, kRayleigh = 3, kEscape = 4, kCoinc = 5
};

// Slots per warp: the fuller the sections run, the fewer iterations a history
// takes.  96 is what 15 words a slot leave room for beside the tables at 32
// warps per SM; with 64 slots of 23 words the paper-scale torso, 1e9 histories,
// took 88.9 ms (97.8 warp instructions a history), with these 76.1 (65.8).
constexpr int kSlotsPerWarp = 96;
constexpr int kSlotsPerLane = kSlotsPerWarp / 32;

// A photon slot's state in shared memory, as arrays over the CTA's slots.
// The loop is bound by issue slots, so a section moves its fields in 16-byte
// accesses: 5 loads and 3 stores a Woodcock step.
//   pos   {x, y, z, path}                        float4
//   dir   {dx, dy, dz, energy}                   float4
//   ring  the last Philox block of the stream    uint4
//   kc    {stream position, counts}              uint2
//   meta  section and flags (read by the vote)   uint32
constexpr size_t kSlotBytes = 16 + 16 + 16 + 8 + 4;
// kc.x = words left | blocks generated << 3 | rejection tries << 25: word i of
// the section (i < words left) is ring[(i - left) & 3].  A section draws at
// most one block, when fewer words are left than it reads, and then leaves at
// most 4 of them unread.
// kc.y = steps | interactions << 16; listmode runs flag a Rayleigh interaction
// in bit 15 (steps stay below 2^15)
constexpr uint32_t kKcBlock = 1u << 3, kKcTry = 1u << 25;
__host__ __device__ constexpr uint32_t kc_left(uint32_t k) { return k & 7u; }
// meta = section | photon << 3 | stream << 4 | kMetaNeeds | kMetaNextMiss |
// material of a pending Rayleigh event << 8 | history of the work item << 16
__host__ __device__ constexpr uint32_t meta(int state, int photon, int stream) {
  return (uint32_t)state | (uint32_t)photon << 3 | (uint32_t)stream << 4;
}

// fields written only at emission, detection and coincidence, in an
// L2-resident global buffer: vector f of slot g of CTA b at
// cold[(b * kColdVecs + f) * n_slots + g]
enum : int {
  C_E0,    // emission point, voxel (listmode)
  C_D0,    // the first photon's emission direction, its path
  C_A,     // first photon at the detector: crystal | ring << 16 | scattered << 31, energy, nx, ny
  C_AD,    // its direction, its LUT position tpos | apos << 16 (scanners with gaps)
  C_B,     // second photon: crystal | ring << 16, nx, ny, LUT position
  C_LM,    // listmode: first photon's z, second photon's z, first photon's counts >> 15
  kColdVecs
};
// Production launches (kDebug false) only add weights: a history that cannot
// reach the accumulator may end as soon as that is certain, and its photons
// may be followed in either order (their streams are independent and the
// coincidence is symmetric in them).  EMIT therefore intersects the emission
// line with the detector cylinder once for both photons:
//   - a photon whose straight line leaves the cylinder axially, by more than
//     a margin far above the FP32 error of the tracked position, is lost
//     unless it interacts (kMetaNeeds).  Likewise the second photon when
//     the first arrived unscattered and trues are not binned.  Such a photon
//     ends its history where it leaves the grid, without a detection pass;
//   - the photon that is less likely to be detected goes first: the one
//     flying towards the nearer axial end when a line misses, else the one
//     with the longer way through the phantom.
// Measured on the paper-scale torso, 1e9 histories: 101.7 -> 88.9 ms; the same
// scanner with gaps and energy resolution, 1e8: 12.32 -> 9.76 ms.
constexpr uint32_t kMetaNeeds = 1u << 6;     // the photon in flight is lost unless it interacts
constexpr uint32_t kMetaNextMiss = 1u << 7;  // the second photon's straight line misses
constexpr int kMetaMaterial = 8, kMetaHistory = 16;
// the margin covers positions after this many steps (make_job)
constexpr uint32_t kMaxStraightSteps = 64;


// 1 << s, and 0 for s >= 32 (the PTX shift clamps its amount to the width)
__device__ __forceinline__ unsigned shl_or_zero(unsigned s) {
  unsigned d;
  asm("shl.b32 %0, %1, %2;" : "=r"(d) : "r"(1u), "r"(s));
  return d;
}

// per-half maximum of two pairs of unsigned 16-bit values
__device__ __forceinline__ unsigned umax16x2(unsigned a, unsigned b) {
  unsigned d;
  asm("max.u16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}

__device__ __forceinline__ float interp_scalar(const float* t, int n_tab, int e0, float e) {
  const float fe = e - (float)e0;
  const int i = max(0, min((int)fe, n_tab - 2));
  const float f = fe - (float)i;
  const float a = t[i], b = t[i + 1];
  return a + f * (b - a);
}

__device__ __forceinline__ float4 interp_xs(const float4* t, int n_tab, int e0, float e) {
  const float fe = e - (float)e0;
  const int i = max(0, min((int)fe, n_tab - 2));
  const float f = fe - (float)i;
  const float4 a = t[i], b = t[i + 1];
  return make_float4(a.x + f * (b.x - a.x), a.y + f * (b.y - a.y), a.z + f * (b.z - a.z), 0.0f);
}

__device__ __forceinline__ long long bin_key(const ScannerParams& S, int ca, int cb, int ra, int rb,
                                             float delta) {
  const int N = S.n_crystals;
  int f = ca + cb, s = 1;
  if (f >= N) {
    f -= N;
    s = -1;
  }
  const int view = f >> 1;
  const int r = s * (N / 2 - (cb - ca)) + N / 2 - 1 - S.rad_off;
  if (r < 0 || r >= S.n_rad) return -1;
  const float g = floorf(delta * S.inv_tof_bin + S.tof_half);
  if (!(g >= 0.0f && g < (float)S.n_tof)) return -1;
  const int plane = ra * S.n_rings + rb;
  return (((long long)plane * S.n_views + view) * S.n_rad + r) * S.n_tof + (int)g;
}

// Gaps between modules and blocks (Sec. 2.2.1-2.2.2).  A photon in a gap
// goes to the crystal at the gap's low (p) or high (1 - p) edge, p the
// relative probability that it is absorbed in the block on the low side:
// its straight line, at slope s = tan(theta) and cos(theta) = c against the
// radial direction, enters the blocks (depth D, faces doi below the
// detection cylinder, gap centred at x = 0, the photon at x0) and is
// absorbed in the first block it crosses with 1 - e^{-mu l1}, in the other
// with e^{-mu l1} (1 - e^{-mu l2}).  Crossing neither, the nearer side.
__device__ __forceinline__ float edge_prob(const ScannerParams& S, float x0, float s, float c, float gap) {
  float l1 = 0.0f, l2 = 0.0f;  // path lengths in the low and high block
  if (s != 0.0f) {
    const float ya = S.doi + (-0.5f * gap - x0) / s, yb = S.doi + (0.5f * gap - x0) / s;
    if (s > 0.0f) {  // the low block is crossed near the face, the high one deeper
      l1 = fmaxf(0.0f, fminf(S.depth, ya)) / c;
      l2 = fmaxf(0.0f, S.depth - fmaxf(0.0f, yb)) / c;
    } else {
      l2 = fmaxf(0.0f, fminf(S.depth, yb)) / c;
      l1 = fmaxf(0.0f, S.depth - fmaxf(0.0f, ya)) / c;
    }
  }
  const float first = s > 0.0f ? l1 : l2, second = s > 0.0f ? l2 : l1;
  const float pf = -expm1f(-S.mu * first);
  const float ps = expf(-S.mu * first) * -expm1f(-S.mu * second);
  const float p1 = s > 0.0f ? pf : ps, p2 = s > 0.0f ? ps : pf;
  if (!(p1 + p2 > 0.0f)) return x0 < 0.0f ? 1.0f : (x0 > 0.0f ? 0.0f : 0.5f);
  return p1 / (p1 + p2);
}

// LUT position and crystal of a detected photon on a scanner with gaps.
// Module m spans azimuth [m mod_phi, (m + 1) mod_phi) as [half gap | module_t
// crystals | half gap], block b the axial range [b blk_pitch, (b + 1)
// blk_pitch) in the same way.  Returns crystal | ring << 16 | lost << 31 in
// the low word (lost: in a gap, gap_mode 1) and tpos | apos << 16 in the high
// word.  Gap_mode 2 assigns a photon in a transaxial gap with u0, then one in
// an inner axial gap with the next of (u0, u1); at the scanner's axial ends
// only one block borders the gap.
__device__ __noinline__ unsigned long long place(const ScannerParams& S, float phi, float hz, float dx, float dy,
                                                 float dz, float nx, float ny, float u0, float u1) {
  const int m = min((int)floorf(phi * S.inv_mod_phi), S.n_mod - 1);
  const float u = phi - (float)m * S.mod_phi;
  int tp, bt = 0, cr = 0;
  float xt = 0.0f;
  if (u < 0.5f * S.gap_gamma) {
    tp = 0;
    bt = m;
    xt = u * S.radius;
  } else if (u >= S.mod_phi - 0.5f * S.gap_gamma) {
    tp = S.module_t + 1;
    bt = m + 1;
    xt = (u - S.mod_phi) * S.radius;
  } else {
    const int j = max(0, min((int)floorf((u - 0.5f * S.gap_gamma) * S.inv_crys_phi), S.module_t - 1));
    tp = j + 1;
    cr = m * S.module_t + j;
  }
  const float z = hz + S.half_len;
  const int b = max(0, min((int)floorf(z * S.inv_blk_pitch), S.n_blk - 1));
  const float w = z - (float)b * S.blk_pitch;
  int al, ba = 0, rg = 0;
  float xa = 0.0f;
  if (w < 0.5f * S.gap_a) {
    al = 0;
    ba = b;
    xa = w;
  } else if (w >= S.blk_pitch - 0.5f * S.gap_a) {
    al = S.module_a + 1;
    ba = b + 1;
    xa = w - S.blk_pitch;
  } else {
    const int j = max(0, min((int)floorf((w - 0.5f * S.gap_a) * S.inv_ring_w), S.module_a - 1));
    al = j + 1;
    rg = b * S.module_a + j;
  }
  const unsigned long long pos = (unsigned long long)((uint32_t)tp | (uint32_t)(b * (S.module_a + 2) + al) << 16)
                                 << 32;
  const bool gt = tp == 0 || tp == S.module_t + 1, ga = al == 0 || al == S.module_a + 1;
  if (S.gap_mode == 1) return pos | (gt || ga ? 1ull << 31 : 0ull) | (uint32_t)cr | (uint32_t)rg << 16;
  const float dn = dx * nx + dy * ny, dt = -dx * ny + dy * nx;
  if (gt) {
    const float p1 = edge_prob(S, xt, dt / dn, dn * rsqrtf(dn * dn + dt * dt), S.gap_t_mm);
    const int c0 = bt * S.module_t;
    cr = u0 < p1 ? (c0 == 0 ? S.n_crystals - 1 : c0 - 1) : (c0 == S.n_crystals ? 0 : c0);
  }
  if (ga) {
    if (ba == 0) {
      rg = 0;
    } else if (ba == S.n_blk) {
      rg = S.n_rings - 1;
    } else {
      const float p1 = edge_prob(S, xa, dz / dn, dn * rsqrtf(dn * dn + dz * dz), S.gap_a);
      rg = (gt ? u1 : u0) < p1 ? ba * S.module_a - 1 : ba * S.module_a;
    }
  }
  return pos | (uint32_t)cr | (uint32_t)rg << 16;
}

// incidence angles (degrees) of direction d at the hit with radial unit
// vector (nx, ny): transaxial atan2(d.t, d.n), axial atan2(d_z, d.n)
__device__ __forceinline__ void angles(float nx, float ny, float3 d, float& alpha, float& beta) {
  const float dn = d.x * nx + d.y * ny;
  const float dt = -d.x * ny + d.y * nx;
  alpha = atan2f(dt, dn) * 57.29577951308232f;
  beta = atan2f(d.z, dn) * 57.29577951308232f;
}


// kDebug: statistics counters and per-history listmode outputs are compiled
// in only when a launch asks for them, so the production loop stays small.
// kOneJob (production launches of a single job with an f32 LUT, the common
// case): the job's index in the kernel parameter space is the constant 0.
// kFixed (production launches of 512-thread CTAs, the default): the slot
// count is a compile-time constant, so every slot field access is an
// immediate offset from the slot's address (measured 10 % faster).
template <int DT, bool kDebug, bool kOneJob = false, bool kFixed = false>
__global__ void __launch_bounds__(512, 2) transport_kernel(const __grid_constant__ BatchParams B) {
  extern __shared__ float4 smem[];
  const unsigned tid = threadIdx.x, bdim = blockDim.x;
  const int n_slots = kFixed ? 16 * kSlotsPerWarp : (int)(bdim >> 5) * kSlotsPerWarp;
  float4* s_pos = smem;
  float4* s_dir = s_pos + n_slots;
  uint4* s_ring = reinterpret_cast<uint4*>(s_dir + n_slots);
  uint2* s_kc = reinterpret_cast<uint2*>(s_ring + n_slots);
  uint32_t* s_meta = reinterpret_cast<uint32_t*>(s_kc + n_slots);
  float4* s_xs = reinterpret_cast<float4*>(s_meta + n_slots);  // the job's tables (n_slots is a multiple of 96)
  __shared__ int s_j;
  __shared__ unsigned long long s_lo;         // first history of the chunk
  __shared__ unsigned s_len, s_next;          // chunk length, next offset to hand out
  __shared__ unsigned long long s_cnt[kStatCount];
  __shared__ uint16_t s_sel[16][32];          // per warp: slot of each lane this iteration
  for (int i = tid; i < kStatCount; i += bdim) s_cnt[i] = 0;
  const unsigned lane_id = tid & 31u;
  const int warp = (int)(tid >> 5);
  const int g0 = warp * kSlotsPerWarp + (int)lane_id;  // this lane refills slots g0, g0 + 32, g0 + 64
  const bool stats = kDebug && B.stats != nullptr;
  int cached = -1;
  uint4* cold = B.cold + (size_t)blockIdx.x * kColdVecs * n_slots;
  auto setC = [&](int f, int g, float x, float y, float z, uint32_t w) {
    cold[f * n_slots + g] = make_uint4(__float_as_uint(x), __float_as_uint(y), __float_as_uint(z), w);
  };

  for (;;) {
    // ---- fetch the next chunk of (job, history range) ----
    if (tid == 0) {
      const unsigned long long c = atomicAdd(B.next_chunk, 1ull);
      int j = -1;
      if (c < B.chunk_end[B.n_jobs - 1]) {
        j = 0;
        while (B.chunk_end[j] <= c) ++j;
        const unsigned long long c0 = j ? B.chunk_end[j - 1] : 0ull;
        const unsigned long long lo = B.jobs[j].first + (c - c0) * B.jobs[j].chunk;
        const unsigned long long hi = B.jobs[j].first + B.jobs[j].n;
        s_lo = lo;
        s_len = (unsigned)min(B.jobs[j].chunk, hi - lo);
        s_next = 0;
      }
      s_j = j;
    }
    __syncthreads();
    const int jcur = s_j;
    if (jcur < 0) break;
    const ListmodeOut lm = kDebug ? B.lm[jcur] : ListmodeOut{nullptr, nullptr, 0};
    if (jcur != cached) {  // stage the job's phantom tables
      const PhantomParams& pg = B.jobs[jcur].ph;
      const int n_xs = pg.n_mat * pg.n_tab;
      float* s_maj = reinterpret_cast<float*>(s_xs + n_xs);
      float* s_kappa = s_maj + pg.n_tab;
      for (int i = tid; i < n_xs; i += bdim) {
        const int mm = i / pg.n_tab, kk = i - mm * pg.n_tab;
        s_xs[i] = pg.xs[mm * pg.n_e + pg.e0 + kk];
      }
      for (int i = tid; i < pg.n_tab; i += bdim) s_maj[i] = pg.maj[pg.e0 + i];
      if (tid < (unsigned)kMaxMaterials) s_kappa[tid] = (int)tid < pg.n_mat ? pg.kappa[tid] : 0.0f;
      cached = jcur;
    }
    __syncthreads();

    // the job's parameters, read from the kernel parameter space (a
    // compile-time index for single-job launches, the CTA-uniform chunk's job
    // otherwise): operands of the instructions, not registers held across the
    // loop (a shared-memory copy made the multi-job instantiations spill)
    const Job& J = [&]() -> const Job& {
      if constexpr (kOneJob) return B.jobs[0];
      else return B.jobs[jcur];
    }();
    const PhantomParams& ph = J.ph;
    const ScannerParams& S = J.sc;
    const float* s_maj = reinterpret_cast<const float*>(s_xs + ph.n_mat * ph.n_tab);
    const float* s_kappa = s_maj + ph.n_tab;
    const uint2 key = make_uint2((uint32_t)J.seed, (uint32_t)(J.seed >> 32));
    const bool blur = S.tof_sigma > 0.0f;

    // warp-aggregated counter increment (lanes of the calling branch)
    auto count = [&](bool pred, int slot) {
      if (!stats) return;
      const unsigned act = __activemask();
      const unsigned b = __ballot_sync(act, pred);
      if (b && lane_id == (unsigned)(__ffs(act) - 1)) atomicAdd(&s_cnt[slot], (unsigned long long)__popc(b));
    };
    // a listmode launch records the history that ends in a slot: its class, bin and weight
    auto record = [&](uint32_t m, int cls, long long key_out, long long q_out) {
      if (kDebug) {
        const unsigned long long h = s_lo + (m >> kMetaHistory);
        const unsigned long long i = (unsigned long long)dbg_idx(B.dbg, kSiteHistOut, (long long)(h - J.first),
                                                                 (long long)J.n);
        if (J.cls_out) J.cls_out[i] = (int8_t)cls;
        if (J.key_out) J.key_out[i] = key_out;
        if (J.q_out) J.q_out[i] = q_out;
        if (stats) atomicAdd(&s_cnt[kStatClass0 + cls], 1ull);
      }
    };

#pragma unroll
    for (int i = 0; i < kSlotsPerLane; ++i) s_meta[g0 + 32 * i] = kEmit;
    unsigned waiting = ~0u;  // without the EMIT count once the work item has handed out its last history
    __syncwarp();

    // words a section reads of its stream, one nibble per section: (EMIT draws its own),
    // 2, 4, 3, 0, 2.  Detection reads S.escape_words (energy blur 2, edge draws 2), at
    // most 4: one block always covers what the ring lacks.
    constexpr uint32_t kNeedNibbles = 0x203420u;

    for (;;) {
      // ---- warp vote: the section that the most slots wait for ----
      // slot counts per state, one byte each (at most 96 slots): states 0..3
      // in lo, 4..7 in hi (sections 4, 5 in its bytes 0, 1), summed over the
      // warp by two reductions.  A state's bit is 1 << 8 st, or 1 << (8 st - 32)
      // in hi, where shift amounts of 32 and more (unsigned wrap included) give 0.
      int st[kSlotsPerLane];
      unsigned lo = 0, hi = 0;
#pragma unroll
      for (int i = 0; i < kSlotsPerLane; ++i) {
        st[i] = (int)(s_meta[g0 + 32 * i] & 7u);
        lo += shl_or_zero(8u * st[i]);
        hi += shl_or_zero(8u * st[i] - 32u);
      }
      const unsigned clo = __reduce_add_sync(0xffffffffu, lo) & waiting, chi = __reduce_add_sync(0xffffffffu, hi);
      if ((clo | (chi & 0xffffu)) == 0u) break;  // no slot holds a history, none is left to start
      // the most-populated section, the lowest on a tie: keys count << 3 | (7 - q)
      // in 16-bit halves, two paired maxima, then the larger half.  A section
      // with slots outranks every empty one (key >= 8), so sec is never empty.
      const unsigned k01 = __byte_perm(clo, 0u, 0x4140) * 8u + 0x00060007u;
      const unsigned k23 = __byte_perm(clo, 0u, 0x4342) * 8u + 0x00040005u;
      const unsigned k45 = __byte_perm(chi, 0u, 0x4140) * 8u + 0x00020003u;
      const unsigned km = umax16x2(umax16x2(k01, k23), k45);
      const unsigned kmax = max(km & 0xffffu, km >> 16);
      const int sec = 7 - (int)(kmax & 7u);
      // ---- pack up to 32 slots in that state onto the lanes ----
      const unsigned below = (1u << lane_id) - 1u;
      int n = 0;
#pragma unroll
      for (int i = 0; i < kSlotsPerLane; ++i) {
        const unsigned mask = __ballot_sync(0xffffffffu, st[i] == sec);
        const int r = n + __popc(mask & below);
        if (st[i] == sec && r < 32) s_sel[warp][r] = (uint16_t)(g0 + 32 * i);
        n += __popc(mask);
      }
      __syncwarp();
      const int g = lane_id < (kmax >> 3) ? (int)dbg_idx(B.dbg, kSiteSlot, s_sel[warp][lane_id], n_slots) : -1;
      __syncwarp();

      // In EMIT a slot takes the work item's next history, if there is one.  Loop control
      // has to be the same in all lanes, so the end of the item is voted on, from the
      // values that the lanes' own atomics returned: another warp may move s_next between
      // two lanes' reads of it.
      unsigned off = ~0u;
      if (sec == kEmit) {
        if (g >= 0) off = atomicAdd(&s_next, 1u);
        if (__any_sync(0xffffffffu, off + 1u >= s_len)) waiting = ~0xffu;
      }

      if (g >= 0) {
        uint32_t m = s_meta[g];
        auto history = [&]() -> unsigned long long { return s_lo + (m >> kMetaHistory); };
        auto block = [&](uint32_t nb, uint32_t stream) -> uint4 {
          const unsigned long long h = history();
          count(true, kStatRng);
          return philox4x32_10(make_uint4((uint32_t)h, (uint32_t)(h >> 32), nb, stream), key);
        };
        // ---- the section's random words r0 .. r3, from the ring and a new block ----
        uint2 kc = make_uint2(0u, 0u);
        uint32_t r0 = 0, r1 = 0, r2 = 0, r3 = 0;
        if (sec != kEmit) {
          kc = s_kc[g];
          uint32_t need = (kNeedNibbles >> (4 * sec)) & 15u;
          if (sec == kEscape) need = S.escape_words;  // energy blur, edge-crystal draws
          if (sec == kCoinc && !blur) need = 0;
          if (need) {
            const uint32_t left = kc_left(kc.x);
            const uint32_t* ring = reinterpret_cast<const uint32_t*>(s_ring + g);
            r0 = ring[(0u - left) & 3u];
            r1 = ring[(1u - left) & 3u];
            if (need > 2) {
              r2 = ring[(2u - left) & 3u];
              r3 = ring[(3u - left) & 3u];
            }
            if (left < need) {  // word i >= left is word i - left of the new block
              const uint4 b = block((kc.x >> 3) & 0x3fffffu, (m >> 4) & 3u);
              s_ring[g] = b;
              kc.x += kKcBlock + 4u;
              r3 = left == 0 ? b.w : left == 1 ? b.z : left == 2 ? b.y : b.x;
              r2 = left == 0 ? b.z : left == 1 ? b.y : left == 2 ? b.x : r2;
              r1 = left == 0 ? b.y : left == 1 ? b.x : r1;
              r0 = left == 0 ? b.x : r0;
            }
          }
        }
        auto set_section = [&](int state) { s_meta[g] = (m & ~7u) | (uint32_t)state; };
        // the slot's history ends: it waits in EMIT for the work item's next one
        auto finish = [&](int cls, long long key_out, long long q_out) {
          record(m, cls, key_out, q_out);
          s_meta[g] = kEmit;
        };

        // ---- emission (stream 0, words 0..6) ----
        const bool emitted = off < s_len;
        float4 pos, dir;
        if (emitted) {
          m = off << kMetaHistory;
          const uint4 b0 = block(0, 0), b1 = block(1, 0);
          const uint32_t w0 = b0.x, w1 = b0.y;
          const unsigned col = __umulhi(w0, (unsigned)ph.n_vox);  // n_vox < 2^31
          const uint2 at = __ldg(ph.alias + dbg_idx(B.dbg, kSiteAlias, col, ph.n_vox));
          const int v = ((w1 >> 9) < at.x) ? (int)col : (int)at.y;
          // v = (iz ny + iy) nx + ix: quotients from a multiply-high with floor(2^32 / d),
          // at most one below the true quotient, then one correction
          const unsigned nxy = (unsigned)(ph.nx * ph.ny);
          unsigned iz = __umulhi((unsigned)v, ph.m_nxy), rem = (unsigned)v - iz * nxy;
          if (rem >= nxy) {
            ++iz;
            rem -= nxy;
          }
          unsigned iy = __umulhi(rem, ph.m_nx), ix = rem - iy * (unsigned)ph.nx;
          if (ix >= (unsigned)ph.nx) {
            ++iy;
            ix -= (unsigned)ph.nx;
          }
          const float ex = ph.ox + ((float)ix + u01(b0.z)) * ph.dx, ey = ph.oy + ((float)iy + u01(b0.w)) * ph.dy,
                      ez = ph.oz + ((float)iz + u01(b1.x)) * ph.dz;
          const float ct = 2.0f * u01(b1.y) - 1.0f;
          float sp, cp;
          sincospif(2.0f * u01(b1.z), &sp, &cp);
          const float st = sqrtf(fmaxf(0.0f, 1.0f - ct * ct));
          float dx = st * cp, dy = st * sp, dz = ct;  // photon A's direction, then the first photon's
          uint32_t flags = meta(kStep, 0, 1);
          if (!kDebug) {
            // axial coordinates of the two straight hits, times a
            const float a = dx * dx + dy * dy, b = ex * dx + ey * dy, c = ex * ex + ey * ey - S.r2;
            const float sq = sqrtf(fmaxf(b * b - a * c, 0.0f)), za = ez * a, lim = J.miss_lim * a;
            const bool miss_a = fabsf(za + (sq - b) * dz) > lim, miss_b = fabsf(za - (sq + b) * dz) > lim;
            const bool b_first = (miss_a || miss_b) ? ez * dz < 0.0f : b > 0.0f;
            if (b_first) {
              dx = -dx;
              dy = -dy;
              dz = -dz;
              flags = meta(kStep, 0, 2);
            }
            if (b_first ? miss_b : miss_a) flags |= kMetaNeeds;
            if (b_first ? miss_a : miss_b) flags |= kMetaNextMiss;
          }
          setC(C_E0, g, ex, ey, ez, (uint32_t)v);
          setC(C_D0, g, dx, dy, dz, 0u);
          s_pos[g] = pos = make_float4(ex, ey, ez, 0.0f);
          s_dir[g] = dir = make_float4(dx, dy, dz, kEmitKeV);
          m |= flags;
          const uint4 b = block(0, (m >> 4) & 3u);
          s_ring[g] = b;
          kc = make_uint2(kKcBlock + 4u, 0u);
          r0 = b.x;
          r1 = b.y;
        }

        // ---- one Woodcock step (a new history takes its first one at once: a
        // vote, a pass over the slots and a reload of its state fewer) ----
        if (sec == kStep || emitted) {
          const uint32_t cnt = kc.y;
          if (!emitted) {
            pos = s_pos[g];
            dir = s_dir[g];
          }
          const float e = dir.w;
          const float mu_max = interp_scalar(s_maj, ph.n_tab, ph.e0, e);
          bool moved = false;
          if ((int)(cnt & 0x7fffu) >= kMaxSteps) {
            finish(kStepLimit, -1, 0);
          } else if (!(mu_max > 0.0f)) {
            // no word was read: with 5 of them left, the ring lacks the oldest; drop the block again
            if (kc_left(kc.x) > 4u) {
              reinterpret_cast<uint32_t*>(s_ring + g)[3] = r0;
              kc.x -= kKcBlock + 4u;
            }
            s_kc[g] = kc;
            set_section(kEscape);
          } else {
            const float px = pos.x, py = pos.y, pz = pos.z;
            const float dx = dir.x, dy = dir.y, dz = dir.z;
            const float dist = -__logf(u01(r0)) / mu_max;
            const float qx = px + dist * dx;
            const float qy = py + dist * dy;
            const float qz = pz + dist * dz;
            const float fx = (qx - ph.ox) * ph.inv_dx;
            const float fy = (qy - ph.oy) * ph.inv_dy;
            const float fz = (qz - ph.oz) * ph.inv_dz;
            // outside the grid is vacuum: straight to the detector, unless the photon
            // is certain to miss it (cnt below 2^16: it did not interact)
            int next = !kDebug && (m & kMetaNeeds) && cnt <= kMaxStraightSteps ? kEmit : kEscape;
            --kc.x;
            moved = fx >= 0.0f && fx < (float)ph.nx && fy >= 0.0f && fy < (float)ph.ny && fz >= 0.0f &&
                    fz < (float)ph.nz;
            if (moved) {
              const int ix = min((int)fx, ph.nx - 1);
              const int iy = min((int)fy, ph.ny - 1);
              const int iz = min((int)fz, ph.nz - 1);
              s_pos[g] = make_float4(qx, qy, qz, pos.w + dist);
              const float2 vx = __ldg(ph.vox + dbg_idx(B.dbg, kSiteVoxel, (unsigned)((iz * ph.ny + iy) * ph.nx + ix),
                                                       ph.n_vox));  // n_vox < 2^31
              const int mat = (int)dbg_idx(B.dbg, kSiteMaterial, __float_as_int(vx.y), ph.n_mat);
              const float4 cum = interp_xs(s_xs + mat * ph.n_tab, ph.n_tab, ph.e0, e);
              const float t = u01(r1) * mu_max;
              --kc.x;
              kc.y = cnt + 1u;
              next = t < vx.x * cum.x ? kCompton : t < vx.x * cum.y ? kRayleigh : t < vx.x * cum.z ? kEmit : kStep;
              if (next == kEmit) {
                count(true, kStatPhoto);
                record(m, kAbsorbed, -1, 0);
              }
              m = (m & ~(7u << kMetaMaterial)) | (uint32_t)mat << kMetaMaterial;  // travels with a Rayleigh event
            }
            s_kc[g] = kc;
            set_section(next);
          }
          count(moved, kStatSteps);
        }

        // ---- one Klein-Nishina try (Kahn's method on x = E/E') ----
        if (sec == kCompton) {
          const float u1 = u01(r0), u2 = u01(r1), u3 = u01(r2);
          kc.x -= 3u;
          const uint32_t tries = (kc.x >> 25) + 1u;
          const float4 dir = s_dir[g];
          const float e = dir.w;
          const float a = e / kRestKeV;
          const float two_a = 2.0f * a;
          float x, c;
          bool accept;
          if (u1 < (1.0f + two_a) / (9.0f + two_a)) {
            x = 1.0f + two_a * u2;
            c = 1.0f - (x - 1.0f) / a;
            accept = u3 < 4.0f * (1.0f / x - 1.0f / (x * x));
          } else {
            x = (1.0f + two_a) / (1.0f + two_a * u2);
            c = 1.0f - (x - 1.0f) / a;
            accept = u3 < 0.5f * (c * c + 1.0f / x);
          }
          count(true, kStatTries);
          kc.x += kKcTry;
          if (accept || (int)tries >= kMaxTries) {
            const float e1 = e / x;
            count(true, kStatCompton);
            kc.x = (kc.x & (kKcTry - 1u)) - 1u;
            kc.y += 1u << 16;
            if (e1 < S.e_kill) {
              finish(kEnergyWindow, -1, 0);
            } else {
              float3 d = make_float3(dir.x, dir.y, dir.z);
              rotate(d, c, u01(r3));
              s_dir[g] = make_float4(d.x, d.y, d.z, e1);
              set_section(kStep);
            }
          }
          s_kc[g] = kc;
        }

        // ---- one Rayleigh try (the material travels in meta) ----
        if (sec == kRayleigh) {
          const float u1 = u01(r0), u2 = u01(r1);
          kc.x -= 2u;
          const uint32_t tries = (kc.x >> 25) + 1u;
          const float4 dir = s_dir[g];
          const float e = dir.w;
          const float er = e / kRestKeV;
          const float b = s_kappa[dbg_idx(B.dbg, kSiteKappa, (m >> kMetaMaterial) & 7u, ph.n_mat)] * er * er;
          const float sv = u1 / (1.0f + b * (1.0f - u1));
          const float c = 1.0f - 2.0f * sv;
          count(true, kStatTries);
          if (u2 < 0.5f * (1.0f + c * c) || (int)tries >= kMaxTries) {
            float3 d = make_float3(dir.x, dir.y, dir.z);
            rotate(d, c, u01(r2));
            count(true, kStatRayleigh);
            s_dir[g] = make_float4(d.x, d.y, d.z, e);
            s_kc[g] = make_uint2((kc.x & (kKcTry - 1u)) - 1u, (kc.y + (1u << 16)) | (kDebug ? 0x8000u : 0u));
            set_section(kStep);
          } else {
            s_kc[g].x = kc.x + kKcTry;
          }
        }

        // ---- the photon reaches the detector cylinder ----
        if (sec == kEscape) {
          const float4 pos4 = s_pos[g], dir = s_dir[g];
          const float px = pos4.x, py = pos4.y, pz = pos4.z;
          const float dx = dir.x, dy = dir.y, dz = dir.z;
          const float e = dir.w;
          float path = pos4.w;
          const float a = dx * dx + dy * dy;
          int cls = kDetected, cr = 0, rg = 0;
          uint32_t pos = 0;  // LUT position tpos | apos << 16 (scanners with gaps)
          float nx = 0.0f, ny = 0.0f, hz_det = 0.0f;
          if (!(a > 0.0f)) {
            cls = kLostAxial;
          } else {
            const float b = px * dx + py * dy;
            const float c = px * px + py * py - S.r2;
            const float sq = sqrtf(fmaxf(b * b - a * c, 0.0f));
            const float t = (b >= 0.0f) ? (-c) / (b + sq) : (sq - b) / a;
            const float hx = px + t * dx, hy = py + t * dy, hz = pz + t * dz;
            hz_det = hz;
            path += t;
            if (!(hz >= -S.half_len && hz < S.half_len)) {
              cls = kLostAxial;
            } else {
              rg = max(0, min((int)floorf((hz + S.half_len) * S.inv_pitch), S.n_rings - 1));
              float phi = atan2f(hy, hx);
              if (phi < 0.0f) phi += 6.283185307179586f;
              cr = max(0, min((int)floorf(phi * S.crystals_per_radian), S.n_crystals - 1));
              nx = hx / S.radius;
              ny = hy / S.radius;
              float ed = e;  // the energy the window tests: blurred by the resolution, if any
              if (S.e_res_k > 0.0f) {
                ed = e + S.e_res_k * sqrtf(e) * (sqrtf(-2.0f * __logf(u01(r0))) * cospif(2.0f * u01(r1)));
              }
              if (ed < S.e_lo || ed > S.e_hi) cls = kEnergyWindow;
              if (S.gap_mode && cls == kDetected) {
                // two words cover both edge draws (the axial one is the second only after a
                // transaxial one); escape_words counts them
                const bool blurred = S.e_res_k > 0.0f;
                const float u0 = S.gap_mode == 2 ? u01(blurred ? r2 : r0) : 0.0f,
                            u1 = S.gap_mode == 2 ? u01(blurred ? r3 : r1) : 0.0f;
                const unsigned long long r = place(S, phi, hz, dx, dy, dz, nx, ny, u0, u1);
                if ((uint32_t)r >> 31) {
                  cls = kLostAxial;  // lost in a gap
                } else {
                  cr = (int)((uint32_t)r & 0xffffu);
                  rg = (int)(((uint32_t)r >> 16) & 0x7fffu);
                }
                pos = (uint32_t)(r >> 32);
              }
            }
          }
          count(cls == kDetected, kStatDetected);
          const uint32_t crg = (uint32_t)cr | (uint32_t)rg << 16;
          if (cls != kDetected) {
            finish(cls, -1, 0);
          } else if (((m >> 3) & 1u) == 0) {  // the first photon: keep it, launch the other one back to back
            const uint32_t nint = kc.y >> 16;
            cold[C_A * n_slots + g] = make_uint4(crg | (nint > 0 ? 1u << 31 : 0u), __float_as_uint(e),
                                                 __float_as_uint(nx), __float_as_uint(ny));
            setC(C_AD, g, dx, dy, dz, pos);
            if (kDebug && lm.out) cold[C_LM * n_slots + g] = make_uint4(__float_as_uint(hz_det), 0u, kc.y >> 15, 0u);
            const uint4 e0 = cold[C_E0 * n_slots + g], d0 = cold[C_D0 * n_slots + g];
            cold[C_D0 * n_slots + g].w = __float_as_uint(path);
            s_pos[g] = make_float4(__uint_as_float(e0.x), __uint_as_float(e0.y), __uint_as_float(e0.z), 0.0f);
            s_dir[g] = make_float4(-__uint_as_float(d0.x), -__uint_as_float(d0.y), -__uint_as_float(d0.z), kEmitKeV);
            s_kc[g] = make_uint2(0u, 0u);
            const bool needs = !kDebug && ((m & kMetaNextMiss) || (nint == 0 && !(J.bin_mask & PSC_BIN_TRUES)));
            s_meta[g] = meta(kStep, 1, 3 - (int)((m >> 4) & 3u)) | (needs ? kMetaNeeds : 0u) | (m & 0xffff0000u);
          } else if (cr == (int)(cold[C_A * n_slots + g].x & 0xffffu)) {
            finish(kSameCrystal, -1, 0);
          } else {
            setC(C_B, g, nx, ny, __uint_as_float(crg), pos);
            if (kDebug && lm.out) cold[C_LM * n_slots + g].y = __float_as_uint(hz_det);
            s_pos[g].w = path;
            // the TOF blur reads stream 0, block 2
            s_kc[g].x = 2u * kKcBlock;
            s_meta[g] = meta(kCoinc, 1, 0) | (m & 0xffff0000u);
          }
        }

        // ---- coincidence: TOF, LOR bin, LUT weight, accumulate ----
        if (sec == kCoinc) {
          const uint4 ca = cold[C_A * n_slots + g], cad = cold[C_AD * n_slots + g], cb = cold[C_B * n_slots + g];
          const float4 dir = s_dir[g];
          const uint32_t acrg = ca.x, bcrg = cb.z;
          const int a_cr = (int)(acrg & 0xffffu), a_rg = (int)((acrg >> 16) & 0x7fffu);
          const int b_cr = (int)(bcrg & 0xffffu), b_rg = (int)(bcrg >> 16);
          const float a_path = __uint_as_float(cold[C_D0 * n_slots + g].w), path = s_pos[g].w;
          const float a_e = __uint_as_float(ca.y), a_nx = __uint_as_float(ca.z), a_ny = __uint_as_float(ca.w);
          const float3 a_d = make_float3(__uint_as_float(cad.x), __uint_as_float(cad.y), __uint_as_float(cad.z));
          const float b_nx = __uint_as_float(cb.x), b_ny = __uint_as_float(cb.y);
          const bool a_first = a_cr < b_cr;
          float delta = 0.5f * (a_first ? a_path - path : path - a_path);
          if (blur) {
            const float gs = sqrtf(-2.0f * logf(u01(r0))) * cospif(2.0f * u01(r1));
            delta += S.tof_sigma * gs;
          }
          const long long key_ = a_first ? bin_key(S, a_cr, b_cr, a_rg, b_rg, delta)
                                         : bin_key(S, b_cr, a_cr, b_rg, a_rg, delta);
          const bool scattered = (acrg >> 31) != 0u || (kc.y >> 16) > 0u;
          const int cls = key_ < 0 ? kOutOfRange : scattered ? kScatter : kTrue;
          const bool take = cls == kScatter ? (J.bin_mask & 1) : cls == kTrue ? (J.bin_mask & 2) : false;
          long long q = 0;
          if (key_ >= 0 && (take || (kDebug && (J.q_out || lm.out)))) {
            float aa, ab, ba, bb;
            angles(a_nx, a_ny, a_d, aa, ab);
            angles(b_nx, b_ny, make_float3(dir.x, dir.y, dir.z), ba, bb);
            int a_tp = a_cr % S.module_t, a_ap = a_rg % S.module_a, b_tp = b_cr % S.module_t,
                b_ap = b_rg % S.module_a;
            if (S.gap_mode) {
              const uint32_t pa = cad.w, pb = cb.w;
              a_tp = (int)(pa & 0xffffu);
              a_ap = (int)(pa >> 16);
              b_tp = (int)(pb & 0xffffu);
              b_ap = (int)(pb >> 16);
            }
            const float w = lut_prob<DT>(J.lut, a_e, aa, ab, a_tp, a_ap, B.dbg) *
                            lut_prob<DT>(J.lut, dir.w, ba, bb, b_tp, b_ap, B.dbg);
            q = __float2ll_rn(w * 4294967296.0f);
          }
          if (kDebug && lm.out) {
            const unsigned long long slot = atomicAdd(lm.count, 1ull);
            if (slot < lm.cap) {
              psc_listmode_event* r = lm.out + slot;
              const uint4 clm = cold[C_LM * n_slots + g];
              r->history = history();
              r->q = key_ < 0 ? 0 : q;
              r->voxel = (int)cold[C_E0 * n_slots + g].w;
              r->cls = cls;
              r->delta_mm = 0.5f * (a_path - path);
              r->energy_kev[0] = a_e;
              r->energy_kev[1] = dir.w;
              float pa = atan2f(a_ny, a_nx), pb = atan2f(b_ny, b_nx);
              r->phi[0] = pa < 0.0f ? pa + 6.283185307179586f : pa;
              r->phi[1] = pb < 0.0f ? pb + 6.283185307179586f : pb;
              r->z_mm[0] = __uint_as_float(clm.x);
              r->z_mm[1] = __uint_as_float(clm.y);
              r->dir[0][0] = a_d.x;
              r->dir[0][1] = a_d.y;
              r->dir[0][2] = a_d.z;
              r->dir[1][0] = dir.x;
              r->dir[1][1] = dir.y;
              r->dir[1][2] = dir.z;
              r->crystal[0] = a_cr;
              r->crystal[1] = b_cr;
              r->ring[0] = a_rg;
              r->ring[1] = b_rg;
              const uint32_t sa = clm.z, sb = kc.y >> 15;
              r->n_scatter[0] = (uint16_t)min(sa >> 1, 65535u);
              r->n_scatter[1] = (uint16_t)min(sb >> 1, 65535u);
              r->rayleigh[0] = (uint8_t)(sa & 1u);
              r->rayleigh[1] = (uint8_t)(sb & 1u);
              for (int b = 0; b < 6; ++b) r->pad[b] = 0;
            }
          }
          // lanes that hit the same bin add their weights first, one atomic per bin
          const unsigned act = __activemask();
          const unsigned takers = __ballot_sync(act, take);
          if (take) {
            const unsigned peers = __match_any_sync(takers, (unsigned long long)key_);
            const unsigned hi = __reduce_add_sync(peers, (unsigned)(q >> 16));
            const unsigned lo = __reduce_add_sync(peers, (unsigned)(q & 0xffff));
            if (lane_id == (unsigned)(__ffs(peers) - 1)) {
              atomicAdd(J.acc + dbg_idx(B.dbg, kSiteAcc, key_,
                                        (long long)S.n_rings * S.n_rings * S.n_views * S.n_rad * S.n_tof),
                        ((unsigned long long)hi << 16) + lo);
              if (stats) atomicAdd(&s_cnt[kStatAtomics], 1ull);
            }
            if (stats) {
              atomicAdd(&s_cnt[kStatBinned], 1ull);
              atomicAdd(&s_cnt[kStatWeight], (unsigned long long)q);
            }
          }
          finish(cls, key_, cls == kOutOfRange ? 0 : q);
        }
      }
      __syncwarp();  // slot updates are visible to the lanes that vote on them next
    }

    __syncthreads();  // every slot is done with the chunk before the next fetch
  }

  if (!stats) return;
  __syncthreads();
  for (int i = threadIdx.x; i < kStatCount; i += blockDim.x)
    if (s_cnt[i]) atomicAdd(B.stats + i, s_cnt[i]);
}

size_t transport_cold_words(int grid, int block) {
  return (size_t)grid * kColdVecs * 4 * (size_t)(block / 32) * kSlotsPerWarp;
}

size_t transport_smem_bytes(const PhantomParams& ph, int block) {
  return kSlotBytes * (size_t)(block / 32) * kSlotsPerWarp +
         sizeof(float4) * (size_t)ph.n_mat * ph.n_tab + sizeof(float) * (ph.n_tab + kMaxMaterials);
}

// Lets a kernel use all the dynamic shared memory that the device has for it.  The limit
// belongs to the kernel on its device: set to each launch's own size, one thread could
// lower it between another's call and launch.
template <class K>
static cudaError_t allow_smem(K kernel) {
  int dev = 0, most = 0;
  cudaFuncAttributes a;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, kernel);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most - (int)a.sharedSizeBytes);
}

template <int DT, bool kDebug, bool kOneJob = false, bool kFixed = false>
static cudaError_t launch_dt(const BatchParams& p, int grid, int block, size_t smem, cudaStream_t s) {
  const cudaError_t e = allow_smem(transport_kernel<DT, kDebug, kOneJob, kFixed>);
  if (e != cudaSuccess) return e;
  transport_kernel<DT, kDebug, kOneJob, kFixed><<<grid, block, smem, s>>>(p);
  return cudaGetLastError();
}

template <int DT>
static cudaError_t launch_dt(const BatchParams& p, int grid, int block, size_t smem, cudaStream_t s) {
  bool debug = p.stats != nullptr;
  for (int j = 0; j < p.n_jobs; ++j)
    debug |= p.jobs[j].cls_out || p.jobs[j].key_out || p.jobs[j].q_out || p.lm[j].out;
  if (debug) return launch_dt<DT, true>(p, grid, block, smem, s);
  if (block != 512) return launch_dt<DT, false>(p, grid, block, smem, s);
  if constexpr (DT == 0) {
    if (p.n_jobs == 1) return launch_dt<0, false, true, true>(p, grid, block, smem, s);
  }
  return launch_dt<DT, false, false, true>(p, grid, block, smem, s);
}

cudaError_t launch_transport(const BatchParams& p, int lut_dtype, int grid, int block, size_t smem,
                             cudaStream_t s) {
  switch (lut_dtype) {
    case 0: return launch_dt<0>(p, grid, block, smem, s);
    case 1: return launch_dt<1>(p, grid, block, smem, s);
    case 2: return launch_dt<2>(p, grid, block, smem, s);
    default: return launch_dt<-1>(p, grid, block, smem, s);
  }
}

// both instantiations of a LUT type share launch bounds and shared memory.
// The query counts dynamic shared memory above 48 KB only once the kernel
// may use it, so the attribute is set first (else the first launch of a
// kernel would size its grid for one CTA per SM).
template <int DT>
static cudaError_t occupancy_dt(int block, size_t smem, int* blocks_per_sm) {
  const cudaError_t e = allow_smem(transport_kernel<DT, false>);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, transport_kernel<DT, false>, block, smem);
}

cudaError_t transport_occupancy(int lut_dtype, int block, size_t smem, int* blocks_per_sm) {
  switch (lut_dtype) {
    case 0: return occupancy_dt<0>(block, smem, blocks_per_sm);
    case 1: return occupancy_dt<1>(block, smem, blocks_per_sm);
    case 2: return occupancy_dt<2>(block, smem, blocks_per_sm);
    default: return occupancy_dt<-1>(block, smem, blocks_per_sm);
  }
}

}  // namespace psc

// engine.h -- launch interface of the persistent phase engine (engine.cu).
#pragma once

#include "common.cuh"

namespace sssp {

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kSmallThreads = 256;  // blocks of a batch of many solves (at least kNfBins threads)
// Grid phases are warp-centric: a warp takes a chunk of 32 * kSelItems fringe
// entries in the selection step and a tile of kTile consecutive edges of the
// relax list in the relax step, with all of a lane's loads in flight together
// and no block barrier inside the loop.
constexpr int kRelaxItems = 4;  // edges per lane per relax tile
constexpr int kSelItems = 4;    // fringe entries per lane per selection chunk
constexpr int kTile = 32 * kRelaxItems;
// A single solve uses one block per this many vertices (at most all co-resident blocks).
constexpr uint32_t kVertsPerBlock = 1024;
// Solo mode (one block runs whole phases with the fringe in shared memory):
// a limit of kSoloCap vertices or more stands for as many as the block has
// slots for.
constexpr uint32_t kSoloCap = 2048;
constexpr uint32_t kSoloMaxDefault = kSoloCap;     // fringe size limit
constexpr uint32_t kSoloEdgesDefault = 2048;       // relax edges above which a solo phase hands off
constexpr uint32_t kNearFarMinDefault = 8192;      // fringe size per block of the solve at which the near/far split starts
constexpr uint32_t kNearFarShareDefault = 8;       // ... and fringe share of n, in 256ths
constexpr size_t kGridSmem = 66 * sizeof(unsigned long long)                                         // reduction scratch, bases
                             + kWarps * kTile * (2 * sizeof(uint32_t) + sizeof(unsigned long long))  // relax tiles
                             + 36 * sizeof(uint32_t)                                                   // range, scan
                             + kWarps * kNfRing * sizeof(uint32_t);                                    // bucket counts
// Slots per thread of a solo block (see solo_large on the choice).
constexpr uint32_t kSoloSmallSpt = 4, kSoloLargeSpt = 8, kSoloLargeWideSpt = 8;
constexpr uint32_t kSoloLargeN = 1u << 17;
constexpr uint32_t kSoloNarrowW = 1u << 29;  // largest cost with 32-bit distances in the slots
constexpr size_t kSoloSlotBytes = sizeof(uint4) + sizeof(uint2), kSoloWideSlotBytes = kSoloSlotBytes + 8;
constexpr size_t kPolicySmem = 1476 * sizeof(float);  // the policy network's weights, after the phase region
constexpr uint32_t kSoloList = 24;  // settled vertices that a warp lists in a phase
constexpr size_t kMaxSmem = kThreads * (kSoloLargeWideSpt * kSoloWideSlotBytes + sizeof(uint32_t)) +
                            kWarps * kSoloList * sizeof(uint4) + kPolicySmem;
// The same for blocks of kSmallThreads, several of which share an SM.
constexpr uint32_t kSmallSpt = 8, kSmallLargeSpt = 16, kSmallLargeWideSpt = 12;
constexpr size_t kMaxSmallSmem = kSmallThreads * (kSmallLargeSpt * kSoloSlotBytes + sizeof(uint32_t)) +
                                 kSmallThreads / 32 * kSoloList * sizeof(uint4) + kPolicySmem;
static_assert(kSmallLargeSpt * kSoloSlotBytes >= kSmallLargeWideSpt * kSoloWideSlotBytes &&
              kSmallLargeSpt * kSoloSlotBytes >= kSmallSpt * kSoloWideSlotBytes, "largest layout");
static_assert(kSmallSpt % 4 == 0 && kSmallLargeSpt % 4 == 0 && kSmallLargeWideSpt % 4 == 0 && kSmallLargeSpt <= 16 &&
              kSmallSpt * kSmallThreads >= kSoloCap && kSmallThreads >= kNfBins, "as for the large blocks");
static_assert(kSoloLargeWideSpt * kSoloWideSlotBytes >= kSoloLargeSpt * kSoloSlotBytes, "largest layout");
static_assert(kSoloSmallSpt % 4 == 0 && kSoloLargeSpt % 4 == 0 && kSoloLargeWideSpt % 4 == 0 && kSoloLargeSpt <= 16,
              "slots are tested four at a time, masks have 16 bits");
static_assert(kSoloSmallSpt * kThreads >= kSoloCap, "a policy's episodes need a slot for each of kSoloCap vertices");

// Graphs whose edges and vertex records take at most this many bytes are
// prefetched into L2 when a solve starts (L2 holds 126 MiB).
constexpr uint64_t kL2PrefetchBytes = 96ull << 20;
struct SolveParams {
  GraphView g;
  SolveWS ws;
  uint32_t source;
  uint32_t crit;
  unsigned long long wait_ns;
  uint32_t solo_max;    // largest fringe run by one block alone (0 = never)
  uint32_t solo_edges;  // relax edges above which a solo phase hands off to the group
  uint32_t nf_min;      // fringe size per block of the solve at which the near/far split starts (0 = never)
  uint32_t nf_target;   // near-part size aimed at when the bound is set (0 = automatic)
  uint32_t nf_share;    // the split also needs |F| >= nf_share * n / 256
  uint32_t solo_spt;    // slots per thread of a solo block
  uint32_t pol_off;     // offset of the policy weights in dynamic shared memory
  const float* policy;  // policy network weights (device) or nullptr
};

// Sets the shared-memory layout of a solve of p->g in *p; returns its dynamic
// shared memory (at most kMaxSmem).
size_t solo_shape(uint32_t crit, SolveParams* p);

// The kernel of one whole solve per cooperative launch (all blocks co-resident;
// one SolveParams by value), kThreads threads per block, solo_shape's dynamic
// shared memory: the instance that fits the solve.
int solve_kind(const SolveParams& p);
const void* grid_kernel(int kind);

}  // namespace sssp

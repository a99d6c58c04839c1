// The resident step kernel (lbm_resident.cu): its plans for a grid or a batch, and its launches.
#pragma once

#include <cuda_runtime.h>

#include <vector>

#include "lbm_device.cuh"
#include "lbm_resident_rules.h"

namespace cmlbm {

// A grid's blocks: nstrip strips of 64 columns times nseg row segments, numbered from block0.
struct ResidentGrid {
    int nstrip, nseg, block0;
};

// What a launch of blocks of at most hmax rows takes.
struct ResidentSizes {
    int nblocks, hmax;
    int tab;              // capacity of a block's send and receive lists
    int box_entries;      // 16-byte words of a block's mailbox (one of two)
    size_t smem;          // dynamic shared memory of a block
    size_t box_bytes;     // the mailboxes of all blocks, both parities
    size_t list_bytes;    // the exchange lists of all blocks
};

struct ResidentPlan {
    ResidentGrid D;
    ResidentSizes Z;
};

// One case of a batch as the kernel sees it (off: element offsets of its two buffers).
struct ResidentCase {
    Geometry G;
    ResidentGrid D;
    long long off[2];
    Consts<float> K;
};

// Cases of a batch whose blocks fit on the device at once: indices and splits, in block order.
struct ResidentWave {
    std::vector<int> cases;
    std::vector<ResidentGrid> D;
    ResidentSizes Z;
};

struct ResidentLaunch {
    int hmax, tab, box_entries;
    int nsteps;
    int flow_sign;        // imposed flow: +1, or -1 once reversed
    unsigned tag0;        // messages of step s carry tag0 + 1 + s
    ulonglong2* box;      // [2][blocks][box_entries], zeroed once
    int* lists;           // exchange lists, one after another
    int* err;             // device error word (0 = ok)
};

// Plan for a grid on a device of nsm SMs (the current device), with as many blocks as make a step
// fastest by itself, or with shared, beside others on other streams (shared_segments); false where its
// state does not fit in their shared memory, a block would have a single row, the grid a single
// column, or shared_segments finds none.
template <typename S, int V>
bool resident_plan(const Geometry&, int nsm, bool shared, ResidentPlan*);

// Zero the caller's mailboxes (box_bytes) and fill its exchange lists (list_bytes), once per plan.
template <typename S, int V>
cudaError_t prepare_resident(const Geometry&, const ResidentPlan&, void* box, void* lists,
                             cudaStream_t);

// Advance `state` in place by nsteps >= 1 steps in one cooperative launch, through prepared
// mailboxes and lists; the tags of consecutive launches continue.
template <typename S, int V>
cudaError_t launch_resident(void* state, const Geometry&, const Consts<float>&,
                            const ResidentPlan&, int nsteps, int flow_sign, unsigned tag0,
                            void* box, void* lists, int* err, cudaStream_t);

// Empty the send lists, so that the waits of the next launch run out (a test of the way out), after
// which the mailboxes and lists have to be prepared again.
cudaError_t mute_resident(const ResidentPlan&, void* lists, cudaStream_t);

// The same for a batch, one launch per wave, the wave of the most blocks first; false where a case
// does not fit.  *step_us: what a step of all waves takes by the planner's model.  The waves of a batch
// may share one set of mailboxes (zeroed by the caller), with tags that continue from launch to
// launch; case_of[b] is the index into `cases` of block b of the wave.
template <typename S, int V>
bool resident_batch_plan(const Geometry*, int ncases, int nsm, std::vector<ResidentWave>*,
                         double* step_us);
template <typename S, int V>
cudaError_t prepare_resident_batch(const ResidentSizes&, const ResidentCase* cases,
                                   const int* case_of, void* lists, cudaStream_t);
template <typename S, int V>
cudaError_t launch_resident_batch(void* base, const ResidentSizes&, const ResidentCase* cases,
                                  const int* case_of, int parity, int nsteps, unsigned tag0,
                                  void* box, void* lists, int* err, cudaStream_t);

}  // namespace cmlbm

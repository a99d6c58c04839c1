// The resident step kernel (lbm_resident.cu): its plan for a grid and its launch.
#pragma once

#include <cuda_runtime.h>

#include "lbm_device.cuh"

namespace cmlbm {

constexpr int kResidentWarps = 16;   // warps of a block; one block per SM

// Split of a grid into blocks of one strip of 64 columns and at most hmax rows.
struct ResidentPlan {
    int nstrip, nseg;     // blocks = nstrip * nseg
    int hmax;             // rows of the tallest block
    int tab;              // capacity of a block's send and receive lists
    int box_entries;      // 16-byte words of a block's mailbox (one of two)
    size_t smem;          // dynamic shared memory of a block
    size_t box_bytes;     // the mailboxes of all blocks, both parities
    size_t list_bytes;    // the exchange lists of all blocks
};

struct ResidentLaunch {
    int nstrip, nseg, hmax, tab, box_entries;
    int nsteps;
    int flow_sign;        // imposed flow: +1, or -1 once reversed
    unsigned tag0;        // messages of step s carry tag0 + 1 + s
    ulonglong2* box;      // [2][blocks][box_entries], zeroed once
    int* lists;           // exchange lists, one after another
    int* err;             // device error word (0 = ok)
};

// Plan for a grid on a device of nsm SMs (the current device); false where its state does not
// fit in their shared memory or a block would be one node wide.
template <typename S, int V>
bool resident_plan(const Geometry&, int nsm, ResidentPlan*);

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

}  // namespace cmlbm

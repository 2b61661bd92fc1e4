// Host-side interface of the resident kernel (resident.cu): many time steps per launch with the
// lattice's state kept on chip.
#pragma once

#include "common.cuh"

namespace lbmem {

// Steps one launch takes at most (its source values sit in shared memory), and steps whose
// staged stencil fields a launch that accumulates holds.
constexpr int kResidentSteps = 256, kResidentAccSteps = 128;
constexpr int kResidentMaxWarps = 16, kResidentMaxRows = 16;
constexpr size_t kControlBytes = 128;  // ahead of the mailboxes
constexpr int kResidentHalo = 4;  // FP32: steps between two exchanges of the tiles' halos

// How a lattice is spread over the GPU: strips of 32 lanes (64 columns in FP32, 32 in the 8-byte
// forms) cut into segments of `rows` rows, one warp each; `warps` such warps and
// `comm` communication warps per thread block, at most one block per SM.  ctas == 0: the lattice does not fit (or is better off elsewhere).
// wait: clock cycles after which a wait for another block or warp gives up; launch: the blocks that are
// launched, all of them except in a test of those waits.
struct ResidentPlan {
    int ctas, strips, rows, segs, warps, comm, total, launch;
    long long wait;
    size_t smem, mail_x, mail_bytes;
};

// The plan of an nx x ny lattice for T = float, double or df and polarization pol; configures its
// kernels.  Once per handle, outside stream capture.
template <typename T>
cudaError_t resident_plan(int nx, int ny, int pol, ResidentPlan *plan);

// n (1 .. kResidentSteps, with accumulate kResidentAccSteps) steps from fin (time word t_in) to
// fout (t_out = t + n) in one cooperative launch.  mail: plan.mail_bytes (control words,
// then mailboxes), cleared once before the first launch and then left to the kernel.  accumulate: the fields at
// the n_slots stencil sites of a.accp through stage (3 n_slots values of T per step) and a second
// launch that adds them to a.accp.acc.  One launch at a time per mail buffer (stream order).
template <typename T>
cudaError_t launch_resident(const StepArgs<T> &a, const T *fin, T *fout, const long long *t_in, long long *t_out,
                            const ResidentPlan &plan, void *mail, int n, bool accumulate, T *stage, int n_slots,
                            cudaStream_t s);

}  // namespace lbmem

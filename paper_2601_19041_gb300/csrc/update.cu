// End of an iteration as separate launches (the per-iteration path):
// k_select (iteration best), k_gb (global best, bounds, succ/pred), or both as
// k_select_gb, and
// k_update (bounded evaporation/deposit fused with the next choice_info).
// The arithmetic is in iter.cuh.
#include "iter.cuh"

namespace hac {

__global__ void k_select(const DevInst *insts)
{
    const DevInst &I = insts[blockIdx.x];
    InstState *st = I.st;
    if (st->t >= I.iters) {
        if (threadIdx.x == 0) st->active = 0;
        return;
    }
    block_iteration_best(I, st);
}

// both at once: no local search runs between them
__global__ void k_select_gb(const DevInst *insts)
{
    const DevInst &I = insts[blockIdx.x];
    InstState *st = I.st;
    if (st->t >= I.iters) {
        if (threadIdx.x == 0) st->active = 0;
        return;
    }
    block_iteration_best(I, st);
    block_global_best(I, st);
}

__global__ void k_gb(const DevInst *insts)
{
    const DevInst &I = insts[blockIdx.x];
    InstState *st = I.st;
    if (!st->active) return;
    block_global_best(I, st);
}

// four slots a thread: 1024 slots of an instance per block of 256 threads
__global__ void k_update(const DevInst *insts, const int2 *slotmap)
{
    const int2 sm = slotmap[blockIdx.x];
    const DevInst &I = insts[sm.x];
    const InstState *st = I.st;
    if (!st->active) return;
    const size_t s = (size_t)sm.y + 4 * threadIdx.x;
    if (s >= (size_t)I.n * I.k_pad) return;
    const int4 j4 = *reinterpret_cast<const int4 *>(I.cand + s);
    const int j[4] = {j4.x, j4.y, j4.z, j4.w};
    const float omega = __double2float_rn(__dsub_rn(1.0, I.rho));
    const float delta = __double2float_rn(__ddiv_rn(1.0, st->L_dep));
    float4 *ch = reinterpret_cast<float4 *>(I.choice + s);
    *ch = update_slots4(I, s, (int)(s / I.k_pad), j, *ch, omega, delta, st->tau_min, st->tau_max);
}

// MMAS schedule end (restart check, next u_gb); one block per instance
__global__ void k_schedule(const DevInst *insts)
{
    const DevInst &I = insts[blockIdx.x];
    InstState *st = I.st;
    if (!st->active || !I.schedule) return;
    block_schedule_end(I, st);
}

void launch_two_opt_ib(const DevInst *d_inst, int count, int max_n, cudaStream_t s);
void launch_two_opt_all(const DevInst *d_inst, int count, int max_m, int max_n, cudaStream_t s);

// Launches only what some instance needs: an iteration of a small instance is
// a chain of launches of a few us each (one n = 100 instance, 50 iterations end
// to end: 4.23 ms with all of them, 3.82 ms).
int launch_iteration_tail(const DevInst *d_inst, int count, const int2 *d_slotmap, int slotmap_len,
                          const TailNeeds &needs, int max_n, cudaStream_t s)
{
    int launched = 2;
    if (needs.ls_all_m > 0) { launch_two_opt_all(d_inst, count, needs.ls_all_m, max_n, s); ++launched; }
    if (needs.ls_ib) {
        k_select<<<count, 256, 0, s>>>(d_inst);
        launch_two_opt_ib(d_inst, count, max_n, s);
        k_gb<<<count, 256, 0, s>>>(d_inst);
        launched += 2;
    } else {
        k_select_gb<<<count, 256, 0, s>>>(d_inst);
    }
    k_update<<<slotmap_len, 256, 0, s>>>(d_inst, d_slotmap);
    if (needs.schedule) { k_schedule<<<count, 256, 0, s>>>(d_inst); ++launched; }
    return launched;
}

}  // namespace hac

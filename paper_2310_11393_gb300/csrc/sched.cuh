// Bookkeeping between the phases of a step, shared by the kernels that do it on their own
// (push.cu) and the field solver, whose launch takes it along (yee.cu): the tile scan of one
// block and the end of a step.
#pragma once

#include "sff_common.cuh"
#include "sff_kernels.h"

namespace sff {

// Block-wide exclusive scan of one int per thread (blockDim a multiple of 32, <= 1024).
__device__ __forceinline__ int block_exclusive_scan(int v, int* s_warp)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int x = v;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, off);
        if (lane >= off) x += y;
    }
    if (lane == 31) s_warp[wid] = x;
    __syncthreads();
    if (wid == 0) {
        int w = lane < nw ? s_warp[lane] : 0;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, w, off);
            if (lane >= off) w += y;
        }
        s_warp[lane] = w;
    }
    __syncthreads();
    const int r = x - v + (wid > 0 ? s_warp[wid - 1] : 0);
    __syncthreads();
    return r;
}

// Chunks of tile t of buffer set q holding c particles from slot base: ctile / crange
// entries from chunk index rc on.
__device__ __forceinline__ void write_chunks(const SimDev& S, int q, int t, int base, int c, int rc)
{
    const int nc = (c + S.chunk - 1) / S.chunk;
    for (int k = 0; k < nc; ++k) {
        S.ctile[q][rc + k] = t;
        const int a = base + k * S.chunk;
        S.crange[q][rc + k] = make_int2(a, min(a + S.chunk, base + c));
    }
}

// Tile scan of one simulation after a push into buffer set q (one block of 1024 threads):
// per tile the particles now in set q (tcnt) and its frame count (fcnt) give
//   set q:      tnum, the chunk offsets coff and the chunk map (ctile, crange) over the
//               slots toff[q] set by the previous scan;
//   set 1 - q:  toff = exclusive scan of tcnt + fcnt, the slots of the next step's push;
// the particle total goes to n_next; the counts, cursors and frame counts are cleared.
// `compact` (set-up): toff[q] = exclusive scan of tcnt first (no slack: the particles are
// then placed there by the caller) and set 1 - q is left alone.
__device__ __forceinline__ void scan_counts(const SimDev& S, int q, bool compact)
{
    __shared__ int s_warp[32];
    const int n = S.nptiles;
    const int tid = threadIdx.x, nth = blockDim.x;
    const int per = (n + nth - 1) / nth;
    const int i0 = min(n, tid * per), i1 = min(n, i0 + per);
    int lp = 0, lc = 0, lk = 0;
    for (int i = i0; i < i1; ++i) {
        const int c = S.tcnt[i];
        lp += c;
        lc += (c + S.chunk - 1) / S.chunk;
        lk += c + S.fcnt[i];
    }
    int rp = block_exclusive_scan(lp, s_warp);
    int rc = block_exclusive_scan(lc, s_warp);
    int rk = block_exclusive_scan(lk, s_warp);
    if (tid == nth - 1) atomicAdd(&S.st->n_next, rp + lp);
    for (int i = i0; i < i1; ++i) {
        const int c = S.tcnt[i];
        if (compact) S.toff[q][i] = rp;
        const int base = compact ? rp : S.toff[q][i];
        S.tnum[q][i] = c;
        S.coff[q][i] = rc;
        write_chunks(S, q, i, base, c, rc);
        if (!compact) S.toff[1 - q][i] = rk;
        rp += c;
        rc += (c + S.chunk - 1) / S.chunk;
        rk += c + S.fcnt[i];
        S.tcnt[i] = 0;
        S.tcur[i] = 0;
        S.fcnt[i] = 0;
    }
    if (tid == nth - 1) {
        if (compact) S.toff[q][n] = rp;
        else S.toff[1 - q][n] = rk;
        S.coff[q][n] = rc;
    }
    __syncthreads();
}

// End of a step (one block): step counter, particle count and buffer parity of every simulation
// of the group, then the next step's chunk numbering and work counters (what k_prefix does), so
// that a step of the same group needs no k_prefix of its own.
__device__ __forceinline__ void end_step(const SimDev* __restrict__ sims, int nsims, int* __restrict__ gprefix,
                                         int* __restrict__ counters)
{
    __shared__ int s_warp[32];
    const int tid = threadIdx.x, nth = blockDim.x;
    const int per = (nsims + nth - 1) / nth;
    const int i0 = min(nsims, tid * per), i1 = min(nsims, i0 + per);
    int l = 0;
    for (int i = i0; i < i1; ++i) {
        const SimDev& S = sims[i];
        DevState* st = S.st;
        const int np = 1 - st->parity;
        st->n_alive = st->n_next;
        st->n_next = 0;
        st->parity = np;
        st->step += 1;
        l += S.coff[np][S.nptiles];
    }
    int r = block_exclusive_scan(l, s_warp);
    for (int i = i0; i < i1; ++i) {
        gprefix[i] = r;
        r += sims[i].coff[sims[i].st->parity][sims[i].nptiles];   // the parity this thread just set
    }
    if (tid == nth - 1) gprefix[nsims] = r;
    if (tid < NCOUNTERS) counters[tid] = 0;
    if (nsims == 1) {
        const SimDev& S = sims[0];
        for (int j = tid; j < S.nscanblk; j += nth) S.scanflags[j] = 0ull;
        if (tid == 0) *S.scanticket = 0;
    }
}

// The rest of a step that rides on the field solver's launch: its first nscan blocks scan the
// tiles of one simulation each, and the last block to finish ends the step.  nscan 0: neither
// (they are launches of their own).
struct StepTail {
    const SimDev* sims;
    int nsims, nscan;
    int* gprefix;
    int* counters;
};

// (calls, so that the registers of the solver's loops do not pay for these)
static __device__ __noinline__ void scan_call(const SimDev& S) { scan_counts(S, 1 - S.st->parity, false); }
static __device__ __noinline__ void end_call(const StepTail& t) { end_step(t.sims, t.nsims, t.gprefix, t.counters); }

// true for a block that scans instead of solving
__device__ __forceinline__ bool tail_scan(const StepTail& t)
{
    if ((int)blockIdx.x >= t.nscan) return false;
    scan_call(t.sims[blockIdx.x]);
    return true;
}

// every block, when its work is done
__device__ __forceinline__ void tail_end(const StepTail& t)
{
    if (t.nscan == 0) return;
    __shared__ int s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(&t.counters[NCOUNTERS - 1], 1) == (int)gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    end_call(t);
}

}  // namespace sff

// whg_kernels_common.cu -- init and raw-state kernels, and the launchers that
// pick the Newton-phase series length.
#include "whg_device.cuh"

namespace whg {

__global__ void __launch_bounds__(WHG_MAX_BLOCK) k_init(WhgState st, WhgBuckets bk, WhgIn in)
{
    const int w = warp_index();
    if (w >= bk.warp0[bk.nb]) return;
    const int b = bucket_of(bk, w);
    WHG_DISPATCH_L(bk.L[b], (init_body<L_>(st, bk, in, b, w)))
}

__global__ void __launch_bounds__(WHG_MAX_BLOCK) k_raw(WhgState st, WhgBuckets bk, WhgOut io, int set)
{
    const int w = warp_index();
    if (w >= bk.warp0[bk.nb]) return;
    const int b = bucket_of(bk, w);
    WHG_DISPATCH_L(bk.L[b], (raw_body<L_>(st, bk, io, set, b, w)))
}

// Ensemble repacking (no counterpart in the paper).  Within every bucket the
// systems still running come first and the stopped ones last, each group in
// its previous order, so that warps whose systems have all stopped skip their
// steps.  Each system's arithmetic involves only its own lanes, so moving it
// to other lanes leaves its results bitwise unchanged.
//
// order[new internal index] = old internal index; one block per bucket: a
// count of running systems, then a stable partition chunk by chunk
// (ballot/popc scan within warps, warp totals in shared memory).
__global__ void __launch_bounds__(1024) k_repack_order(WhgState st, WhgBuckets bk, int* order)
{
    const int b = blockIdx.x;
    if (b >= bk.nb) return;                                  // whole block
    const int s0 = bk.sys0[b], s1 = bk.sys0[b + 1];
    const int lane = (int)(threadIdx.x & 31u), wid = (int)(threadIdx.x >> 5), nw = (int)(blockDim.x >> 5);
    __shared__ int part[32];
    __shared__ int total;
    int cnt = 0;
    for (int s = s0 + (int)threadIdx.x; s < s1; s += (int)blockDim.x) cnt += st.status[s] == 0;
#pragma unroll
    for (int o = 16; o; o >>= 1) cnt += __shfl_xor_sync(WHG_FULL_MASK, cnt, o);
    if (lane == 0) part[wid] = cnt;
    __syncthreads();
    if (threadIdx.x == 0) {
        int t = 0;
        for (int i = 0; i < nw; ++i) t += part[i];
        total = t;
    }
    __syncthreads();
    const int nlive = total;
    int base_live = 0, base_stopped = 0;
    for (int c0 = s0; c0 < s1; c0 += (int)blockDim.x) {     // same trip count in every thread
        const int s = c0 + (int)threadIdx.x;
        const bool valid = s < s1;
        const bool live = valid && st.status[s] == 0;
        const unsigned bal = __ballot_sync(WHG_FULL_MASK, live);
        const int in_warp = __popc(bal & ((1u << lane) - 1u));
        __syncthreads();                                     // previous readers of part[] are done
        if (lane == 0) part[wid] = __popc(bal);
        __syncthreads();
        int before = 0, chunk_live = 0;
        for (int i = 0; i < nw; ++i) {
            const int v = part[i];
            before += i < wid ? v : 0;
            chunk_live += v;
        }
        const int excl = before + in_warp;                   // running systems before s in the chunk
        if (valid) {
            const int pos = live ? base_live + excl : nlive + base_stopped + ((int)threadIdx.x - excl);
            order[s0 + pos] = s;
        }
        const int nvalid = s1 - c0 < (int)blockDim.x ? s1 - c0 : (int)blockDim.x;
        base_live += chunk_live;
        base_stopped += nvalid - chunk_live;
    }
}

// Gather the state into dst in the new order: lane arrays for every lane in
// use (lanes that hold no system keep their index), per-system arrays once
// per system.  dst has the layout of src.
__global__ void __launch_bounds__(256) k_repack_gather(WhgState src, WhgState dst, WhgBuckets bk,
                                                       const int* order)
{
    const long long li = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int w = (int)(li >> 5);
    if (w >= bk.warp0[bk.nb]) return;
    const int lane = (int)(li & 31);
    const int b = bucket_of(bk, w);
    const int L = bk.L[b], spw = 32 / L;
    const int slot = lane / L, p = lane - slot * L;
    const int local = (w - bk.warp0[b]) * spw + slot;
    size_t from = (size_t)li;
    int s_new = -1, s_old = -1;
    if (slot < spw && local < bk.sys0[b + 1] - bk.sys0[b]) {
        s_new = bk.sys0[b] + local;
        s_old = order[s_new];
        WHG_CHECK(src, s_old >= bk.sys0[b] && s_old < bk.sys0[b + 1], WHG_BOUND_REPACK);
        const int lo = s_old - bk.sys0[b];
        from = (size_t)(bk.warp0[b] + lo / spw) * 32 + (size_t)(lo % spw) * L + p;
    }
    WHG_CHECK(src, (long long)from < src.nl && li < src.nl, WHG_BOUND_LANE);
    dst.m[li] = src.m[from];
    dst.qx[li] = src.qx[from];
    dst.qy[li] = src.qy[from];
    dst.qz[li] = src.qz[from];
    dst.vx[li] = src.vx[from];
    dst.vy[li] = src.vy[from];
    dst.vz[li] = src.vz[from];
    dst.a0[li] = src.a0[from];
    if (s_new >= 0 && p == 0) {
        const size_t S = (size_t)src.S;
        dst.m0[s_new] = src.m0[s_old];
        dst.dt[s_new] = src.dt[s_old];
        dst.M[s_new] = src.M[s_old];
        dst.rej2[s_new] = src.rej2[s_old];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            dst.xcm[k * S + s_new] = src.xcm[k * S + s_old];
            dst.vcm[k * S + s_new] = src.vcm[k * S + s_old];
        }
        dst.nstep[s_new] = src.nstep[s_old];
        dst.nplan[s_new] = src.nplan[s_old];
        dst.status[s_new] = src.status[s_old];
        dst.perm[s_new] = src.perm ? src.perm[s_old] : s_old;
    }
}

}  // namespace whg

cudaError_t whg_launch_repack(const WhgState& st, const WhgState& scratch, const WhgBuckets& bk, int* order,
                              cudaStream_t stream)
{
    whg::k_repack_order<<<bk.nb, 1024, 0, stream>>>(st, bk, order);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const long long lanes = (long long)bk.warp0[bk.nb] * 32;
    const int grid = (int)((lanes + 255) / 256);
    if (grid > 0) whg::k_repack_gather<<<grid, 256, 0, stream>>>(st, scratch, bk, order);
    return cudaGetLastError();
}

cudaError_t whg_launch_init(const WhgState& st, const WhgBuckets& bk, const WhgIn& in, const WhgLaunch& l)
{
    whg::k_init<<<l.grid, l.block, 0, l.stream>>>(st, bk, in);
    return cudaGetLastError();
}

cudaError_t whg_launch_raw(const WhgState& st, const WhgBuckets& bk, const WhgOut& o, int set,
                           const WhgLaunch& l)
{
    whg::k_raw<<<l.grid, l.block, 0, l.stream>>>(st, bk, o, set);
    return cudaGetLastError();
}

static int sm_count()
{
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return sms;
}

// Three step kernels, the same bits from each (whg_wide.cuh, step_body):
// * four lanes per planet while its warps, four times as many, stay within 8
//   per SM (2 per sub-partition), or 12 for systems of 6 or more planets, whose
//   pair rounds it saves most.  us per step, four lanes / one: 8 planets 608
//   systems (4 warps per SM) 2.21 / 4.08, 1216 (8) 2.88 / 4.14, 1824 (12)
//   3.64 / 4.11, 2432 (16) 5.55 / 4.11; 5 planets 777 (5) 2.97 / 3.45,
//   1500 (10) 3.65 / 3.45; 2 planets 4864 (8) 2.58 / 2.96, 9728 (16) 5.25 / 2.99;
// * one lane per planet, registers for one warp's own chain of instructions
//   (182; k_step<.., 1>), up to 8 warps per SM;
// * one lane per planet, 128 registers, above: the resident warps count.  182 /
//   128 registers: 2432 systems (4 warps per SM) 4.11 / 4.47, 4096 (6.7) 4.70 /
//   4.89, 4864 (8) 5.23 / 5.50, 8192 (13.5) 10.2 / 7.37.
static bool wide_warps(const WhgState& st, const WhgBuckets& bk, int sms)
{
    if (st.full_rotation) return false;              // interaction schedule without reactions: FP64 only
    int least = 8;
    for (int b = 0; b < bk.nb; ++b) least = bk.L[b] < least ? bk.L[b] : least;
    return whg_wide_warps(bk) <= (least >= 6 ? 12 : 8) * sms;
}

// Blocks for an ensemble of several lane-group sizes: as many consecutive warps,
// which are of one size but for the bucket borders, as make one block per SM, at
// most 8.  Every size has its own unrolled step of ~35 KB of code, and with one-warp
// blocks, dealt out over the SMs, each SM ran most of them side by side, more than
// its instruction cache holds.  us per step, compact systems of 2 to 8 planets,
// one-warp blocks / these: 300 2.9 / 2.6, 1500 10.4 / 3.3, 4096 11.9 / 4.8, 7000
// 14.3 / 5.9, 12,000 16.9 / 9.0, 65,536 37.1 / 36.9; 4096 of them at steps of P/7, with
// a few systems redone in FP64 each step, 18.0 / 5.0 (15.8 when all was FP64).
static WhgLaunch mixed_blocks(const WhgLaunch& l, const WhgBuckets& bk, int warps, int sms)
{
    WhgLaunch m = l;
    if (!l.auto_block || bk.nb < 2 || sms < 1) return m;
    const int per = (warps + sms - 1) / sms, w = per < 1 ? 1 : (per < WHG_MAX_BLOCK / 32 ? per : WHG_MAX_BLOCK / 32);
    m.block = 32 * w;
    m.grid = (warps + w - 1) / w;
    return m;
}

// The work queue balances SMs, but deals one-warp units of every lane-group size to
// all of them.  Ensembles of several sizes do without up to 128 warps per SM: us per
// step, queue / blocks as above: 9000 compact systems 18.3 / 8.2, 20,000 19.7 / 13.5,
// 65,536 39.1 / 36.7, 200,000 (217 warps per SM) 103.2 / 104.3.
bool whg_plain_steps(const WhgBuckets& bk, const WhgLaunch& l)
{
    return bk.warp0[bk.nb] <= (l.auto_block && bk.nb > 1 ? 128 : 8) * sm_count();
}

cudaError_t whg_launch_step(const WhgState& st, const WhgBuckets& bk, long long n, int newton_terms,
                            int gr_mode, const WhgLaunch& l)
{
    const int sms = l.sms > 0 ? l.sms : sm_count();
    const bool wide = wide_warps(st, bk, sms);
    const int warps = wide ? whg_wide_warps(bk) : bk.warp0[bk.nb];
    const WhgLaunch m = mixed_blocks(l, bk, warps, sms);
    if (wide)
        return newton_terms == 6 ? whg_launch_step_wide_nt6(st, bk, n, gr_mode, m)
                                 : whg_launch_step_wide_nt8(st, bk, n, gr_mode, m);
    if (warps <= 8 * sms)
        return newton_terms == 6 ? whg_launch_step_few_nt6(st, bk, n, gr_mode, m)
                                 : whg_launch_step_few_nt8(st, bk, n, gr_mode, m);
    return newton_terms == 6 ? whg_launch_step_nt6(st, bk, n, gr_mode, m)
                             : whg_launch_step_nt8(st, bk, n, gr_mode, m);
}

cudaError_t whg_launch_step_queue(const WhgState& st, const WhgBuckets& bk, long long n, int newton_terms,
                                  int gr_mode, const WhgQueue& q, cudaStream_t stream)
{
    return newton_terms == 6 ? whg_launch_step_queue_nt6(st, bk, n, gr_mode, q, stream)
                             : whg_launch_step_queue_nt8(st, bk, n, gr_mode, q, stream);
}

cudaError_t whg_launch_read(const WhgState& st, const WhgBuckets& bk, const WhgOut& o, int newton_terms,
                            const WhgLaunch& l)
{
    return newton_terms == 6 ? whg_launch_read_nt6(st, bk, o, l) : whg_launch_read_nt8(st, bk, o, l);
}

cudaError_t whg_launch_energy(const WhgState& st, const WhgBuckets& bk, const WhgOut& o, int newton_terms,
                              int gr_mode, const WhgLaunch& l)
{
    return newton_terms == 6 ? whg_launch_energy_nt6(st, bk, o, gr_mode, l)
                             : whg_launch_energy_nt8(st, bk, o, gr_mode, l);
}

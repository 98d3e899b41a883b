// sm_103a kernels of the interval-voting hot path (arXiv:2401.04576, Section 3.1):
// hit staging, coarse-grid voting, voting of explicit / bisected cells, top-K selection and
// the final max-vote estimate.
#include <cuda_runtime.h>

#include <climits>
#include <cstdint>

#include "../../include/apo.h"
#include "cert_vote.cuh"
#include "kernels.cuh"

namespace apo {

// ---------------------------------------------------------------------------------------
// Bulk (TMA) copy global -> shared with an mbarrier, every wait bounded.
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ unsigned smem_u32(const void *p) {
    return static_cast<unsigned>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t *bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_inval(uint64_t *bar) {
    asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, unsigned bytes, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
constexpr long kWaitLimit = 1L << 22;

// Waits for phase `parity` of an mbarrier for at most `limit` polls.  On running out it sets
// ST_TIMEOUT in *status (if given) and returns false; the caller then leaves the barrier's
// work undone and the kernel ends normally, so the context stays usable.
__device__ bool bounded_wait(uint64_t *bar, unsigned parity, long limit, unsigned *status) {
    for (long it = 0; it < limit; it++)
        if (mbar_try_wait(bar, parity)) return true;
    if (status) atomicOr(status, ST_TIMEOUT);
    return false;
}

// Copies up to two blocks (bytes0 / bytes1: multiples of 16, 16-byte aligned ends) of an
// event's hit records into shared memory with one mbarrier.  Returns false (and flags
// ST_TIMEOUT) if the copies did not complete within the wait limit; the caller then skips
// the block's work.
__device__ bool stage_to_smem(void *dst0, const void *src0, unsigned bytes0, void *dst1,
                              const void *src1, unsigned bytes1, uint64_t *bar, unsigned *status) {
    if (threadIdx.x == 0) {
        mbar_init(bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncthreads();
    if (bytes0 + bytes1 == 0) return true;
    if (threadIdx.x == 0) {
        mbar_expect_tx(bar, bytes0 + bytes1);
        if (bytes0) bulk_g2s(dst0, src0, bytes0, bar);
        if (bytes1) bulk_g2s(dst1, src1, bytes1, bar);
    }
    if (bounded_wait(bar, 0, kWaitLimit, status)) return true;
    // give the copies in flight a second bounded chance before leaving the shared memory
    bounded_wait(bar, 0, kWaitLimit, nullptr);
    return false;
}

// Diagnostic: every thread waits on an mbarrier whose expected bytes never arrive (no copy
// is issued, so nothing is in flight), with a short limit.  The wait must run out and
// report ST_TIMEOUT; used to test the timeout path without any device fault.
__global__ void k_wait_never(long limit, unsigned *status) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        mbar_expect_tx(&bar, 16);
    }
    __syncthreads();
    bounded_wait(&bar, 0, limit, status);
}

void launch_wait_never(long limit, unsigned *status, cudaStream_t s) {
    k_wait_never<<<1, 32, 0, s>>>(limit, status);
}

// ---------------------------------------------------------------------------------------
// Series constants [rd(1/k), ru(1/k)] computed once on the device.
// ---------------------------------------------------------------------------------------
__global__ void k_series_consts(SeriesConsts *out) {
    int i = threadIdx.x;
    if (i < 16) {
        int k = series_divisor(i);
        out->d_lo[i] = __drcp_rd((double)k);
        out->d_hi[i] = __drcp_ru((double)k);
        out->f_lo[i] = __frcp_rd((float)k);
        out->f_hi[i] = __frcp_ru((float)k);
    }
}

void launch_series_consts(SeriesConsts *dev_out, cudaStream_t s) {
    k_series_consts<<<1, 32, 0, s>>>(dev_out);
}

// ---------------------------------------------------------------------------------------
// Stage: gather each event's hits into contiguous FP64 and outward-rounded FP32 records,
// validating wire ids, drifts and hit counts.  n_hits[e] < 0 marks an invalid event.
// ---------------------------------------------------------------------------------------
__global__ void k_stage(DevGeom g, int n_events, const int32_t *offsets, const int32_t *wire_id,
                        const double *drift, HitRecD *hd, HitRecF *hf, int32_t *n_hits,
                        uint32_t *active, int32_t *done, unsigned *status, int32_t *hit_track) {
    int e = blockIdx.x;
    if (e >= n_events) return;
    __shared__ int bad;
    if (threadIdx.x == 0) bad = 0;
    __syncthreads();
    int a = offsets[e], b = offsets[e + 1];
    int n = b - a;
    if (n < 0 || a < 0 || n > kHitCap) {
        if (threadIdx.x < 8) active[(long long)e * 8 + threadIdx.x] = 0u;
        if (threadIdx.x == 0) {
            n_hits[e] = APO_EINVAL;
            done[e] = 0;
            atomicOr(status, n > kHitCap ? ST_TOOMANY : ST_BADOFFS);
        }
        return;
    }
    if (hit_track)
        for (int i = threadIdx.x; i < n; i += blockDim.x) hit_track[a + i] = -1;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        int w = wire_id[a + i];
        double d = drift[a + i];
        bool ok = (w >= 0 && w < g.n_wires && d >= 0.0 && d <= 1e300);
        if (!ok) { bad = 1; continue; }
        HitRecD rd;
        HitRecF rf;
        for (int j = 0; j < 8; j++) rd.v[j] = g.wire[j][w];
        rd.v[8] = d;
        rd.pad = 0.0;
        for (int j = 0; j < 9; j++) {
            rf.lo[j] = __double2float_rd(rd.v[j]);
            rf.hi[j] = __double2float_ru(rd.v[j]);
        }
        rf.pad[0] = rf.pad[1] = 0.f;
        hd[(long long)e * kHitCap + i] = rd;
        hf[(long long)e * kHitCap + i] = rf;
    }
    __syncthreads();
    if (threadIdx.x < 8) {   // every valid hit starts active
        int lo = 32 * threadIdx.x;
        uint32_t m = bad ? 0u : (n >= lo + 32 ? 0xffffffffu : (n > lo ? (1u << (n - lo)) - 1u : 0u));
        active[(long long)e * 8 + threadIdx.x] = m;
    }
    if (threadIdx.x == 0) {
        done[e] = 0;
        if (bad) { n_hits[e] = APO_EINVAL; atomicOr(status, ST_BADHIT); }
        else n_hits[e] = n;
    }
}

void launch_stage(const DevGeom &g, int n_events, const int32_t *offsets, const int32_t *wire_id,
                  const double *drift, HitRecD *hd, HitRecF *hf, int32_t *n_hits, uint32_t *active,
                  int32_t *done, unsigned *status, cudaStream_t s, int32_t *hit_track) {
    if (n_events <= 0) return;
    k_stage<<<n_events, 128, 0, s>>>(g, n_events, offsets, wire_id, drift, hd, hf, n_hits, active,
                                      done, status, hit_track);
}

// ---------------------------------------------------------------------------------------
// Coarse-grid voting.  A tile is the (d0, z0) cells of one (phi0 bin, omega bin), in two parts
// when they exceed a block; thread = (d0 bin, z0 bin), looping over the tan(lambda) bins, which
// share the tan(lambda)-free prefix of the program.  Before that, every hit is tested once on
// the tile's parent cell (all its d0, z0, tan(lambda) bins joined): interval operations are
// inclusion-isotonic and the guards only fire on a parent when they fire on a child, so a hit
// that fails there fails on every child cell; skipping it leaves every vote unchanged.
// Writes votes[e][lin], lin = d + Bd (p + Bp (w + Bw (z + Bz l))), or each tile's K best cells,
// and the per-event histogram of vote counts.
// ---------------------------------------------------------------------------------------
// The end of a coarse block: each thread's vote counts (its cell (d, p, w, z), tan(lambda) bins l0 .. l1 - 1)
// to vo or, with cand_k and every bin, the block's K best cells; the histogram added to hist_e
// (may be null).  hist_s: kHistBins zeros in shared memory.  The block has whole warps, and so at
// least a thread per tan(lambda) bin.
__device__ __forceinline__ void coarse_output(const DevGeom &g, const VotePlanes &pl, bool has_cell, int d, int p,
                                              int w, int z, int l0, int l1, uint32_t *hist_s, uint32_t *hist_e,
                                              int32_t *vo, uint64_t *cand_k, int32_t *cand_v, int K) {
    const int Bd = g.bins[0], Bp = g.bins[1], Bw = g.bins[2], Bz = g.bins[3], Bl = g.bins[4];
    const int tid = threadIdx.x, nthr = blockDim.x;
    auto vote_of = [&](int l) { return pl.get(l); };
    for (int l = l0; l < l1 && has_cell; l++) {
        const int v = vote_of(l);
        if (!cand_k) {
            long long lin = d + (long long)Bd * (p + (long long)Bp * (w + (long long)Bw * (z + (long long)Bz * l)));
            vo[lin] = v;
        }
        atomicAdd(&hist_s[v], 1u);
    }
    __syncthreads();
    for (int i = tid; i < kHistBins && hist_e; i += nthr)
        if (hist_s[i]) atomicAdd(&hist_e[i], hist_s[i]);
    if (cand_k) {
        // The part's K best cells by (votes desc, key asc), from its own histogram: every
        // cell above v_t, then the lowest keys at v_t.  Within a part, cells in the order
        // (tan(lambda) bin, thread) are in key order.  Any cell among the event's K best is
        // among its part's K best, so these candidates are all the selection needs.
        __shared__ int s_vt, s_need, s_above;
        // warp 0: suffix sums of the histogram from the top, 32 bins a step
        if (tid < 32) {
            int cum = 0;
            bool found = false;
            for (int top = kHistBins - 1; top >= 0 && !found; top -= 32) {
                const int v = top - tid;
                const int h = v >= 0 ? (int)hist_s[v] : 0;
                int inc = h;   // cells with votes in [v, top]
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, inc, o);
                    if (tid >= o) inc += y;
                }
                const unsigned hit = __ballot_sync(0xffffffffu, v >= 0 && cum + inc >= K);
                if (hit) {   // the first bin from the top where the count reaches K
                    const int b = __ffs(hit) - 1;
                    const int incb = __shfl_sync(0xffffffffu, inc, b), hb = __shfl_sync(0xffffffffu, h, b);
                    if (tid == 0) {
                        s_vt = top - b;
                        s_above = cum + incb - hb;
                        s_need = K - (cum + incb - hb);
                    }
                    found = true;
                } else {
                    cum += __shfl_sync(0xffffffffu, inc, 31);
                }
            }
            if (!found && tid == 0) {   // fewer than K cells in the part
                s_vt = -1;
                s_above = cum;
                s_need = 0;
            }
        }
        __syncthreads();
        const int vt = s_vt, need = s_need, above = s_above;
        const int lane = tid & 31, wid = tid >> 5, nwarps = nthr >> 5;
        const unsigned lt = (1u << lane) - 1u;
        // Ranks in key order ((tan(lambda) bin, thread) order): per bin and warp, counts of
        // cells above v_t / at v_t from ballots; exclusive prefixes over warps, then over
        // bins; a cell's rank is its bin's base + its warp's prefix + its lane's prefix.
        __shared__ int s_wa[8][32], s_wb[8][32], s_ba[33], s_bb[33];
        for (int l = 0; l < Bl; l++) {
            const int v = has_cell ? vote_of(l) : -1;
            const unsigned ma = __ballot_sync(0xffffffffu, v > vt), mb = __ballot_sync(0xffffffffu, v == vt);
            if (lane == 0) { s_wa[wid][l] = __popc(ma); s_wb[wid][l] = __popc(mb); }
        }
        __syncthreads();
        if (tid < Bl) {   // exclusive prefix over warps, bin by bin
            int ra = 0, rb = 0;
            for (int q = 0; q < nwarps; q++) {
                const int xa = s_wa[q][tid], xb = s_wb[q][tid];
                s_wa[q][tid] = ra;
                s_wb[q][tid] = rb;
                ra += xa;
                rb += xb;
            }
            s_ba[tid] = ra;   // the bin's totals, turned into bases below
            s_bb[tid] = rb;
        }
        __syncthreads();
        if (tid == 0) {   // exclusive prefix over bins
            int ra = 0, rb = 0;
            for (int l = 0; l < Bl; l++) {
                const int xa = s_ba[l], xb = s_bb[l];
                s_ba[l] = ra;
                s_bb[l] = rb;
                ra += xa;
                rb += xb;
            }
            s_ba[Bl] = ra;
            s_bb[Bl] = rb;
        }
        __syncthreads();
        for (int l = 0; l < Bl; l++) {
            const int v = has_cell ? vote_of(l) : -1;
            const bool a = v > vt, b = v == vt;
            const unsigned ma = __ballot_sync(0xffffffffu, a), mb = __ballot_sync(0xffffffffu, b);
            int pos = -1;
            if (a) {
                pos = s_ba[l] + s_wa[wid][l] + __popc(ma & lt);
            } else if (b) {
                const int rb = s_bb[l] + s_wb[wid][l] + __popc(mb & lt);
                if (rb < need) pos = above + rb;
            }
            if (pos >= 0 && pos < K) {   // always below K when the counts agree; never past it
                int idx[5] = {d, p, w, z, l};
                cand_k[pos] = pack_key(g, idx);
                cand_v[pos] = v;
            }
        }
        const int runB = s_bb[Bl];
        const int placed = above + (runB < need ? runB : need);
        for (int i = placed + tid; i < K; i += nthr) {   // a part with fewer than K cells
            cand_k[i] = 0;
            cand_v[i] = -1;
        }
    }
}

// Adds a thread's six work counts to the diagnostic counters: whole FP64 evaluations (with
// certified decisions: pairs left undecided), FP64 prefixes, FP64 tails, then the FP32 ones.
__device__ __forceinline__ void add_counts(unsigned long long *ctr, const unsigned (&cnt)[6]) {
    if (!ctr) return;
    const int slot[6] = {0, 1, 2, 4, 5, 6};
#pragma unroll
    for (int i = 0; i < 6; i++) {
        unsigned long long x = cnt[i];
        for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
        if ((threadIdx.x & 31) == 0 && x) atomicAdd(&ctr[slot[i]], x);
    }
}

// FP64 (K = 64), outward FP32 (K = 32) and midpoint-form voting, decided by certified FP32 values.
// Phase 1: the parent tests of the block's tiles, one (tile, hit) per thread, give the mask of hits
// that can vote and the error bound that every cell of a tile shares; phase 2 the tan(lambda) bins
// of a kept hit that the tile's cells can vote in, and for a hit without a bound (wide cells) one
// from its bins' boxes; phase 3, tile by tile and without barriers,
// the bare values per (cell, hit, bin), bit-sliced counters; undecided pairs go to the warp's queue.
// What bounds it: FP32 issue.  The FP64 pipe (about 1.7 directed operations per clock and SM)
// evaluated every pair before; now about one pair in 10^4 reaches it.  256 events on 16^5 cells:
// FP64 votes 377 -> 9.7 ms (K best per tile), midpoint form 1077 -> 5.3 ms; FP32 votes of 1024 events
// 55.7 -> 31.5 ms.  3.1 (FP32) and 2.9 (FP64) instructions a clock and SM of 4.
//
// FP32 pairs without a bound (wide cells) are the program's at once, all bins of a hit after one prefix: 256 events,
// 16x3x2x16x7 cells, 1.30 -> 0.56 ms; one event, 5x6x6x5x5 cells, 0.148 -> 0.088 ms.
//
// A block is 128 threads and takes up to four tiles, so that phases 1 and 2, whose chains a single
// tile cannot hide, keep all its warps busy (fewer where the launch would have too few blocks).
// Phase 2's bin tests take 39.5 ms to 33.4 (FP32, 1024 events); with one tile a block they cost more
// than they gave (41.3 -> 44.4 ms).
// Grids with few (d0, z0) cells put `group` tiles side by side in the block (full votes only: the K
// best are kept per tile), so that its warps stay full.
constexpr int kCoarseThreads = 128, kCoarseMaxGroup = 8, kCoarseRounds = 4;
// Fewest cells of a tile whose every kept hit is tested by bin: from there a block has its tiles one after
// another; side by side (64 cells or fewer) the test costs more than it saves.  256 events, FP32, with / without:
// 25 cells 0.95 / 0.84 ms, 64: 1.34 / 1.28, 81: 1.52 / 1.75, 128: 1.62 / 1.95 (FP64 likewise).
constexpr int kCoarseBinCells = 65;
struct CoarsePlan {
    int parts, per;          // parts of a (phi0, omega) tile's cells, cells of a part (= one tile)
    int group, tiles;        // tiles side by side, tiles per block (group or one after another)
    long long n_tiles;       // of one event
};
// n_ev: events of the launch
__host__ __device__ inline CoarsePlan coarse_plan(const DevGeom &g, bool lists, long long n_ev) {
    CoarsePlan P;
    const int n = g.bins[0] * g.bins[3];
    P.parts = (n + kCoarseThreads - 1) / kCoarseThreads;
    P.per = (n + P.parts - 1) / P.parts;
    P.n_tiles = (long long)P.parts * g.bins[1] * g.bins[2];
    const int fit = kCoarseThreads / P.per;
    P.group = lists || fit < 2 ? 1 : (fit > kCoarseMaxGroup ? kCoarseMaxGroup : fit);
    P.tiles = P.group;
    if (P.group == 1) {   // at least two waves of four blocks on 152 SMs
        const long long r = P.n_tiles * n_ev / (2 * 4 * 152);
        P.tiles = r < 1 ? 1 : (r > kCoarseRounds ? kCoarseRounds : (int)r);
    }
    return P;
}

struct CoarseSmem {   // of a cert coarse block; every offset a multiple of 16
    static constexpr size_t hits = 0;
    static constexpr size_t queue = kHitCap * 80;
    static constexpr size_t hist = queue + sizeof(WarpQueue) * (kCoarseThreads / 32);
    static constexpr size_t bar = hist + ((kHistBins * 4 + 15) & ~size_t(15));
    static constexpr size_t L = bar + 16;
    __host__ __device__ static size_t mask(int Bl) { return L + ((8 * (size_t)Bl + 15) & ~size_t(15)); }
    __host__ __device__ static size_t box(int Bl, const CoarsePlan &P) { return mask(Bl) + 32 * (size_t)P.tiles; }
    __host__ __device__ static size_t err(int Bl, const CoarsePlan &P) {
        return box(Bl, P) + ((sizeof(CertBox) * (size_t)P.tiles + 15) & ~size_t(15));
    }
    // per (tile, hit): the tan(lambda) bins in question, those without a bound; the (tile, hit)s of phase 2
    __host__ __device__ static size_t bins(int Bl, const CoarsePlan &P) {
        return err(Bl, P) + sizeof(float) * kHitCap * (size_t)P.tiles;
    }
    __host__ __device__ static size_t own(int Bl, const CoarsePlan &P) {
        return bins(Bl, P) + sizeof(uint32_t) * kHitCap * (size_t)P.tiles;
    }
    __host__ __device__ static size_t list(int Bl, const CoarsePlan &P) {
        return own(Bl, P) + sizeof(uint32_t) * kHitCap * (size_t)P.tiles;
    }
    __host__ __device__ static size_t total(int Bl, const CoarsePlan &P) {
        return list(Bl, P) + 16 + sizeof(uint16_t) * kHitCap * (size_t)P.tiles;
    }
};

// Tiles [tile0, tile0 + P.tiles) of event ev by one block of 128 threads; cand_e / cand_v: the
// event's candidate lists, Kc per tile (null: full votes to vo).
template <int K>
__device__ __forceinline__ void coarse_block(const DevGeom &g, const CoarsePlan &P, int ev, long long tile0,
                                             const HitRecD *hd, const HitRecF *hf, const int32_t *n_hits,
                                             const uint32_t *active, int32_t *vo, uint32_t *hist_e,
                                             unsigned *status, unsigned long long *ctr, unsigned char *smem,
                                             uint64_t *cand_k = nullptr, int32_t *cand_v = nullptr, int Kc = 0) {
    const int Bd = g.bins[0], Bp = g.bins[1], Bw = g.bins[2], Bz = g.bins[3], Bl = g.bins[4];
    const int ntile = Bd * Bz, nthr = kCoarseThreads, tid = threadIdx.x, lane = tid & 31;
    unsigned char *hs = smem + CoarseSmem::hits;
    WarpQueue &q = reinterpret_cast<WarpQueue *>(smem + CoarseSmem::queue)[tid >> 5];
    uint32_t *hist_s = reinterpret_cast<uint32_t *>(smem + CoarseSmem::hist);
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem + CoarseSmem::bar);
    float2 *Ls = reinterpret_cast<float2 *>(smem + CoarseSmem::L);
    uint32_t *mask_s = reinterpret_cast<uint32_t *>(smem + CoarseSmem::mask(Bl));
    CertBox *box_s = reinterpret_cast<CertBox *>(smem + CoarseSmem::box(Bl, P));
    float *err_s = reinterpret_cast<float *>(smem + CoarseSmem::err(Bl, P));
    uint32_t *bins_s = reinterpret_cast<uint32_t *>(smem + CoarseSmem::bins(Bl, P));
    uint32_t *own_s = reinterpret_cast<uint32_t *>(smem + CoarseSmem::own(Bl, P));
    uint32_t *n_list = reinterpret_cast<uint32_t *>(smem + CoarseSmem::list(Bl, P));
    uint16_t *list_s = reinterpret_cast<uint16_t *>(n_list + 4);
    const unsigned all = Bl >= 32 ? 0xffffffffu : ((1u << Bl) - 1u);
    const bool outgoing = g.k.outgoing != 0, single = P.group == 1;
    const HitRecD *hd_e = hd + (long long)ev * kHitCap;
    const HitRecF *hf_e = hf + (long long)ev * kHitCap;

    int nh = n_hits[ev];
    if (nh < 0) nh = 0;
    for (int i = tid; i < kHistBins; i += nthr) hist_s[i] = 0;
    for (int i = tid; i < 8 * P.tiles; i += nthr) mask_s[i] = 0;
    for (int l = tid; l < Bl; l += nthr) Ls[l] = Prog<K>::tanl(edge(g, 4, 0, l));
    if (tid == 0) *n_list = 0;
    for (int i = tid; i < P.tiles; i += nthr) {   // the tiles' parents
        const long long t = tile0 + i;
        if (t >= P.n_tiles) break;
        const int part = (int)(t % P.parts), pw = (int)(t / P.parts), p = pw % Bp, w = pw / Bp;
        const int c0 = part * P.per, c1 = c0 + P.per < ntile ? c0 + P.per : ntile;
        const bool row = c0 / Bd == (c1 - 1) / Bd;   // cells of one z0 bin
        const int i0[5] = {row ? c0 % Bd : 0, p, w, c0 / Bd, 0};
        const int i1[5] = {row ? (c1 - 1) % Bd : Bd - 1, p, w, (c1 - 1) / Bd, Bl - 1};
        box_s[i] = cert_span<K>(g, 0, i0, i1);
    }
    const bool ok = stage_to_smem(hs, hf_e, (unsigned)nh * 80u, nullptr, nullptr, 0u, bar, status);
    __syncthreads();
    if (tid == 0) mbar_inval(bar);   // the barrier's memory may be set up again by a later call
    if (!ok) nh = 0;
    unsigned cnt[6] = {0, 0, 0, 0, 0, 0};

    // phase 1: a warp's 32 items are one word of one tile's hit mask
    const uint32_t *act = active ? active + (long long)ev * 8 : nullptr;
    const int nw = (nh + 31) >> 5;
    for (int i = tid; i < P.tiles * nw * 32; i += nthr) {
        const int tl = i / (nw * 32), h = i - tl * nw * 32;
        const long long t = tile0 + tl;
        bool keep = h < nh && t < P.n_tiles && (!act || ((act[h >> 5] >> (h & 31)) & 1u));
        float e = NAN;
        if (keep) {
            e = box_error<K>(box_s + tl, hs + h * 80, outgoing);
            keep = !(e < 0.f);
            cnt[3]++;
        }
        const unsigned m = __ballot_sync(0xffffffffu, keep);
        if (lane == 0) mask_s[tl * 8 + (h >> 5)] = m;
        if (keep) {
            const int x = tl * kHitCap + h;
            const bool ok = e < 1e30f, test = !box_s[tl].guard && (!ok || P.per >= kCoarseBinCells);
            err_s[x] = ok ? e : 0.f;
            bins_s[x] = test ? 0u : all;
            own_s[x] = 0u;
            if (test) list_s[atomicAdd(n_list, 1u)] = (uint16_t)(x | (ok ? 0 : 1 << 15));
        }
    }
    __syncthreads();
    // phase 2: one (tile, hit, bin) per thread.  Of 16^5 cells' (tile, hit, bin)s a quarter of those
    // phase 1 kept go, and with them their tails; tiles of few cells would spend more here than
    // that, so there only the hits without a bound come: a box of one bin mostly has one.
    {
        const int n = (int)*n_list * Bl;
        for (int i = tid; i < n; i += nthr) {
            const int y = list_s[i / Bl], x = y & 0x7fff, l = i % Bl, tl = x / kHitCap;
            const void *rec = hs + (x % kHitCap) * 80;
            const float2 L = K == kMid ? make_float2(Ls[l].x, Ls[l].x) : Ls[l];   // its centre: a point
            if (!(y >> 15)) {
                if (!box_refuses<K>(box_s + tl, L, rec, err_s[x], outgoing)) atomicOr(&bins_s[x], 1u << l);
                cnt[3]++;
            } else {
                CertBox b = box_s[tl];
                b.v[5] = L;
                const float e = box_error<K>(&b, rec, outgoing);
                if (!(e < 0.f)) atomicOr(e < 1e30f ? &bins_s[x] : &own_s[x], 1u << l);
                if (e >= 0.f && e < 1e30f) atomicMax(reinterpret_cast<int *>(&err_s[x]), __float_as_int(e));
            }
        }
    }
    __syncthreads();

    // phase 3
    for (int r = 0; r < (single ? P.tiles : 1); r++) {
        const int tl = single ? r : tid / P.per;
        const long long t = tile0 + tl;
        const int part = (int)(t % P.parts), pw = (int)(t / P.parts);
        const int k = single ? tid : tid - tl * P.per, cell = part * P.per + k;
        const bool has = tl < P.tiles && t < P.n_tiles && k < P.per && cell < ntile;
        const int p = has ? pw % Bp : 0, w = has ? pw / Bp : 0;
        const int d = has ? cell % Bd : 0, z = has ? cell / Bd : 0;
        if (single && t >= P.n_tiles) break;
        VotePlanes pl;
        pl.clear();
        const Cell<double> c64{edge(g, 0, 0, d), sin_phi0(g, 0, p), cos_phi0(g, 0, p), edge(g, 2, 0, w),
                               edge(g, 3, 0, z), {0.0, 0.0}};
        bool guard;
        const bool mir = omega_sign<K>(c64.W, &guard);
        const typename Prog<K>::CellT c = Prog<K>::cell(g, 0, p, c64, mir);
        // another lane's pair: its cell from its number
        auto solve = [&](int ol, int oh, bool own, uint32_t om) -> uint32_t {
            const int ot = (tid & ~31) + ol, otl = single ? r : ot / P.per;
            const long long u = tile0 + otl;
            const int oc = (int)(u % P.parts) * P.per + (single ? ot : ot - otl * P.per), opw = (int)(u / P.parts);
            return resolve<K>(g, 0, oc % Bd, opw % Bp, opw / Bp, oc / Bd, 0, om, own, hd_e + oh, hf_e + oh);
        };
        auto take = [&](uint32_t v) { pl.add(v); };
        int nq = 0, wd = -1;
        uint32_t m = 0;
        for (;;) {
            while (has && !m && ++wd < nw) m = mask_s[tl * 8 + wd];
            const bool more = __any_sync(0xffffffffu, m != 0u);
            uint32_t unk = 0;
            int h = 0;
            bool own = false;
            if (m) {
                h = wd * 32 + __ffs(m) - 1;
                m &= m - 1;
                const float e = err_s[tl * kHitCap + h];
                uint32_t lm = bins_s[tl * kHitCap + h], yes = 0;
                own = true;   // a level-0 cell's own bound is several times a tile's
                if (guard) {
                    yes = all;
                } else {
                    unk = own_s[tl * kHitCap + h];
                    if (K == 32 && unk) {   // the tile's lanes share the bins: no queue
                        yes = program_f32(g, c64, 0, 0, unk, hs + h * 80);
                        unk = 0u;
                    }
                }
                if (!guard && lm) {
                    const typename Prog<K>::HitT hx = Prog<K>::hit(hs + h * 80, mir);
                    const typename Prog<K>::Pre pre = Prog<K>::prefix(c, hx);
                    cnt[4]++;
                    const int dir = settle_direction<K>(Prog<K>::direction(pre, outgoing, e), c64, hd_e + h, hs + h * 80);
                    if (dir == cert::kNo) unk = 0;
                    if (dir == cert::kYes) {
                        cnt[5] += __popc(lm);
#pragma unroll 1
                        while (lm) {
                            const int l = __ffs(lm) - 1;
                            lm &= lm - 1;
                            const int v = Prog<K>::vote(pre, Ls[l], c, hx, e);
                            yes |= (uint32_t)(v == cert::kYes) << l;
                            unk |= (uint32_t)(v == cert::kUnknown) << l;
                        }
                    }
                }
                pl.add(yes);
                cnt[0] += __popc(unk);
            }
            if (more) nq = q.push(nq, lane, h, own, unk);
            if (nq >= 32 || (!more && nq)) {
                q.drain(nq, lane, solve, take);
                nq = 0;
            }
            if (!more) break;
        }
        if (cand_k) {
            coarse_output(g, pl, has, d, p, w, z, 0, Bl, hist_s, hist_e, nullptr, cand_k + t * Kc, cand_v + t * Kc, Kc);
            __syncthreads();
            for (int i = tid; i < kHistBins; i += nthr) hist_s[i] = 0;
            __syncthreads();
        } else {
            for (int l = 0; l < Bl && has; l++) {
                const int v = pl.get(l);
                vo[d + (long long)Bd * (p + (long long)Bp * (w + (long long)Bw * (z + (long long)Bz * l)))] = v;
                atomicAdd(&hist_s[v], 1u);
            }
        }
    }
    if (!cand_k) {
        __syncthreads();
        for (int i = tid; i < kHistBins && hist_e; i += nthr)
            if (hist_s[i]) atomicAdd(&hist_e[i], hist_s[i]);
    }
    add_counts(ctr, cnt);
    __syncthreads();   // shared memory is reused by the caller's next step
}

// Resident blocks per SM the compiler plans for: caps registers at 64K / (128 x this).
#ifndef APO_COARSE_MIN_BLOCKS
#define APO_COARSE_MIN_BLOCKS 4
#endif
template <int K>
__global__ void __launch_bounds__(kCoarseThreads, APO_COARSE_MIN_BLOCKS)
k_vote_coarse(const __grid_constant__ DevGeom g, CoarsePlan P, int ev0, const HitRecD *hd, const HitRecF *hf,
              const int32_t *n_hits, const uint32_t *active, int32_t *votes, uint32_t *hist, unsigned *status,
              unsigned long long *ctr, uint64_t *cand_k, int32_t *cand_v, int Kc, const int32_t *skip) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int e = blockIdx.y;
    if (skip && skip[ev0 + e]) return;
    const long long ncell = (long long)g.bins[0] * g.bins[1] * g.bins[2] * g.bins[3] * g.bins[4];
    // candidates: Kc slots per tile, an event's tiles in order
    const long long co = (long long)e * P.n_tiles * Kc;
    coarse_block<K>(g, P, ev0 + e, (long long)blockIdx.x * P.tiles, hd, hf, n_hits, active,
                    votes ? votes + (long long)e * ncell : nullptr,
                    hist ? hist + (long long)e * kHistBins : nullptr, status, ctr, smem,
                    cand_k ? cand_k + co : nullptr, cand_v ? cand_v + co : nullptr, Kc);
}

// The exact-phase program on the coarse grid: FP64, the same tiles.  Full votes: a block takes
// `group` tiles side by side, so that its 128 threads have a cell each, and gridDim.z blocks share their
// tan(lambda) bins where there are too few; K best lists: one tile, in whole warps.  Never fewer
// than 32 threads: the mask's words, and the bins' prefixes of coarse_output, are one thread's each.
// One event, exact phase: 10^5 cells 7.9 -> 4.3 ms with the bins shared, max-set search on 2x256x16x2x8 26.0 -> 21.8 ms
// (23.4 with one cell per thread); 16 events of 10^5 the same.
constexpr int kExactMaxGroup = 32;
struct ExactSmem {
    static constexpr size_t hits = 0;
    static constexpr size_t hist = kHitCap * 80;
    static constexpr size_t mask = hist + ((kHistBins * 4 + 15) & ~size_t(15));
    static constexpr size_t bar = mask + 32 * kExactMaxGroup;
    static constexpr size_t L = bar + 16;
    __host__ __device__ static size_t total(int Bl) { return L + 16 * (size_t)Bl; }
};
struct ExactPlan {
    CoarsePlan P;
    int threads, split;
};
__host__ inline ExactPlan exact_plan(const DevGeom &g, bool lists, int n_ev) {
    ExactPlan E{coarse_plan(g, true, 1), 0, 1};
    const int fit = kCoarseThreads / E.P.per;
    E.P.group = E.P.tiles = lists || fit < 2 ? 1 : (fit > kExactMaxGroup ? kExactMaxGroup : fit);
    E.threads = (E.P.group * E.P.per + 31) & ~31;
    if (!lists) {   // two waves of three blocks on 152 SMs
        const long long blocks = (E.P.n_tiles + E.P.group - 1) / E.P.group * n_ev, want = 2 * 3 * 152;
        E.split = blocks >= want ? 1 : (int)((want + blocks - 1) / blocks);
        if (E.split > g.bins[4]) E.split = g.bins[4];
    }
    return E;
}

__global__ void __launch_bounds__(kCoarseThreads, 3)
k_vote_coarse_exact(DevGeom g, CoarsePlan P, int ev0, const HitRecD *hd, const int32_t *n_hits, const uint32_t *active,
                    int32_t *votes, uint32_t *hist, unsigned *status, unsigned long long *ctr, uint64_t *cand_k,
                    int32_t *cand_v, int Kc, const int32_t *skip) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int e = blockIdx.y, ev = ev0 + e;
    if (skip && skip[ev]) return;
    const int Bd = g.bins[0], Bp = g.bins[1], Bz = g.bins[3], Bl = g.bins[4];
    const int ntile = Bd * Bz, nthr = blockDim.x, tid = threadIdx.x, lane = tid & 31;
    const long long tile0 = (long long)blockIdx.x * P.group;
    const int l0 = (int)(blockIdx.z * Bl / gridDim.z), l1 = (int)((blockIdx.z + 1) * Bl / gridDim.z);   // its bins
    unsigned char *hs = smem + ExactSmem::hits;
    uint32_t *hist_s = reinterpret_cast<uint32_t *>(smem + ExactSmem::hist);
    uint32_t *mask_s = reinterpret_cast<uint32_t *>(smem + ExactSmem::mask);
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem + ExactSmem::bar);
    IV<double> *Ls = reinterpret_cast<IV<double> *>(smem + ExactSmem::L);
    int nh = n_hits[ev];
    if (nh < 0) nh = 0;
    for (int i = tid; i < kHistBins; i += nthr) hist_s[i] = 0;
    for (int i = tid; i < 8 * P.group; i += nthr) mask_s[i] = 0;
    for (int l = tid; l < Bl; l += nthr) Ls[l] = edge(g, 4, 0, l);
    const bool ok = stage_to_smem(hs, hd + (long long)ev * kHitCap, (unsigned)nh * 80u, nullptr, nullptr, 0u, bar,
                                  status);
    __syncthreads();
    if (!ok) nh = 0;
    const SeriesConsts &k = g.k;
    unsigned cnt[6] = {0, 0, 0, 0, 0, 0};
    const uint32_t *act = active ? active + (long long)ev * 8 : nullptr;
    const int nw = (nh + 31) >> 5;
    // a warp's 32 items are one word of one tile's hit mask
    for (int i = tid; i < P.group * nw * 32; i += nthr) {
        const int tl = i / (nw * 32), h = i - tl * nw * 32;
        const long long t = tile0 + tl;
        bool keep = h < nh && t < P.n_tiles && (!act || ((act[h >> 5] >> (h & 31)) & 1u));
        if (keep) {
            const int pw = (int)(t / P.parts), p = pw % Bp, w = pw / Bp;
            const int c0 = (int)(t % P.parts) * P.per, c1 = c0 + P.per < ntile ? c0 + P.per : ntile;
            const bool row = c0 / Bd == (c1 - 1) / Bd;   // cells of one z0 bin
            const Cell<double> par{edge_span(g, 0, 0, row ? c0 % Bd : 0, row ? (c1 - 1) % Bd : Bd - 1), sin_phi0(g, 0, p),
                                   cos_phi0(g, 0, p), edge(g, 2, 0, w), edge_span(g, 3, 0, c0 / Bd, (c1 - 1) / Bd),
                                   edge_span(g, 4, 0, l0, l1 - 1)};
            cnt[0]++;
            keep = vote_pair_exact(par, load_hit<double>(hs + h * 80), k);
        }
        const unsigned m = __ballot_sync(0xffffffffu, keep);
        if (lane == 0) mask_s[tl * 8 + (h >> 5)] = m;
    }
    __syncthreads();
    const int tl = tid / P.per, kc = tid - tl * P.per;
    const long long t = tile0 + tl;
    const int part = (int)(t % P.parts), pw = (int)(t / P.parts), cell = part * P.per + kc;
    const bool has_cell = tl < P.group && t < P.n_tiles && cell < ntile;   // other threads idle
    const int p = has_cell ? pw % Bp : 0, w = has_cell ? pw / Bp : 0;
    const int d = has_cell ? cell % Bd : 0, z = has_cell ? cell / Bd : 0;
    Cell<double> c{edge(g, 0, 0, d), sin_phi0(g, 0, p), cos_phi0(g, 0, p), edge(g, 2, 0, w), edge(g, 3, 0, z), Ls[0]};
    const bool mir = mirror_cell(c);
    const bool wguard = !gt0(c.W.lo);
    const IV<double> R = recip(c.W);
    const unsigned all = Bl >= 32 ? 0xffffffffu : ((1u << Bl) - 1u);
    VotePlanes pl;
    pl.clear();
    for (int wd = 0; wd < nw && has_cell; wd++) {
        uint32_t m = mask_s[tl * 8 + wd];
        while (m) {
            const int h = wd * 32 + __ffs(m) - 1;
            m &= m - 1;
            if (wguard) { pl.add(all); continue; }
            Hit<double> hx = load_hit<double>(hs + h * 80);
            if (mir) mirror_hit(hx);
            const Pre<double> pre = prefix<double>(c, hx, k);
            cnt[1]++;
            if (pre.novote) continue;
            if (pre.guard) { pl.add(all); continue; }
            uint32_t v = 0;
#pragma unroll 1
            for (int l = l0; l < l1; l++)
                if (tail_exact(pre, Ls[l], hx, R, c.W, k)) v |= 1u << l;
            cnt[2] += l1 - l0;
            pl.add(v);
        }
    }
    const long long ncell = (long long)ntile * Bp * g.bins[2] * Bl;
    const long long co = ((long long)e * gridDim.x + blockIdx.x) * Kc;   // lists: one tile a block
    coarse_output(g, pl, has_cell, d, p, w, z, l0, l1, hist_s, hist ? hist + (long long)e * kHistBins : nullptr,
                  votes ? votes + (long long)e * ncell : nullptr, cand_k ? cand_k + co : nullptr,
                  cand_v ? cand_v + co : nullptr, Kc);
    add_counts(ctr, cnt);
}

// ---------------------------------------------------------------------------------------
// Midpoint-form voting (APO_F64_MID, Section 3.1's variant with the quantities of d^Ax at
// the voxel centre) of explicit cells; level 0 and bisected cells are coarse_block<kMid> and
// children_block<kMid>.
// ---------------------------------------------------------------------------------------
// One cell per thread, all hits of its event.
__global__ void __launch_bounds__(256)
k_vote_cells_mid(DevGeom g, const HitRecD *hd, const int32_t *n_hits, const uint32_t *active, int level,
                 const uint64_t *keys, long long n_per_ev, int32_t *out_votes, unsigned *status) {
    extern __shared__ __align__(16) unsigned char smem[];
    unsigned char *hs = smem;
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem + kHitCap * 80);
    const int ev = blockIdx.y;
    int nh = n_hits[ev];
    if (nh < 0) nh = 0;
    bool ok = stage_to_smem(hs, hd + (long long)ev * kHitCap, (unsigned)nh * 80u, nullptr, nullptr, 0u,
                            bar, status);
    __syncthreads();
    if (!ok) nh = 0;
    const long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n_per_ev) return;
    int idx[5];
    unpack_key(g, keys[(long long)ev * n_per_ev + j], idx);
    const long long o = (long long)ev * n_per_ev + j;
    bool valid = true;
#pragma unroll
    for (int a = 0; a < 5; a++) valid = valid && idx[a] < (g.bins[a] << level);
    if (!valid) {   // a key outside the grid of this level: no lookup, vote count -1
        out_votes[o] = -1;
        return;
    }
    const IV<double> Le = edge(g, 4, level, idx[4]);
    const Cell<double> c{edge(g, 0, level, idx[0]), sin_phi0(g, level, idx[1]), cos_phi0(g, level, idx[1]),
                         edge(g, 2, level, idx[2]), edge(g, 3, level, idx[3]), Le};
    MidCentre m;
    sincos_phi0_centre(g, level, idx[1], m.S0, m.C0);
    m.D = pt::centre(c.D);
    m.W = pt::centre(c.W);
    m.Z = pt::centre(c.Z);
    const double Lm = pt::centre(Le);
    const uint32_t *act = active ? active + (long long)ev * 8 : nullptr;
    int v = 0;
    for (int h = 0; h < nh; h++) {
        if (act && !((act[h >> 5] >> (h & 31)) & 1u)) continue;
        v += mid_vote_pair(c, m, Lm, load_hit<double>(hs + h * 80)) ? 1 : 0;
    }
    out_votes[o] = v;
}

template <int K> static void launch_coarse_cert(const DevGeom &g, int ev0, int n_ev, const HitRecD *hd,
                                               const HitRecF *hf, const int32_t *n_hits, const uint32_t *active,
                                               int32_t *votes, uint32_t *hist, unsigned *status, cudaStream_t s,
                                               unsigned long long *ctr, uint64_t *cand_k, int32_t *cand_v, int Kc,
                                               const int32_t *skip) {
    const CoarsePlan P = coarse_plan(g, cand_k != nullptr, n_ev);
    dim3 grid((unsigned)((P.n_tiles + P.tiles - 1) / P.tiles), n_ev);
    k_vote_coarse<K><<<grid, kCoarseThreads, CoarseSmem::total(g.bins[4], P), s>>>(
        g, P, ev0, hd, hf, n_hits, active, votes, hist, status, ctr, cand_k, cand_v, Kc, skip);
}

int coarse_lists(const DevGeom &g, int) { return (int)coarse_plan(g, true, 1).n_tiles; }

void launch_vote_coarse(const DevGeom &g, int prec, int ev0, int n_ev, const HitRecD *hd,
                        const HitRecF *hf, const int32_t *n_hits, int32_t *votes, uint32_t *hist,
                        unsigned *status, cudaStream_t s, unsigned long long *ctr,
                        const uint32_t *active, uint64_t *cand_k, int32_t *cand_v, int K, const int32_t *skip) {
    if (n_ev <= 0) return;
    if (prec == APO_F64_MID) {
        launch_coarse_cert<kMid>(g, ev0, n_ev, hd, hf, n_hits, active, votes, hist, status, s, ctr, cand_k, cand_v, K, skip);
    } else if (prec == APO_F64_EXACT) {
        const ExactPlan E = exact_plan(g, cand_k != nullptr, n_ev);
        dim3 grid((unsigned)((E.P.n_tiles + E.P.group - 1) / E.P.group), n_ev, E.split);
        k_vote_coarse_exact<<<grid, E.threads, ExactSmem::total(g.bins[4]), s>>>(
            g, E.P, ev0, hd, n_hits, active, votes, hist, status, ctr, cand_k, cand_v, K, skip);
    } else if (prec == APO_F32) {
        launch_coarse_cert<32>(g, ev0, n_ev, hd, hf, n_hits, active, votes, hist, status, s, ctr, cand_k, cand_v, K, skip);
    } else {   // APO_F64 and APO_F64_FILTERED: the same votes, the same kernel
        launch_coarse_cert<64>(g, ev0, n_ev, hd, hf, n_hits, active, votes, hist, status, s, ctr, cand_k, cand_v, K, skip);
    }
}

// ---------------------------------------------------------------------------------------
// Voting of explicit cells given by keys, one per thread, looping over all hits of its event.
// The cell of a key: false when the key lies outside the level's grid.
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ bool key_cell(const DevGeom &g, int level, uint64_t key, int idx[5], Cell<double> &c) {
    unpack_key(g, key, idx);
    bool valid = true;
#pragma unroll
    for (int a = 0; a < 5; a++) valid = valid && idx[a] < (g.bins[a] << level);
    if (valid)
        c = Cell<double>{edge(g, 0, level, idx[0]), sin_phi0(g, level, idx[1]), cos_phi0(g, level, idx[1]),
                         edge(g, 2, level, idx[2]), edge(g, 3, level, idx[3]), edge(g, 4, level, idx[4])};
    return valid;
}
// Floats in the order of signed integers (an involution), and the smallest range around a warp's.
__device__ __forceinline__ int fkey(float x) { const int b = __float_as_int(x); return b ^ ((b >> 31) & 0x7fffffff); }
__device__ __forceinline__ float2 warp_range(float lo, float hi) {
    const int l = __reduce_min_sync(0xffffffffu, fkey(lo)), h = __reduce_max_sync(0xffffffffu, fkey(hi));
    return make_float2(__int_as_float(l ^ ((l >> 31) & 0x7fffffff)), __int_as_float(h ^ ((h >> 31) & 0x7fffffff)));
}
// The smallest box around the cells of the warp's lanes (`has`; at least one), from their FP32 ends v.  One
// that reaches omega = 0 is a guard: it has no bound.
__device__ __forceinline__ CertBox warp_box(const float2 (&v)[6], bool has) {
    CertBox b;
#pragma unroll
    for (int q = 0; q < 6; q++) b.v[q] = warp_range(has ? v[q].x : INFINITY, has ? v[q].y : -INFINITY);
    b.mir = b.v[3].y < 0.f;
    b.guard = !b.mir && !(b.v[3].x > 0.f);
    if (b.mir)
        for (int q = 0; q < 4; q++)
            if (q != 2) b.v[q] = make_float2(-b.v[q].y, -b.v[q].x);
    return b;
}

// FP64 (K = 64) and outward FP32 (K = 32) votes, decided by certified FP32 end points (see
// coarse_block).  The parent is the smallest box around the warp's 32 cells: for the 32 children
// of one cell, as apo_refine lists them, that cell; for scattered keys it is wide, or holds both signs
// of omega, and decides little.  FP64 pairs then go one by one with their own bounds.  FP32 pairs are
// the program's: all of them where no hit has a bound, or those of the first hit that leaves a quarter of the
// lanes undecided and of the hits after it.
// FP64, the children of 33 kept cells of 37 events: 0.76 -> 0.055 ms.  FP32, 8 events x 65536 keys within three
// cells of a track's: 0.23 ms, scattered: 0.30 ms; children of 2048 cells of 16 events: 0.32 ms (the program alone,
// one key a thread: 0.27, 0.27 and 0.49 ms; pairs one by one as in FP64: 0.30, 0.63 and 0.42 ms).
constexpr int kCellsThreads = 128, kCellsOpen = 8;   // undecided lanes from which a warp stops certifying
struct WarpScratch {   // one warp's parent, and its queue
    CertBox box;
    float err[kHitCap];
    uint32_t mask[8];
    WarpQueue q;
};
struct CellsSmem {
    static constexpr size_t hits = 0;
    static constexpr size_t warp = kHitCap * 80;
    static constexpr size_t bar = warp + sizeof(WarpScratch) * (kCellsThreads / 32);
    static constexpr size_t total = bar + 16;
};
template <int K>
__global__ void __launch_bounds__(kCellsThreads, 4)
k_vote_cells(const __grid_constant__ DevGeom g, const HitRecD *hd, const HitRecF *hf, const int32_t *n_hits,
             const uint32_t *active, int level, const uint64_t *keys, long long n_per_ev, int32_t *out_votes,
             unsigned *status) {
    extern __shared__ __align__(16) unsigned char smem[];
    unsigned char *hs = smem + CellsSmem::hits;
    const int tid = threadIdx.x, lane = tid & 31, ev = blockIdx.y;
    WarpScratch &ws = reinterpret_cast<WarpScratch *>(smem + CellsSmem::warp)[tid >> 5];
    const bool outgoing = g.k.outgoing != 0;
    int nh = n_hits[ev];
    if (nh < 0) nh = 0;
    const HitRecD *hd_e = hd + (long long)ev * kHitCap;
    const HitRecF *hf_e = hf + (long long)ev * kHitCap;
    const bool ok = stage_to_smem(hs, hf_e, (unsigned)nh * 80u, nullptr, nullptr, 0u,
                                  reinterpret_cast<uint64_t *>(smem + CellsSmem::bar), status);
    __syncthreads();
    if (!ok) nh = 0;
    const int nw = (nh + 31) >> 5;
    const uint32_t *act = active ? active + (long long)ev * 8 : nullptr;
    const long long j0 = (long long)blockIdx.x * kCellsThreads + (tid & ~31), j = j0 + lane;   // this warp's keys
    const uint64_t *keys_e = keys + (long long)ev * n_per_ev;
    Cell<double> c64{};
    int idx[5] = {0, 0, 0, 0, 0};
    const bool in = j < n_per_ev, has = in && key_cell(g, level, keys_e[j], idx, c64);
    // the cell's FP32 ends: rounded to nearest, or outward for the FP32 program (converted once: conversions
    // from FP64 run on its pipe)
    float2 fe[6];
    const IV<double> de[6] = {c64.D, c64.S0, c64.C0, c64.W, c64.Z, c64.L};
#pragma unroll
    for (int q = 0; q < 6; q++) {
        const IV<float> o = to_prec<float>(de[q]);
        fe[q] = K == 32 ? make_float2(o.lo, o.hi) : make_float2((float)de[q].lo, (float)de[q].hi);
    }
    // the warp's parent, one hit per lane; without one when the cells are on both sides of omega = 0
    bool plain = !__any_sync(0xffffffffu, has) ||
                 (__any_sync(0xffffffffu, has && fe[3].y < 0.f) && __any_sync(0xffffffffu, has && !(fe[3].y < 0.f)));
    if (!plain) {
        const CertBox box = warp_box(fe, has);
        // a hull over more than a radian of phi0 has hardly a bound
        plain = K == 32 && (box.v[1].y - box.v[1].x > 1.f || box.v[2].y - box.v[2].x > 1.f);
        if (lane == 0) ws.box = box;
        __syncwarp();
    }
    {
        bool open = true;
        for (int h = lane; h < nw * 32; h += 32) {
            bool keep = h < nh && (!act || ((act[h >> 5] >> (h & 31)) & 1u));
            float e = NAN;
            if (keep && !plain) e = box_error<K>(&ws.box, hs + h * 80, outgoing);
            open = open && !(e < 1e30f);
            keep = keep && !(e < 0.f);
            ws.err[h] = e;
            const unsigned m = __ballot_sync(0xffffffffu, keep);
            if (lane == 0) ws.mask[h >> 5] = m;
        }
        plain = plain || __all_sync(0xffffffffu, open);
        __syncwarp();
    }
    bool guard;
    const bool mir = omega_sign<K>(c64.W, &guard);
    auto flip = [&](int q) { return mir ? cert::X<0>{-fe[q].y, -fe[q].x, 0.f} : cert::X<0>{fe[q].x, fe[q].y, 0.f}; };
    const cert::CellX<0> c{flip(0), flip(1), xf<0>(fe[2]), flip(3), xf<0>(fe[4]), xf<0>(fe[5])};
    const cert::X<0> R = cert::recip(c.W);
    int v = 0, nq = 0, wd = 0;
    uint32_t m = nw ? ws.mask[0] : 0u;
    auto next = [&]() {   // the next hit in question, the same for all lanes; -1: none left
        while (!m && ++wd < nw) m = ws.mask[wd];
        return m ? wd * 32 + __ffs(m) - 1 : -1;
    };
    auto solve = [&](int ol, int oh, bool own, uint32_t om) -> uint32_t {
        int x[5];
        unpack_key(g, keys_e[j0 + ol], x);
        return resolve<K>(g, level, x[0], x[1], x[2], x[3], x[4], om, own, hd_e + oh, hf_e + oh);
    };
    auto take = [&](uint32_t b) { v += (int)b; };
    for (int h; !(K == 32 && plain) && (h = next()) >= 0; m &= m - 1) {
        const float e = ws.err[h];
        int r = has ? (guard ? cert::kYes : cert::kUnknown) : cert::kNo;
        if (r == cert::kUnknown && e < 1e30f) {
            const cert::HitX<0> hx = cert_hit<0>(hs + h * 80, mir);
            const cert::PreX<0> pre = cert::prefix(c, hx);
            r = cert_direction(pre, outgoing, e);
            if (r == cert::kYes) r = cert_tail(pre, c.L, hx, R, c.W, e);
        }
        const unsigned open = __ballot_sync(0xffffffffu, r == cert::kUnknown);
        if (K == 32 && __popc(open) >= kCellsOpen) break;
        v += r == cert::kYes;
        // the keys need not be one cell's children: their own bounds first (FP64)
        nq = ws.q.push(nq, lane, h, true, r == cert::kUnknown ? 1u : 0u);
        if (nq >= 32) {
            ws.q.drain(nq, lane, solve, take);
            nq = 0;
        }
    }
    if (nq) ws.q.drain(nq, lane, solve, take);
    if constexpr (K == 32) {   // what is left
        IV<float> f[6];
#pragma unroll
        for (int q = 0; q < 6; q++) f[q] = {fe[q].x, fe[q].y};
        Cell<float> x{f[0], f[1], f[2], f[3], f[4], f[5]};
        mirror_cell(x);
        const bool all = le0(x.W.lo);
        const IV<float> Rx = recip(x.W);
        for (int h; (h = next()) >= 0; m &= m - 1) {
            if (!has) continue;
            Hit<float> hx = load_hit<float>(hs + h * 80);
            if (mir) mirror_hit(hx);
            const Pre<float> p = prefix(x, hx, g.k);
            v += all || (!p.novote && (p.guard || tail(p, x.L, hx, Rx, x.W, g.k)));
        }
    }
    if (in) out_votes[(long long)ev * n_per_ev + j] = has ? v : -1;   // -1: a key outside the level's grid
}

// The exact-phase program on explicit cells, FP64.
__global__ void __launch_bounds__(256)
k_vote_cells_exact(DevGeom g, const HitRecD *hd, const int32_t *n_hits, const uint32_t *active, int level,
                   const uint64_t *keys, long long n_per_ev, int32_t *out_votes, unsigned *status) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int ev = blockIdx.y;
    int nh = n_hits[ev];
    if (nh < 0) nh = 0;
    const bool ok = stage_to_smem(smem, hd + (long long)ev * kHitCap, (unsigned)nh * 80u, nullptr, nullptr, 0u,
                                  reinterpret_cast<uint64_t *>(smem + kHitCap * 80), status);
    __syncthreads();
    if (!ok) nh = 0;
    const long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n_per_ev) return;
    const uint32_t *act = active ? active + (long long)ev * 8 : nullptr;
    int idx[5], v = -1;   // -1: a key outside the level's grid
    Cell<double> c;
    if (key_cell(g, level, keys[(long long)ev * n_per_ev + j], idx, c)) {
        v = 0;
        for (int h = 0; h < nh; h++) {
            if (act && !((act[h >> 5] >> (h & 31)) & 1u)) continue;
            v += vote_pair_exact(c, load_hit<double>(smem + h * 80), g.k) ? 1 : 0;
        }
    }
    out_votes[(long long)ev * n_per_ev + j] = v;
}

// Children of kept cells, two per thread: the children 2 idx + bit of a parent that differ
// only in the tan(lambda) bit share every tan(lambda)-free step of the program, so one
// prefix per hit serves both tails.  Pair j of an event: children 2 idx + bit of parent j / 16
// for the bit pattern b = j % 16 on d0 .. z0, with tan(lambda) bit 0 and 1 (slots
// 32 (j / 16) + b and + 16 of the event's outputs).
__device__ __forceinline__ void pair_index(const DevGeom &g, uint64_t parent, int b, int idx[5]) {
    unpack_key(g, parent, idx);
#pragma unroll
    for (int a = 0; a < 4; a++) idx[a] = 2 * idx[a] + ((b >> a) & 1);
    idx[4] = 2 * idx[4];   // tan(lambda) bit 0
}
__device__ __forceinline__ void pair_store(const DevGeom &g, const int idx[5], long long j, int v0, int v1,
                                           uint64_t *out_keys_e, int32_t *out_votes_e) {
    const uint64_t key0 = pack_key(g, idx);
    const long long o = (j / 16) * 32 + j % 16;
    out_keys_e[o] = key0;
    out_votes_e[o] = v0;
    out_keys_e[o + 16] = key0 + (1ULL << g.key_shift[4]);
    out_votes_e[o + 16] = v1;
}

// FP64 (K = 64), outward FP32 (K = 32) and midpoint-form votes of the children, decided by certified
// FP32 values (see coarse_block).  A warp takes `np` parents, two at a time, and works by itself: no
// block barrier after the hits are staged.  One evaluation with errors per (parent, hit) gives the
// bound that the parent's 32 children share, and drops the hits that none of them can get.  Undecided
// pairs collect over all the warp's parents.  FP32 issue and instruction fetch bound it: the
// evaluation with errors and the reference program are long straight code, so a warp runs them
// rarely and on as many lanes as there are (eight parents a warp; with two, 24 multi-track events took 133 ms
// instead of 118).  Before, every child hit that passed an FP32 test was evaluated on the FP64 pipe:
// 160 events of the max-set schedule, FP64 level 366 -> 13.6 ms, the FP32 levels 21.3 -> 15.7 ms.
constexpr int kChildThreads = 128, kChildParents = 8;   // most parents of a warp
struct ChildScratch {
    CertBox box[kChildParents];
    float2 axis[kChildParents][2][6];   // the children's ends per axis, bit 0 and 1: conversions from
                                        // FP64, which run on its pipe, once per parent
    uint16_t err[kChildParents][kHitCap];   // bounds as bf16 rounded up: four blocks fit an SM
    uint32_t mask[kChildParents][8];
    WarpQueue q;
};
struct ChildSmem {
    static constexpr size_t hits = 0;
    static constexpr size_t warp = kHitCap * 80;
    static constexpr size_t bar = warp + sizeof(ChildScratch) * (kChildThreads / 32);
    static constexpr size_t total = bar + 16;
};
// A bound >= 0 (or NaN) as bf16, rounded up.
__device__ __forceinline__ uint16_t bound_up(float e) {
    return e < 1e30f ? (uint16_t)((__float_as_uint(e) + 0xffffu) >> 16) : (uint16_t)0x7fc0u;
}
// Parents per warp (even): eight where that leaves four waves of 16 warps on each of 152 SMs, else
// fewer (256 events x 64 parents: two a warp 2.05 ms, six 2.78 ms, FP32 levels of 1024 events).
__device__ __forceinline__ int child_parents(long long n_par) {
    const long long r = n_par / (4 * 152 * 16) & ~1LL;
    return r < 2 ? 2 : (r > kChildParents ? kChildParents : (int)r);
}

// Children of parents [p0, p0 + np) of one event, those below n_par, by one warp; hits staged at hs.
template <int K>
__device__ __forceinline__ void children_warp(const DevGeom &g, const unsigned char *hs, ChildScratch &ws, int nh,
                                              const uint32_t *act, int level, const uint64_t *parents_e, long long p0,
                                              int np, long long n_par, const HitRecD *hd_e, const HitRecF *hf_e,
                                              uint64_t *out_keys_e, int32_t *out_votes_e) {
    const int lane = threadIdx.x & 31;
    const bool outgoing = g.k.outgoing != 0;
    if (n_par - p0 < np) np = (int)(n_par - p0);
    for (int i = lane; i < 8 * kChildParents; i += 32) ws.mask[i >> 3][i & 7] = 0u;
    if constexpr (K == kMid) {
        if (lane < np) {
            int x[5];
            unpack_key(g, parents_e[p0 + lane], x);
#pragma unroll
            for (int a = 0; a < 5; a++) x[a] *= 2;
            const int x1[5] = {x[0] + 1, x[1] + 1, x[2] + 1, x[3] + 1, x[4] + 1};
            ws.box[lane] = cert_span<K>(g, level, x, x1);
        }
    } else {
        for (int i = lane; i < np * 12; i += 32) {
            const int pl = i / 12, q = i % 6, bit = i / 6 & 1;
            int x[5];
            unpack_key(g, parents_e[p0 + pl], x);
            const int at = q == 0 ? x[0] : q < 3 ? x[1] : q == 3 ? x[2] : q == 4 ? x[3] : x[4];
            ws.axis[pl][bit][q] = axis_float(g, level, q, 2 * at + bit);
        }
        __syncwarp();
        if (lane < np) ws.box[lane] = float_box(ws.axis[lane]);
    }
    __syncwarp();
    for (int i = lane; i < np * nh; i += 32) {
        const int pl = i / nh, h = i - pl * nh;
        if (act && !((act[h >> 5] >> (h & 31)) & 1u)) continue;
        const float e = box_error<K>(&ws.box[pl], hs + h * 80, outgoing);
        if (e < 0.f) continue;
        ws.err[pl][h] = bound_up(e);
        atomicOr(&ws.mask[pl][h >> 5], 1u << (h & 31));
    }
    // keys, and votes from 0: counted votes and those of undecided pairs are added as they come
    for (int i = lane; i < np * 16; i += 32) {
        int x[5];
        pair_index(g, parents_e[p0 + (i >> 4)], i & 15, x);
        pair_store(g, x, p0 * 16 + i, 0, 0, out_keys_e, out_votes_e);
    }
    __syncwarp();
    const int nw = (nh + 31) >> 5;
    int nq = 0;
    // one undecided pair (16 parent + child bits)
    auto finish = [&](int pair, int oh, bool own, uint32_t om) {
        int x[5];
        pair_index(g, parents_e[p0 + (pair >> 4)], pair & 15, x);
        const uint32_t y = resolve<K>(g, level, x[0], x[1], x[2], x[3], x[4], om, own, hd_e + oh, hf_e + oh);
        const long long o = (p0 + (pair >> 4)) * 32 + (pair & 15);
        if (y & 1u) atomicAdd(&out_votes_e[o], 1);
        if (y & 2u) atomicAdd(&out_votes_e[o + 16], 1);
    };
#pragma unroll 1
    for (int s = 0; s < np; s += 2) {
        const int pl = s + (lane >> 4);
        const bool has = pl < np;
        bool guard = false, mir;
        typename Prog<K>::CellT c;
        float2 L0, L1;
        if constexpr (K == kMid) {
            int idx[5] = {0, 0, 0, 0, 0};
            if (has) pair_index(g, parents_e[p0 + pl], lane & 15, idx);
            const Cell<double> c64{edge(g, 0, level, idx[0]), sin_phi0(g, level, idx[1]), cos_phi0(g, level, idx[1]),
                                   edge(g, 2, level, idx[2]), edge(g, 3, level, idx[3]), edge(g, 4, level, idx[4])};
            mir = omega_sign<K>(c64.W, &guard);
            c = Prog<K>::cell(g, level, idx[1], c64, mir);
            L0 = Prog<K>::tanl(c64.L);
            L1 = Prog<K>::tanl(edge(g, 4, level, idx[4] + 1));
        } else {
            const int bit[4] = {lane & 1, lane >> 1 & 1, lane >> 2 & 1, lane >> 3 & 1}, pa = has ? pl : 0;
            mir = ws.axis[pa][bit[2]][3].y < 0.f;
            c = Prog<K>::cell(ws.axis[pa], bit, mir);
            L0 = ws.axis[pa][0][5];
            L1 = ws.axis[pa][1][5];
        }
        int v0 = 0, v1 = 0, wd = -1;
        uint32_t m = 0;
        for (;;) {
            while (has && !m && ++wd < nw) m = ws.mask[pl][wd];
            const bool more = __any_sync(0xffffffffu, m != 0u);
            uint32_t unk = 0;
            int h = 0;
            bool own = false;
            if (m) {
                h = wd * 32 + __ffs(m) - 1;
                m &= m - 1;
                const float e = __uint_as_float((unsigned)ws.err[pl][h] << 16);
                if (guard) {
                    v0++;
                    v1++;
                } else if (!(e < 1e30f)) {
                    if constexpr (K == 32) {
                        int x[5];
                        pair_index(g, parents_e[p0 + pl], lane & 15, x);
                        const uint32_t y = resolve<K>(g, level, x[0], x[1], x[2], x[3], x[4], 3u, true, nullptr, hs + h * 80);
                        v0 += y & 1u;
                        v1 += y >> 1;
                    } else {
                        unk = 3u;
                        own = true;
                    }
                } else {
                    const typename Prog<K>::HitT hx = Prog<K>::hit(hs + h * 80, mir);
                    const typename Prog<K>::Pre pre = Prog<K>::prefix(c, hx);
                    const int dir = Prog<K>::direction(pre, outgoing, e);
                    if (dir == cert::kUnknown) unk = 3u;
                    if (dir == cert::kYes) {
#pragma unroll 1
                        for (int b = 0; b < 2; b++) {
                            const int v = Prog<K>::vote(pre, b ? L1 : L0, c, hx, e);
                            if (v == cert::kYes) { if (b) v1++; else v0++; }
                            unk |= (uint32_t)(v == cert::kUnknown) << b;
                        }
                    }
                }
            }
            if (more) nq = ws.q.push(nq, 16 * s + lane, lane, h, own, unk);
            if (nq >= 32 || (!more && s + 2 >= np && nq)) {
                ws.q.drain(nq, lane, finish);
                nq = 0;
            }
            if (!more) break;
        }
        if (v0) atomicAdd(&out_votes_e[(p0 + pl) * 32 + (lane & 15)], v0);
        if (v1) atomicAdd(&out_votes_e[(p0 + pl) * 32 + (lane & 15) + 16], v1);
    }
}

#ifndef APO_CHILD_MIN_BLOCKS
#define APO_CHILD_MIN_BLOCKS 4
#endif
template <int K>
__global__ void __launch_bounds__(kChildThreads, APO_CHILD_MIN_BLOCKS)
k_vote_children(const __grid_constant__ DevGeom g, const HitRecD *hd, const HitRecF *hf, const int32_t *n_hits,
                const uint32_t *active, int level, const uint64_t *parents, int n_par,
                const int32_t *n_valid, uint64_t *out_keys, int32_t *out_votes, unsigned *status, const int32_t *skip) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int ev = blockIdx.y;
    if (skip && skip[ev]) return;
    // n_valid (may be null): parents 0 .. n_valid[ev] - 1 of the event's n_par slots are
    // real; a block past them has nothing to do (the condition is uniform in the block)
    const long long n_here = n_valid ? (long long)n_valid[ev] : (long long)n_par;
    const int np = child_parents(n_here * gridDim.y);
    const long long b0 = (long long)blockIdx.x * np * (kChildThreads / 32);   // the block's first parent
    if (b0 >= n_here) return;
    int nh = n_hits[ev];
    if (nh < 0) nh = 0;
    const bool ok = stage_to_smem(smem + ChildSmem::hits, hf + (long long)ev * kHitCap, (unsigned)nh * 80u, nullptr,
                                  nullptr, 0u, reinterpret_cast<uint64_t *>(smem + ChildSmem::bar), status);
    __syncthreads();
    if (!ok) nh = 0;
    const long long p0 = b0 + (long long)(threadIdx.x >> 5) * np;
    if (p0 >= n_here) return;
    children_warp<K>(g, smem + ChildSmem::hits, reinterpret_cast<ChildScratch *>(smem + ChildSmem::warp)[threadIdx.x >> 5],
                     nh, active ? active + (long long)ev * 8 : nullptr, level, parents + (long long)ev * n_par, p0, np,
                     n_here, hd + (long long)ev * kHitCap, hf + (long long)ev * kHitCap,
                     out_keys + (long long)ev * n_par * 32, out_votes + (long long)ev * n_par * 32);
}

// The exact-phase program on children, FP64.  NT: threads per block, 256 or 128; the 128-thread
// form asks for three resident blocks per SM (12 warps), which the register count otherwise
// limits to 8 warps.
template <int NT>
__global__ void __launch_bounds__(NT, NT == 128 ? 3 : 1)
k_vote_children_exact(DevGeom g, const HitRecD *hd, const int32_t *n_hits, const uint32_t *active, int level,
                      const uint64_t *parents, int n_par, const int32_t *n_valid, uint64_t *out_keys,
                      int32_t *out_votes, unsigned *status, const int32_t *skip) {
    extern __shared__ __align__(16) unsigned char smem[];
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem + kHitCap * 80);
    const int ev = blockIdx.y;
    if (skip && skip[ev]) return;
    const long long n_here = n_valid ? (long long)n_valid[ev] : (long long)n_par;
    if ((long long)blockIdx.x * blockDim.x >= n_here * 16) return;
    int nh = n_hits[ev];
    if (nh < 0) nh = 0;
    const bool ok = stage_to_smem(smem, hd + (long long)ev * kHitCap, (unsigned)nh * 80u, nullptr, nullptr, 0u, bar,
                                  status);
    __syncthreads();
    if (!ok) nh = 0;
    const long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n_here * 16) return;
    const uint32_t *act = active ? active + (long long)ev * 8 : nullptr;
    int idx[5];
    pair_index(g, parents[(long long)ev * n_par + j / 16], (int)(j % 16), idx);
    Cell<double> c{edge(g, 0, level, idx[0]), sin_phi0(g, level, idx[1]), cos_phi0(g, level, idx[1]),
                   edge(g, 2, level, idx[2]), edge(g, 3, level, idx[3]), edge(g, 4, level, idx[4])};
    const IV<double> L1 = edge(g, 4, level, idx[4] + 1);
    const bool mir = mirror_cell(c);
    const bool wguard = !gt0(c.W.lo);
    const IV<double> R = recip(c.W);
    int v0 = 0, v1 = 0;
    for (int h = 0; h < nh; h++) {
        if (act && !((act[h >> 5] >> (h & 31)) & 1u)) continue;
        if (wguard) { v0++; v1++; continue; }
        Hit<double> hx = load_hit<double>(smem + h * 80);
        if (mir) mirror_hit(hx);
        const Pre<double> pre = prefix<double>(c, hx, g.k);
        if (pre.novote) continue;
        if (pre.guard) { v0++; v1++; continue; }
        if (tail_exact(pre, c.L, hx, R, c.W, g.k)) v0++;
        if (tail_exact(pre, L1, hx, R, c.W, g.k)) v1++;
    }
    pair_store(g, idx, j, v0, v1, out_keys + (long long)ev * n_par * 32, out_votes + (long long)ev * n_par * 32);
}

void launch_vote_keys(const DevGeom &g, int prec, int n_ev, const HitRecD *hd, const HitRecF *hf,
                      const int32_t *n_hits, int level, const uint64_t *keys, long long n_per_ev,
                      int32_t *votes, cudaStream_t s, const uint32_t *active) {
    if (n_ev <= 0 || n_per_ev <= 0) return;
    dim3 grid((unsigned)((n_per_ev + kCellsThreads - 1) / kCellsThreads), n_ev);
    if (prec == APO_F64_MID) {
        k_vote_cells_mid<<<dim3((unsigned)((n_per_ev + 255) / 256), n_ev), 256, kHitCap * 80 + 16, s>>>(
            g, hd, n_hits, active, level, keys, n_per_ev, votes, nullptr);
    } else if (prec == APO_F64_EXACT) {
        k_vote_cells_exact<<<dim3((unsigned)((n_per_ev + 255) / 256), n_ev), 256, kHitCap * 80 + 16, s>>>(
            g, hd, n_hits, active, level, keys, n_per_ev, votes, nullptr);
    } else if (prec == APO_F32) {
        k_vote_cells<32><<<grid, kCellsThreads, CellsSmem::total, s>>>(g, hd, hf, n_hits, active, level, keys, n_per_ev,
                                                                       votes, nullptr);
    } else {   // APO_F64 and APO_F64_FILTERED: the same votes, the same kernel
        k_vote_cells<64><<<grid, kCellsThreads, CellsSmem::total, s>>>(g, hd, hf, n_hits, active, level, keys, n_per_ev,
                                                                       votes, nullptr);
    }
}

template <int K>
static void launch_children_cert(const DevGeom &g, int n_ev, const HitRecD *hd, const HitRecF *hf,
                                 const int32_t *n_hits, const uint32_t *active, int level, const uint64_t *parents,
                                 int n_par, const int32_t *n_valid, uint64_t *out_keys, int32_t *out_votes,
                                 cudaStream_t s, const int32_t *skip) {
    dim3 grid((unsigned)(((long long)n_par + kChildThreads / 16 - 1) / (kChildThreads / 16)), n_ev);   // two parents a warp
    k_vote_children<K><<<grid, kChildThreads, ChildSmem::total, s>>>(g, hd, hf, n_hits, active, level, parents, n_par,
                                                                     n_valid, out_keys, out_votes, nullptr, skip);
}

void launch_vote_children(const DevGeom &g, int prec, int n_ev, const HitRecD *hd,
                          const HitRecF *hf, const int32_t *n_hits, int child_level,
                          const uint64_t *parents, int n_par, uint64_t *child_keys,
                          int32_t *child_votes, cudaStream_t s, const uint32_t *active, int block,
                          const int32_t *n_valid, const int32_t *skip) {
    if (n_ev <= 0 || n_par <= 0) return;
    if (block != 128) block = 256;   // of the exact-phase kernel
    if (prec == APO_F64_MID) {
        launch_children_cert<kMid>(g, n_ev, hd, hf, n_hits, active, child_level, parents, n_par, n_valid, child_keys,
                                   child_votes, s, skip);
    } else if (prec == APO_F64_EXACT) {
        const size_t sm = kHitCap * 80 + 16;
        dim3 grid((unsigned)(((long long)n_par * 16 + block - 1) / block), n_ev);
        if (block == 128)
            k_vote_children_exact<128><<<grid, 128, sm, s>>>(g, hd, n_hits, active, child_level, parents, n_par, n_valid,
                                                             child_keys, child_votes, nullptr, skip);
        else
            k_vote_children_exact<256><<<grid, 256, sm, s>>>(g, hd, n_hits, active, child_level, parents, n_par, n_valid,
                                                             child_keys, child_votes, nullptr, skip);
    } else if (prec == APO_F32) {
        launch_children_cert<32>(g, n_ev, hd, hf, n_hits, active, child_level, parents, n_par, n_valid, child_keys,
                                 child_votes, s, skip);
    } else {   // APO_F64 and APO_F64_FILTERED: the same votes, the same kernel
        launch_children_cert<64>(g, n_ev, hd, hf, n_hits, active, child_level, parents, n_par, n_valid, child_keys,
                                 child_votes, s, skip);
    }
}

// Sets every vote kernel's dynamic shared-memory limit now, outside any stream capture.
void init_kernel_attributes() {
    const int lim = 96 * 1024;   // on the current device, every time a geometry is created there
    cudaFuncSetAttribute(k_vote_coarse<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    cudaFuncSetAttribute(k_vote_coarse<kMid>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    cudaFuncSetAttribute(k_vote_children<kMid>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    cudaFuncSetAttribute(k_vote_coarse<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    cudaFuncSetAttribute(k_vote_coarse_exact, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    cudaFuncSetAttribute(k_vote_children<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    cudaFuncSetAttribute(k_vote_children<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    cudaFuncSetAttribute(k_vote_children_exact<256>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    cudaFuncSetAttribute(k_vote_children_exact<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    cudaFuncSetAttribute(k_vote_cells<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    cudaFuncSetAttribute(k_vote_cells<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
}

// ---------------------------------------------------------------------------------------
// Coarse top-K: threshold from the vote histogram, then an order-preserving compaction.
// Keeps every cell with votes above the threshold v* and the lowest-key cells at v*, so the
// kept set is the K best by (votes desc, key asc).  From the histogram: A = #(v > v*) < K
// and need = K - A.  One pass over the event's votes in key order, 4096 cells per tile,
// each thread 4 consecutive cells (one 16-byte load where aligned); cells above v* go to
// slot (rank among them), cells at v* to slot A + (rank among them) while that is < K.
// A tile with nothing to keep costs one barrier; the pass ends once all A cells and
// `need` tied cells are placed.  Votes are clamped to [0, kHitCap] as the histogram does.
// ---------------------------------------------------------------------------------------
constexpr int kSelThreads = 1024;
constexpr int kSelTile = 4 * kSelThreads;

// One event's selection by one block of any multiple-of-32 size (tiles of 4 cells per
// thread): vo = the event's level-0 votes, hist_e its histogram, ok_ / ov its K outputs.
__device__ __forceinline__ void select_coarse_block(const DevGeom &g, const int32_t *vo, const uint32_t *hist_e,
                                                    int K, uint64_t *ok_, int32_t *ov) {
    __shared__ int s_vstar, s_need, s_above;
    __shared__ int s_warp[32];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nwarps = blockDim.x >> 5;
    const long long tile = 4LL * blockDim.x;
    const long long n = (long long)g.bins[0] * g.bins[1] * g.bins[2] * g.bins[3] * g.bins[4];
    if (tid == 0) {
        long long cum = 0;
        int vstar = -1, need = 0;
        for (int v = kHistBins - 1; v >= 0; v--) {
            long long h = hist_e[v];
            if (cum + h >= K) { vstar = v; need = (int)(K - cum); break; }
            cum += h;
        }
        s_vstar = vstar;
        s_need = need;
        s_above = (int)cum;
    }
    __syncthreads();
    const int vstar = s_vstar, need = s_need, above = s_above;
    const bool vec = (n % 4 == 0) && ((reinterpret_cast<uintptr_t>(vo) & 15) == 0);
    int runA = 0, runB = 0;   // cells above v* / at v* in the tiles before this one
    for (long long t0 = 0; t0 < n; t0 += tile) {
        if (runA >= above && runB >= need) break;
        const long long j0 = t0 + 4LL * tid;
        int v[4];
        if (vec && j0 + 3 < n) {
            int4 q = __ldcs(reinterpret_cast<const int4 *>(vo + j0));
            v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
        } else {
#pragma unroll
            for (int r = 0; r < 4; r++) v[r] = j0 + r < n ? __ldcs(vo + j0 + r) : INT_MIN;
        }
        int a = 0, b = 0;
#pragma unroll
        for (int r = 0; r < 4; r++) {
            if (v[r] != INT_MIN) v[r] = v[r] < 0 ? 0 : (v[r] > kHitCap ? kHitCap : v[r]);
            a += v[r] > vstar;
            b += v[r] == vstar;
        }
        if (!__syncthreads_or(a > 0 || (b > 0 && runB < need))) continue;
        // block exclusive scan of (a, b) packed as a + (b << 16); a tile holds < 2^16 cells
        const int x = a + (b << 16);
        int inc = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        if (lane == 31) s_warp[wid] = inc;
        __syncthreads();
        int w = lane < nwarps ? s_warp[lane] : 0;
        int winc = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, winc, o);
            if (lane >= o) winc += y;
        }
        const int wpre = __shfl_sync(0xffffffffu, winc - w, wid);
        const int total = __shfl_sync(0xffffffffu, winc, 31);
        const int pre = wpre + inc - x;
        int pa = runA + (pre & 0xffff), pb = runB + (pre >> 16);
#pragma unroll
        for (int r = 0; r < 4; r++) {
            const bool ka = v[r] > vstar, kb = v[r] == vstar;
            int pos = -1;
            if (ka) pos = pa++;
            else if (kb) { if (pb < need) pos = above + pb; pb++; }
            if (pos >= 0 && pos < K) {
                long long rr = j0 + r;
                int idx[5];
                for (int q = 0; q < 5; q++) { idx[q] = (int)(rr % g.bins[q]); rr /= g.bins[q]; }
                ok_[pos] = pack_key(g, idx);
                ov[pos] = v[r];
            }
        }
        runA += total & 0xffff;
        runB += total >> 16;
        __syncthreads();   // s_warp is rewritten by the next scanned tile
    }
    __syncthreads();
}

__global__ void __launch_bounds__(kSelThreads)
k_select_coarse(DevGeom g, int ev0, const int32_t *votes, const uint32_t *hist, int K,
                uint64_t *out_keys, int32_t *out_votes, const int32_t *skip) {
    const int e = blockIdx.x, ev = ev0 + e;
    if (skip && skip[ev]) return;
    const long long n = (long long)g.bins[0] * g.bins[1] * g.bins[2] * g.bins[3] * g.bins[4];
    select_coarse_block(g, votes + (long long)e * n, hist + (long long)e * kHistBins, K,
                        out_keys + (long long)ev * K, out_votes + (long long)ev * K);
}

// Top-K of level 0 from the coarse blocks' candidates (see launch_vote_coarse): the same v*
// and need from the event's histogram as k_select_coarse; every candidate above v* is kept
// (there are exactly `above` of them), then the `need` lowest keys at v*.  In each block's
// list the candidates at v* come in key order, so the lowest keys overall come from a
// merge: `need` rounds, each taking the smallest head over the lists.
__global__ void __launch_bounds__(kSelThreads)
k_select_candidates(int ev0, const uint64_t *cand_k, const int32_t *cand_v, int n_lists,
                    const uint32_t *hist, int K, uint64_t *out_keys, int32_t *out_votes, const int32_t *skip) {
    extern __shared__ int s_head[];          // n_lists heads
    __shared__ int s_vstar, s_need, s_above, s_nA;
    __shared__ unsigned long long s_red[32];
    const int e = blockIdx.x, ev = ev0 + e, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    if (skip && skip[ev]) return;
    const uint64_t *ck = cand_k + (long long)e * n_lists * K;
    const int32_t *cv = cand_v + (long long)e * n_lists * K;
    uint64_t *ok_ = out_keys + (long long)ev * K;
    int32_t *ov = out_votes + (long long)ev * K;
    if (tid == 0) {
        long long cum = 0;
        int vstar = -1, need = 0;
        for (int v = kHistBins - 1; v >= 0; v--) {
            long long h = hist[(long long)e * kHistBins + v];
            if (cum + h >= K) { vstar = v; need = (int)(K - cum); break; }
            cum += h;
        }
        s_vstar = vstar;
        s_need = need;
        s_above = (int)cum;
        s_nA = 0;
    }
    __syncthreads();
    const int vstar = s_vstar, need = s_need, above = s_above;
    for (long long i = tid; i < (long long)n_lists * K; i += blockDim.x) {
        const int v = cv[i];
        if (v > vstar) {
            const int pos = atomicAdd(&s_nA, 1);
            if (pos < K) { ok_[pos] = ck[i]; ov[pos] = v; }
        }
    }
    for (int t = tid; t < n_lists; t += blockDim.x) {
        int j = 0;
        while (j < K && cv[(long long)t * K + j] != vstar) j++;
        s_head[t] = j;
    }
    __syncthreads();
    const int nwarps = blockDim.x >> 5;
    for (int r = 0; r < need; r++) {
        unsigned long long best = ~0ULL;   // (key << 13) | list: keys of at most 50 bits
        for (int t = tid; t < n_lists; t += blockDim.x) {
            const int j = s_head[t];
            if (j < K) {
                const unsigned long long x = (ck[(long long)t * K + j] << 13) | (unsigned long long)t;
                best = x < best ? x : best;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long y = __shfl_down_sync(0xffffffffu, best, o);
            best = y < best ? y : best;
        }
        if (lane == 0) s_red[wid] = best;
        __syncthreads();
        if (tid == 0) {
            unsigned long long b = ~0ULL;
            for (int q = 0; q < nwarps; q++) b = s_red[q] < b ? s_red[q] : b;
            const int t = (int)(b & 8191ULL);
            ok_[above + r] = b >> 13;
            ov[above + r] = vstar;
            int j = s_head[t] + 1;
            while (j < K && cv[(long long)t * K + j] != vstar) j++;
            s_head[t] = j;
        }
        __syncthreads();
    }
}

void launch_select_candidates(const DevGeom &, int ev0, int n_ev, const uint64_t *cand_k,
                              const int32_t *cand_v, int n_lists, const uint32_t *hist, int K,
                              uint64_t *out_keys, int32_t *out_votes, cudaStream_t s, const int32_t *skip) {
    if (n_ev <= 0) return;
    k_select_candidates<<<n_ev, kSelThreads, sizeof(int) * (size_t)n_lists, s>>>(
        ev0, cand_k, cand_v, n_lists, hist, K, out_keys, out_votes, skip);
}

void launch_select_coarse(const DevGeom &g, int ev0, int n_ev, const int32_t *votes,
                          const uint32_t *hist, int K, uint64_t *out_keys, int32_t *out_votes,
                          cudaStream_t s, const int32_t *skip) {
    if (n_ev <= 0) return;
    k_select_coarse<<<n_ev, kSelThreads, 0, s>>>(g, ev0, votes, hist, K, out_keys, out_votes, skip);
}

// ---------------------------------------------------------------------------------------
// Per-event bitonic sort of (votes desc, key asc) packed as ((1023 - v) << 50) | key.
// ---------------------------------------------------------------------------------------
constexpr int kSortMax = 4096;
// One warp sorts or merges 64 entries, two a lane, in registers: the bitonic steps of block sizes
// size0 .. size1 with strides below 64.
__device__ __forceinline__ void warp_sort64(uint64_t *s, int base, int size0, int size1) {
    const int lane = threadIdx.x & 31, i = base + lane;
    uint64_t a = s[i], b = s[i + 32];
    for (int size = size0; size <= size1; size <<= 1) {
        const bool ua = (i & size) == 0, ub = ((i + 32) & size) == 0;
        if (size >= 64 && (a > b) == ua) { const uint64_t x = a; a = b; b = x; }
        for (int st = size >= 64 ? 16 : size >> 1; st > 0; st >>= 1) {
            const uint64_t pa = __shfl_xor_sync(0xffffffffu, a, st), pb = __shfl_xor_sync(0xffffffffu, b, st);
            const bool low = (lane & st) == 0;
            a = (low == ua) == (pa < a) ? pa : a;
            b = (low == ub) == (pb < b) ? pb : b;
        }
    }
    s[i] = a;
    s[i + 32] = b;
}
// Ascending bitonic sort by the block (whole warps).  Steps with strides below 64 run in registers,
// one pass per block size instead of six (2048 entries: 15 passes through shared memory and 6
// through registers instead of 66; the six levels of 1024 events 0.77 -> 0.46 ms).
__device__ void block_sort(uint64_t *s, int n_pow2) {
    const int wid = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const bool regs = n_pow2 >= 64;
    if (regs) {
        for (int base = 64 * wid; base < n_pow2; base += 64 * nwarps) warp_sort64(s, base, 2, 64);
        __syncthreads();
    }
    for (int size = regs ? 128 : 2; size <= n_pow2; size <<= 1) {
        for (int stride = size >> 1; stride > (regs ? 32 : 0); stride >>= 1) {
            for (int i = threadIdx.x; i < n_pow2 / 2; i += blockDim.x) {
                int lo = 2 * i - (i & (stride - 1));
                int hi = lo + stride;
                bool up = ((lo & size) == 0);
                uint64_t x = s[lo], y = s[hi];
                if ((x > y) == up) { s[lo] = y; s[hi] = x; }
            }
            __syncthreads();
        }
        if (regs) {
            for (int base = 64 * wid; base < n_pow2; base += 64 * nwarps) warp_sort64(s, base, size, size);
            __syncthreads();
        }
    }
}
__device__ __forceinline__ int pow2_ge(int n) {
    int p = 1;
    while (p < n) p <<= 1;
    return p;
}
constexpr uint64_t kKeyMask = (1ULL << 50) - 1;

__device__ void load_sorted(uint64_t *s, const uint64_t *keys, const int32_t *votes, int n, int np2) {
    for (int i = threadIdx.x; i < np2; i += blockDim.x)
        s[i] = i < n ? (((uint64_t)(1023 - votes[i]) << 50) | (keys[i] & kKeyMask)) : ~0ULL;
    __syncthreads();
    block_sort(s, np2);
}

// One event's top-K by one block: s = shared scratch of pow2_ge(n_in) entries.
__device__ __forceinline__ void topk_block(const uint64_t *keys_e, const int32_t *votes_e, int n_in, int K,
                                           uint64_t *out_keys_e, int32_t *out_votes_e, uint64_t *s) {
    int np2 = pow2_ge(n_in);
    load_sorted(s, keys_e, votes_e, n_in, np2);
    for (int i = threadIdx.x; i < K; i += blockDim.x) {
        uint64_t x = i < n_in ? s[i] : ~0ULL;
        out_keys_e[i] = x & kKeyMask;
        out_votes_e[i] = i < n_in ? 1023 - (int)(x >> 50) : 0;
    }
    __syncthreads();
}

__global__ void __launch_bounds__(1024)
k_topk(const uint64_t *keys, const int32_t *votes, int n_in, int K, uint64_t *out_keys,
       int32_t *out_votes, const int32_t *skip) {
    __shared__ uint64_t s[kSortMax];
    const int e = blockIdx.x;
    if (skip && skip[e]) return;
    topk_block(keys + (long long)e * n_in, votes + (long long)e * n_in, n_in, K, out_keys + (long long)e * K,
               out_votes + (long long)e * K, s);
}

void launch_topk(int n_ev, const uint64_t *keys, const int32_t *votes, int n_in, int K,
                 uint64_t *out_keys, int32_t *out_votes, cudaStream_t s, const int32_t *skip) {
    if (n_ev <= 0) return;
    k_topk<<<n_ev, 1024, 0, s>>>(keys, votes, n_in, K, out_keys, out_votes, skip);
}

// ---------------------------------------------------------------------------------------
// Final estimate (Section 3.3) and, for multi-track extraction, hit masking.  Per event
// (one block) in round `round`: stop (done) if no hit is active or the best final vote
// count is below min_votes; otherwise write track `round`: over the maximum-vote cells in
// ascending key order, the mean of the cell centres and the half-extent of their union per
// axis, in round-to-nearest.  Then deactivate every active hit that votes (FP64) for at
// least one maximum-vote cell with its drift widened to [max(rd(d - width), 0),
// ru(d + width)] (the paper's hit finding with a widened box, Section 3.3).
// ---------------------------------------------------------------------------------------
constexpr int kEstChunk = 256;

// One event's estimate and hit masking by one block (any multiple of 32 threads, at least
// 64): keys_e / votes_e the last level's cells, active_e its 8 mask words, done_e its flag,
// hd_e its staged hits, te its max_tracks records, n_tracks_e its count, a0 its first hit
// in the batch (for hit_track).  s: shared scratch of kSortMax entries; s_cen: of
// kEstChunk x 5.
__device__ __forceinline__ void estimate_mask_block(const DevGeom &g, const uint64_t *keys_e, const int32_t *votes_e,
                                                    int n_in, int level, int nh, uint32_t *active_e,
                                                    int32_t *done_e, const HitRecD *hd_e, int round,
                                                    int max_tracks, int min_votes, double width,
                                                    apo_track *te, int32_t *n_tracks_e, int a0,
                                                    int32_t *hit_track, uint64_t *s, double *s_cen) {
    __shared__ long long s_lo[5], s_hi[5];
    __shared__ uint32_t act0[8], act1[8];
    __shared__ int s_m;
    const int tid = threadIdx.x;
    if (*done_e) return;
    if (round == 0) {
        if (tid < max_tracks) {
            for (int a = 0; a < 5; a++) { te[tid].p[a] = 0.0; te[tid].w[a] = 0.0; }
            te[tid].votes = (tid == 0 && nh < 0) ? nh : 0;
            te[tid].n_hits = nh < 0 ? 0 : nh;
        }
        if (tid == 0) *n_tracks_e = 0;
    }
    if (nh < 0) {
        __syncthreads();
        if (tid == 0) *done_e = 1;
        __syncthreads();
        return;
    }
    if (tid < 8) act0[tid] = act1[tid] = active_e[tid];
    __syncthreads();
    int na = 0;
    for (int i = 0; i < 8; i++) na += __popc(act0[i]);
    if (na == 0) {
        __syncthreads();
        if (tid == 0) *done_e = 1;
        __syncthreads();
        return;
    }
    if (tid == 0) s_m = 0;
    if (tid < 5) { s_lo[tid] = okey(1e300); s_hi[tid] = okey(-1e300); }
    int np2 = pow2_ge(n_in);
    load_sorted(s, keys_e, votes_e, n_in, np2);
    // the maximum-vote cells are s[0, m) after the sort
    const uint64_t top = s[0] >> 50;
    const int vmax = 1023 - (int)top;
    {
        int cnt = 0;
        for (int i = tid; i < n_in; i += blockDim.x) cnt += (s[i] >> 50) == top;
        if (cnt) atomicAdd(&s_m, cnt);
    }
    __syncthreads();
    const int m = s_m;
    if (vmax < min_votes) {
        if (tid == 0) *done_e = 1;
        __syncthreads();
        return;
    }
    // Centres of the m cells, staged per chunk by all threads; thread a < 5 then adds axis
    // a's centres in key order (the same round-to-nearest sequence as a serial loop).  The
    // union's ends are order-free: min / max through atomics on value-ordered keys.
    double sum = 0.0;
    for (int c0 = 0; c0 < m; c0 += kEstChunk) {
        const int cn = m - c0 < kEstChunk ? m - c0 : kEstChunk;
        for (int q = tid; q < cn * 5; q += blockDim.x) {
            const int j = q / 5, a = q - 5 * j;
            int idx[5];
            unpack_key(g, s[c0 + j] & kKeyMask, idx);
            IV<double> ed = edge(g, a, level, idx[a]);
            s_cen[q] = __dmul_rn(__dadd_rn(ed.lo, ed.hi), 0.5);
            atomicMin(&s_lo[a], okey(ed.lo));
            atomicMax(&s_hi[a], okey(ed.hi));
        }
        __syncthreads();
        if (tid < 5)
            for (int j = 0; j < cn; j++) sum = __dadd_rn(sum, s_cen[5 * j + tid]);
        __syncthreads();
    }
    if (tid < 5) {
        apo_track &t = te[round];
        const double lo_min = __longlong_as_double(okey_inv(s_lo[tid]));
        const double hi_max = __longlong_as_double(okey_inv(s_hi[tid]));
        t.p[tid] = __ddiv_rn(sum, (double)m);
        t.w[tid] = __dmul_rn(__dsub_rn(hi_max, lo_min), 0.5);
        if (tid == 0) {
            t.votes = vmax;
            t.n_hits = nh;
            *n_tracks_e = round + 1;
        }
    }
    const bool last = round + 1 >= max_tracks;
    if (last && !hit_track) {   // no later round needs the masks
        if (tid == 0) *done_e = 1;
        __syncthreads();
        return;
    }
    const long long pairs = (long long)m * nh;
    for (long long q = tid; q < pairs; q += blockDim.x) {
        const int j = (int)(q / nh), i = (int)(q % nh);
        if (!((act0[i >> 5] >> (i & 31)) & 1u)) continue;
        if (!((act1[i >> 5] >> (i & 31)) & 1u)) continue;   // already masked by another cell
        int idx[5];
        unpack_key(g, s[j] & kKeyMask, idx);
        Cell<double> c{edge(g, 0, level, idx[0]), sin_phi0(g, level, idx[1]), cos_phi0(g, level, idx[1]),
                       edge(g, 2, level, idx[2]), edge(g, 3, level, idx[3]), edge(g, 4, level, idx[4])};
        if (vote_widened(g, c, hd_e + i, width)) atomicAnd(&act1[i >> 5], ~(1u << (i & 31)));
    }
    __syncthreads();
    if (tid < 8) active_e[tid] = act1[tid];
    if (hit_track) {   // the hits this track took: active before, masked now
        for (int i = tid; i < nh; i += blockDim.x)
            if (((act0[i >> 5] & ~act1[i >> 5]) >> (i & 31)) & 1u) hit_track[a0 + i] = round;
    }
    if (tid == 0) {
        int left = 0;
        for (int i = 0; i < 8; i++) left += __popc(act1[i]);
        if (left == 0 || last) *done_e = 1;
    }
    __syncthreads();
}

__global__ void __launch_bounds__(256)
k_estimate_mask(const __grid_constant__ DevGeom g, const uint64_t *keys, const int32_t *votes, int n_in, int level,
                const int32_t *n_hits, uint32_t *active, int32_t *done, const HitRecD *hd,
                int round, int max_tracks, int min_votes, double width, apo_track *out,
                int32_t *n_tracks, const int32_t *offsets, int32_t *hit_track) {
    __shared__ uint64_t s[kSortMax];
    __shared__ double s_cen[kEstChunk * 5];
    const int e = blockIdx.x;
    estimate_mask_block(g, keys + (long long)e * n_in, votes + (long long)e * n_in, n_in, level, n_hits[e],
                        active + (long long)e * 8, done + e, hd + (long long)e * kHitCap, round, max_tracks,
                        min_votes, width, out + (long long)e * max_tracks, n_tracks + e,
                        hit_track ? offsets[e] : 0, hit_track, s, s_cen);
}

void launch_estimate_mask(const DevGeom &g, int n_ev, const uint64_t *keys, const int32_t *votes,
                          int n_in, int level, const int32_t *n_hits, uint32_t *active, int32_t *done,
                          const HitRecD *hd, int round, int max_tracks, int min_votes, double width,
                          apo_track *out, int32_t *n_tracks, cudaStream_t s, const int32_t *offsets,
                          int32_t *hit_track) {
    if (n_ev <= 0) return;
    k_estimate_mask<<<n_ev, 256, 0, s>>>(g, keys, votes, n_in, level, n_hits, active, done, hd, round,
                                          max_tracks, min_votes, width, out, n_tracks, offsets,
                                          hit_track);
}

}  // namespace apo

namespace apo {

// ---------------------------------------------------------------------------------------
// Histogram of level-0 votes (for apo_refine on caller-provided coarse votes).
// ---------------------------------------------------------------------------------------
__global__ void k_hist(const int32_t *votes, long long n, uint32_t *hist) {
    __shared__ uint32_t hs[kHistBins];
    const int e = blockIdx.y;
    for (int i = threadIdx.x; i < kHistBins; i += blockDim.x) hs[i] = 0;
    __syncthreads();
    const int32_t *v = votes + (long long)e * n;
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < n;
         j += (long long)gridDim.x * blockDim.x) {
        int x = v[j];
        x = x < 0 ? 0 : (x > kHitCap ? kHitCap : x);
        atomicAdd(&hs[x], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kHistBins; i += blockDim.x)
        if (hs[i]) atomicAdd(&hist[(long long)e * kHistBins + i], hs[i]);
}

void launch_hist(int n_ev, const int32_t *votes, long long n, uint32_t *hist, cudaStream_t s) {
    if (n_ev <= 0) return;
    dim3 grid(64, n_ev);
    k_hist<<<grid, 256, 0, s>>>(votes, n, hist);
}

// 32 children of each key (level + 1)
__global__ void k_children(DevGeom g, const uint64_t *keys, long long n, uint64_t *out) {
    long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n * 32) return;
    int idx[5], b = (int)(j % 32);
    unpack_key(g, keys[j / 32], idx);
#pragma unroll
    for (int a = 0; a < 5; a++) idx[a] = 2 * idx[a] + ((b >> a) & 1);
    out[j] = pack_key(g, idx);
}

void launch_children(const DevGeom &g, const uint64_t *keys, long long n, uint64_t *out, cudaStream_t s) {
    if (n <= 0) return;
    k_children<<<(unsigned)((n * 32 + 255) / 256), 256, 0, s>>>(g, keys, n, out);
}

}  // namespace apo

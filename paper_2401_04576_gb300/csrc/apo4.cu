// The paper's own 4-D search on the GPU (include/apo4.h; arXiv:2401.04576 Sections 3.1-3.3,
// Tables tabGridDef and HelixParametes): voxel voting in the midpoint form behind the disk
// pre-filter, the per-event maximum-vote statistics, the estimate, hit finding and the
// reference-point update, all queued on the caller's stream without host round trips.
#include <cuda_runtime.h>

#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <vector>

#include "../../include/apo4.h"
#include "cert4.cuh"
#include "fourd.cuh"
#include "kernels.cuh"

using namespace apo;

struct apo4_chamber {
    DevGeom dg;      // only the wire table and n_wires are set (for the hit staging)
    int device;
    std::vector<void *> allocs;
};

namespace {

int fail4(int code, const char *fmt, ...) {
    char msg[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(msg, sizeof(msg), fmt, ap);
    va_end(ap);
    set_last_error(msg);
    return code;
}

#define CU4(call)                                                                       \
    do {                                                                                \
        cudaError_t e_ = (call);                                                        \
        if (e_ != cudaSuccess)                                                          \
            return fail4(APO_ECUDA, "%s: %s (%s:%d)", #call, cudaGetErrorString(e_), __FILE__, \
                         __LINE__);                                                     \
    } while (0)

size_t al256(size_t x) { return (x + 255) & ~size_t(255); }

// One iteration's grid shape and the constants of the search, by value to the kernels.
struct Iter4 {
    double w[4];
    int n[4];
    long long ncol, nvox;
    double p_gev, b_tesla, disk_radius, hit_factor;
};

// Maximum-vote statistics of one event: count, index sums, index extent per axis.
struct Stats4 {
    unsigned long long cnt, sum[4];
    int mn[4], mx[4];
};

struct Layout4 {
    size_t status, nh, hd, hf, active, done, lo, ref, vmax, stats, lo2, ref2, active2, stats2, votes, end;
    int chunk;
    long long max_nvox;
};

Layout4 layout4(const apo4_opts *o, int ne) {
    Layout4 L{};
    long long mv = 1;
    for (int k = 0; k < 3; k++) {
        long long v = 1;
        for (int a = 0; a < 4; a++) v *= o->n[k][a];
        if (k < o->n_iter && v > mv) mv = v;
    }
    L.max_nvox = mv;
    long long c = (1LL << 30) / (8 * mv);
    L.chunk = (int)(c < 1 ? 1 : (c > ne ? (ne > 0 ? ne : 1) : c));
    size_t n = (size_t)(ne > 0 ? ne : 1);
    size_t off = 0;
    L.status = off; off += 256;
    L.nh = off; off += al256(sizeof(int32_t) * n);
    L.hd = off; off += al256(sizeof(HitRecD) * n * kHitCap);
    L.hf = off; off += al256(sizeof(HitRecF) * n * kHitCap);
    L.active = off; off += al256(sizeof(uint32_t) * n * 8);
    L.done = off; off += al256(sizeof(int32_t) * n);
    L.lo = off; off += al256(sizeof(double) * n * 4);
    L.ref = off; off += al256(sizeof(double) * n * 2);
    L.vmax = off; off += al256(sizeof(int32_t) * n * 2);
    L.stats = off; off += al256(sizeof(Stats4) * n);
    // per-sign state of iteration 3 (sign-major: sign s of event e at s n + e)
    L.lo2 = off; off += al256(sizeof(double) * 2 * n * 4);
    L.ref2 = off; off += al256(sizeof(double) * 2 * n * 2);
    L.active2 = off; off += al256(sizeof(uint32_t) * 2 * n * 8);
    L.stats2 = off; off += al256(sizeof(Stats4) * 2 * n);
    L.votes = off; off += al256(sizeof(int32_t) * 2 * (size_t)mv * (size_t)L.chunk);
    L.end = off;
    return L;
}

int check_opts(const apo4_opts *o) {
    if (!o) return fail4(APO_EINVAL, "opts is NULL");
    if (o->n_iter < 1 || o->n_iter > 3) return fail4(APO_EINVAL, "n_iter must be 1..3");
    if (o->precision != APO_F64 && o->precision != APO_F32)
        return fail4(APO_EINVAL, "precision must be APO_F64 or APO_F32");
    if (o->per_sign != 0 && o->per_sign != 1) return fail4(APO_EINVAL, "per_sign must be 0 or 1");
    if (!(o->p_gev > 0) || !(o->b_tesla > 0) || !(o->disk_radius >= 0) || !(o->hit_factor >= 0))
        return fail4(APO_EINVAL, "p_gev, b_tesla > 0 and disk_radius, hit_factor >= 0 required");
    for (int k = 0; k < o->n_iter; k++) {
        long long v = 1;
        for (int a = 0; a < 4; a++) {
            if (o->n[k][a] < 1 || o->n[k][a] > 4096) return fail4(APO_EINVAL, "n[%d][%d] out of range", k, a);
            if (!(o->w[k][a] > 0)) return fail4(APO_EINVAL, "w[%d][%d] must be > 0", k, a);
            v *= o->n[k][a];
        }
        if (o->n[k][3] > 32) return fail4(APO_EINVAL, "n[%d][3] (z0 voxels) must be <= 32", k);
        if (v > (1LL << 28)) return fail4(APO_EINVAL, "iteration %d has more than 2^28 voxels", k);
    }
    return APO_OK;
}

Iter4 iter4(const apo4_opts *o, int k) {
    Iter4 it{};
    for (int a = 0; a < 4; a++) { it.w[a] = o->w[k][a]; it.n[a] = o->n[k][a]; }
    it.ncol = (long long)it.n[0] * it.n[1] * it.n[2];
    it.nvox = it.ncol * it.n[3];
    it.p_gev = o->p_gev;
    it.b_tesla = o->b_tesla;
    it.disk_radius = o->disk_radius;
    it.hit_factor = o->hit_factor;
    return it;
}

}  // namespace

namespace apo {

// ---- precision helpers: FP64 end points as intervals / points of T ----
template <typename T> __device__ __forceinline__ IV<T> box_iv(double lo, double hi);
template <> __device__ __forceinline__ IV<double> box_iv<double>(double lo, double hi) { return {lo, hi}; }
template <> __device__ __forceinline__ IV<float> box_iv<float>(double lo, double hi) {
    return {__double2float_rd(lo), __double2float_ru(hi)};
}
template <typename T> __device__ __forceinline__ T rn(double x);
template <> __device__ __forceinline__ double rn<double>(double x) { return x; }
template <> __device__ __forceinline__ float rn<float>(double x) { return __double2float_rn(x); }
template <typename T> __device__ __forceinline__ T up(double x);   // rd of the disk radius
template <> __device__ __forceinline__ double up<double>(double x) { return x; }
template <> __device__ __forceinline__ float up<float>(double x) { return __double2float_ru(x); }

template <typename T> __device__ __forceinline__ HitP<T> hit_point(const HitRecD &r) {
    return {rn<T>(r.v[0]), rn<T>(r.v[1]), rn<T>(r.v[2]), rn<T>(r.v[3]), rn<T>(r.v[4]), rn<T>(r.v[5]),
            rn<T>(r.v[6]), rn<T>(r.v[7]), rn<T>(r.v[8])};
}
template <typename T> __device__ __forceinline__ HitI<T> hit_iv(const HitRecD &r) {
    return {box_iv<T>(r.v[0], r.v[0]), box_iv<T>(r.v[1], r.v[1]), box_iv<T>(r.v[5], r.v[5]),
            box_iv<T>(r.v[6], r.v[6])};
}

// voxel edge lo + i w (round to nearest)
__device__ __forceinline__ double edge4(double lo, int i, double w) { return __dadd_rn(lo, __dmul_rn((double)i, w)); }
__device__ __forceinline__ double mid4(double a, double b) { return __dmul_rn(__dadd_rn(a, b), 0.5); }

// ---------------------------------------------------------------------------------------
// Voting.  Block: a tile of 8 x 8 x depth voxel columns (x_c, y_c, R) of one event (depth 8, so that
// the columns that pass fill whole warps, or 4 or 2 where there would be too few blocks).  First it
// tests every column of its tile against the disk pre-filter (Eq. ApoVoteDisk) and the centre's
// validity and writes zero votes for the columns that fail.  Then its threads take the groups of
// 2 x 2 x 2 columns with a passing one, 16 groups at a time, a column each: every active hit
// over the column's z0 voxels and both signs of tan(lambda), with vote counters bit-sliced over
// the z0 voxels; a warp (four groups) works by itself.
//
// The votes (of the program in T) are decided by certified FP32 values (cert4.cuh).  Per (group,
// hit) one evaluation with errors over the group's columns and z0 voxels gives the bound that all
// its pairs share, in chunks of 16 hits, one evaluation per thread (over each half of the z0 voxels
// where the whole range decides nothing, then per column); pairs left undecided are queued by warp
// and evaluated by the program itself.  FP32 issue bounds it; evaluating every pair was bound by the
// FP64 pipe, and in FP32 by the instructions of correctly rounded quotients and roots: FP32, 48
// electrons, 380 -> 225 ms; FP64, 2 electrons, 788 -> 13.6 ms.  Blocks of one warp took the latter
// to 21.3 ms.  Always eight columns deep: two events' search 22.8 against 16.0 ms.
// ---------------------------------------------------------------------------------------
constexpr int k4Threads = 128, k4Side = 8, k4MaxTile = k4Side * k4Side * k4Side, k4Groups = k4MaxTile / 8;
constexpr int k4Slots = k4Threads / 8, k4Chunk = 16;

template <typename T> struct Col4 {
    IV<T> X, Y, Rv;
    Ctr4<T> m;
};

template <typename T>
__device__ __forceinline__ Col4<T> column4(const Iter4 &it, const double *le, const double *rf, int ix, int iy, int iR) {
    const double xl = edge4(le[0], ix, it.w[0]), xh = edge4(le[0], ix + 1, it.w[0]);
    const double yl = edge4(le[1], iy, it.w[1]), yh = edge4(le[1], iy + 1, it.w[1]);
    const double rl = edge4(le[2], iR, it.w[2]), rh = edge4(le[2], iR + 1, it.w[2]);
    Col4<T> c;
    c.X = box_iv<T>(xl, xh);
    c.Y = box_iv<T>(yl, yh);
    c.Rv = box_iv<T>(rl, rh);
    c.m = centre4<T>(rn<T>(mid4(xl, xh)), rn<T>(mid4(yl, yh)), rn<T>(mid4(rl, rh)),
                     rn<T>(it.p_gev), rn<T>(it.b_tesla), rn<T>(rf[0]), rn<T>(rf[1]));
    return c;
}

template <int K> __device__ __forceinline__ cert::X<K> wide(float v) {   // a value rounded to v
    return cert::point(cert::sc<K>(v));
}
template <int K> __device__ __forceinline__ cert::X<K> wide(float lo, float hi) {
    cert::X<K> r;
    r.lo = lo;
    r.hi = hi;
    r.e = 2.f * cert::rnd<K>(cert::mag2(lo, hi)) + cert::kTiny;
    return r;
}
template <int K> __device__ __forceinline__ cert::X<K> wide(cert::X<0> x) { return wide<K>(x.lo, x.hi); }

// The ranges of some columns' constants (in Col4X's order) and intervals, from their FP32 values.
struct Group4 { float2 m[8], box[3]; };

// bound4 over a group's columns; out of the callers' registers
template <int K>
__device__ __noinline__ cert::Bound4 group_bound(const Group4 *gp, float zc0, float zc1, float z0, float z1,
                                                 const cert::Hit4X<cert::Pt> *hp) {
    cert::Col4X<cert::X<K>> M;
    cert::Hit4X<cert::X<K>> H;
    const cert::Pt *hs = &hp->x0;
    cert::X<K> *dst = &M.xc, *hd = &H.x0;
#pragma unroll
    for (int i = 0; i < 8; i++) dst[i] = wide<K>(gp->m[i].x, gp->m[i].y);
#pragma unroll
    for (int i = 0; i < 9; i++) hd[i] = wide<K>(hs[i].v);
    M.ion.e *= 2.f;   // an approximate reciprocal
    return cert::bound4<K>(M, cert::Box4X<K>{wide<K>(gp->box[0].x, gp->box[0].y), wide<K>(gp->box[1].x, gp->box[1].y),
                                             wide<K>(gp->box[2].x, gp->box[2].y)},
                           wide<K>(zc0, zc1), wide<K>(z0, z1), H);
}

// A column of the tile at (x0, y0, R0): k = 8 group + sub, both with x fastest.
__device__ __forceinline__ void tile_column(int k, int x0, int y0, int r0, int &ix, int &iy, int &iR) {
    const int gr = k >> 3, sub = k & 7;
    ix = x0 + 2 * (gr & 3) + (sub & 1);
    iy = y0 + 2 * ((gr >> 2) & 3) + ((sub >> 1) & 1);
    iR = r0 + 2 * (gr >> 4) + (sub >> 2);
}

// The program's votes of one (column, hit) for the z0 voxels b0 (tan(lambda) > 0) and b1 (< 0).
template <typename T>
__device__ __noinline__ uint2 resolve4(const Iter4 &it, const double *le, const double *rf, int ix, int iy, int iR,
                                       const HitRecD *rec, uint32_t b0, uint32_t b1) {
    const Col4<T> c = column4<T>(it, le, rf, ix, iy, iR);
    const HitP<T> h = hit_point<T>(*rec);
    const HitI<T> w = hit_iv<T>(*rec);
    uint2 yes = make_uint2(0u, 0u);
    uint32_t m = b0 | b1;
    while (m) {
        const int iz = __ffs(m) - 1;
        const uint32_t bit = 1u << iz;
        m &= m - 1;
        const double zl = edge4(le[3], iz, it.w[3]), zh = edge4(le[3], iz + 1, it.w[3]);
        const Pre4<T> pre = prefix4<T>(c.m, rn<T>(mid4(zl, zh)), h);
        if (pre.guard) {
            yes.x |= b0 & bit;
            yes.y |= b1 & bit;
            continue;
        }
        const IV<T> A2 = a2_4<T>(c.X, c.Y, box_iv<T>(zl, zh), w);
#pragma unroll 1
        for (int s = 0; s < 2; s++) {
            if (!((s ? b1 : b0) & bit)) continue;
            if (pair4<T>(c.m, pre, s ? -1 : 1, h, A2, c.Rv)) { if (s) yes.y |= bit; else yes.x |= bit; }
        }
    }
    return yes;
}

struct Queue4 { uint32_t id[64], b0[64], b1[64]; };   // lane | hit << 8; voxels of either sign of tan(lambda)

template <typename T>
__global__ void __launch_bounds__(k4Threads, 4)
k4_vote(const __grid_constant__ Iter4 it, int ev0, const int32_t *n_hits, const HitRecD *hd,
        const uint32_t *active, const double *lo, const double *ref, int32_t *votes, int32_t *vmax, int sign_only, int depth) {
    constexpr int K = sizeof(T) == 8 ? 64 : 32;
    __shared__ cert::Hit4X<cert::Pt> s_h[kHitCap];
    __shared__ unsigned char s_i[kHitCap], s_grp[k4Groups];
    __shared__ float s_zc[32];
    __shared__ float2 s_z[32];
    __shared__ uint32_t s_pass[k4MaxTile / 32];
    __shared__ Group4 s_g[k4Slots];
    __shared__ float s_e0[k4Slots][k4Chunk], s_e1[k4Slots][k4Chunk], s_eps[k4Slots][k4Chunk];
    __shared__ Queue4 s_q[k4Threads / 32];
    __shared__ int s_n, s_ng, s_vmax[2];
    const int el = blockIdx.y, e = ev0 + el, tid = threadIdx.x, lane = tid & 31;
    Queue4 &q = s_q[tid >> 5];
    int nh = n_hits[e];
    if (nh < 0) nh = 0;
    if (tid == 0) { s_n = 0; s_vmax[0] = s_vmax[1] = 0; }
    __syncthreads();
    const uint32_t *act = active + (long long)e * 8;
    const HitRecD *hde = hd + (long long)e * kHitCap;
    for (int i = tid; i < nh; i += k4Threads) {
        if (!((act[i >> 5] >> (i & 31)) & 1u)) continue;
        const int j = atomicAdd(&s_n, 1);
        cert::Pt *f = &s_h[j].x0;
#pragma unroll
        for (int k = 0; k < 9; k++) f[k].v = (float)hde[i].v[k];
        s_i[j] = (unsigned char)i;
    }
    const double *le = lo + (long long)e * 4;
    for (int iz = tid; iz < it.n[3]; iz += k4Threads) {
        const double zl = edge4(le[3], iz, it.w[3]), zh = edge4(le[3], iz + 1, it.w[3]);
        s_zc[iz] = (float)mid4(zl, zh);
        s_z[iz] = make_float2((float)zl, (float)zh);
    }
    const double *rf = ref + (long long)e * 2;
    const int nz = it.n[3];
    int32_t *vo = votes + (long long)el * 2 * it.nvox;
    const int tx = (it.n[0] + k4Side - 1) / k4Side, ty = (it.n[1] + k4Side - 1) / k4Side;
    const int x0 = k4Side * (blockIdx.x % tx), y0 = k4Side * (blockIdx.x / tx % ty), r0 = depth * (blockIdx.x / tx / ty);
    const int ntile = k4Side * k4Side * depth;
    // disk pre-filter of the tile; failing columns get zero votes
    for (int k = tid; k < ntile; k += k4Threads) {
        int ix, iy, iR;
        tile_column(k, x0, y0, r0, ix, iy, iR);
        const bool in = ix < it.n[0] && iy < it.n[1] && iR < it.n[2];
        bool pass = false;
        if (in) {
            const Col4<T> c = column4<T>(it, le, rf, ix, iy, iR);
            pass = disk4<T>(c.X, c.Y, c.Rv, up<T>(it.disk_radius)) && c.m.valid;
            const long long col = ix + (long long)it.n[0] * (iy + (long long)it.n[1] * iR);
            if (!pass)
                for (int s = 0; s < 2; s++)
                    if (sign_only < 0 || s == sign_only)
                        for (int iz = 0; iz < nz; iz++) vo[(long long)s * it.nvox + col + it.ncol * iz] = 0;
        }
        const unsigned m = __ballot_sync(0xffffffffu, pass);
        if (lane == 0) s_pass[k >> 5] = m;
    }
    __syncthreads();
    if (tid < 32) {   // the groups with a passing column, in order
        int n = 0;
        for (int g0 = 0; g0 < ntile / 8; g0 += 32) {
            const int gr = g0 + lane;
            const bool any = gr < ntile / 8 && ((s_pass[gr >> 2] >> (8 * (gr & 3))) & 255u) != 0u;
            const unsigned m = __ballot_sync(0xffffffffu, any);
            if (any) s_grp[n + __popc(m & ((1u << lane) - 1u))] = (unsigned char)gr;
            n += __popc(m);
        }
        if (lane == 0) s_ng = n;
    }
    __syncthreads();
    const int na = s_n, ng = s_ng, slot = tid >> 3, half = (nz + 1) >> 1;
    const uint32_t allz = nz >= 32 ? 0xffffffffu : ((1u << nz) - 1u);
    const uint32_t all0 = sign_only == 1 ? 0u : allz, all1 = sign_only == 0 ? 0u : allz;
    int mx[2] = {0, 0};
    for (int g0 = 0; g0 < ng; g0 += k4Slots) {
        const int ns = ng - g0 < k4Slots ? ng - g0 : k4Slots;
        const int k = slot < ns ? 8 * s_grp[g0 + slot] + (tid & 7) : 0;
        const bool has = slot < ns && ((s_pass[k >> 5] >> (k & 31)) & 1u);
        int ix, iy, iR;
        tile_column(k, x0, y0, r0, ix, iy, iR);
        const Col4<T> cd = column4<T>(it, le, rf, ix, iy, iR);
        const T cR = cd.m.R;
        const cert::Col4X<cert::Pt> m{{(float)cd.m.xc}, {(float)cd.m.yc}, {(float)cR}, {(float)cd.m.aL}, {(float)cd.m.ox},
                                      {(float)cd.m.oy}, {cert::rcp_a((float)cd.m.on)}, {(float)cd.m.psi_ref}};
        const cert::Box4X<0> b{cert::mk<0>(cd.X.lo, cd.X.hi), cert::mk<0>(cd.Y.lo, cd.Y.hi),
                               cert::mk<0>((double)cd.Rv.lo - (double)cR, (double)cd.Rv.hi - (double)cR)};
        const bool guard = cd.m.guard;
        {   // the group's ranges over its passing columns (the eight lanes of a slot)
            const cert::Pt *src = &m.xc;
            auto hull8 = [&](float l, float h) {
                if (!has) { l = INFINITY; h = -INFINITY; }
#pragma unroll
                for (int o = 1; o < 8; o <<= 1) {
                    l = fminf(l, __shfl_xor_sync(0xffffffffu, l, o));
                    h = fmaxf(h, __shfl_xor_sync(0xffffffffu, h, o));
                }
                return make_float2(l, h);
            };
            __syncwarp();   // the last groups' bounds have been read
#pragma unroll
            for (int i = 0; i < 8; i++) {
                const float2 r = hull8(src[i].v, src[i].v);
                if ((tid & 7) == 0) s_g[slot].m[i] = r;
            }
            const float2 bx = hull8(b.X_.lo, b.X_.hi), by = hull8(b.Y_.lo, b.Y_.hi), br = hull8(b.dR.lo, b.dR.hi);
            if ((tid & 7) == 0) { s_g[slot].box[0] = bx; s_g[slot].box[1] = by; s_g[slot].box[2] = br; }
        }
        uint32_t pl[2][9];
#pragma unroll
        for (int s = 0; s < 2; s++)
#pragma unroll
            for (int i = 0; i < 9; i++) pl[s][i] = 0u;
        auto add_votes = [&](int s, uint32_t v) {
#pragma unroll
            for (int i = 0; i < 9; i++) {
                const uint32_t cy = pl[s][i] & v;
                pl[s][i] ^= v;
                v = cy;
            }
        };
        int nq = 0;
        for (int j0 = 0; j0 < na; j0 += k4Chunk) {
            const int nc = na - j0 < k4Chunk ? na - j0 : k4Chunk;
            __syncwarp();
            for (int i = lane; i < 4 * nc; i += 32) {   // the warp's own four groups
                const int sl = (tid >> 5) * 4 + i / nc, j = i % nc;
                if (sl >= ns) continue;
                cert::Bound4 f0 = group_bound<K>(s_g + sl, s_zc[0], s_zc[nz - 1], s_z[0].x, s_z[nz - 1].y, s_h + j0 + j), f1 = f0;
                if (!(f0.e < 1e30f) && nz > 1) {
                    f0 = group_bound<K>(s_g + sl, s_zc[0], s_zc[half - 1], s_z[0].x, s_z[half - 1].y, s_h + j0 + j);
                    f1 = group_bound<K>(s_g + sl, s_zc[half], s_zc[nz - 1], s_z[half].x, s_z[nz - 1].y, s_h + j0 + j);
                }
                s_e0[sl][j] = f0.e;
                s_e1[sl][j] = f1.e;
                s_eps[sl][j] = fmaxf(f0.eps, f1.eps);
            }
            __syncwarp();
            for (int j = 0; j < nc; j++) {
                uint32_t b0 = 0, b1 = 0, u0 = 0, u1 = 0;
                if (has && guard) {
                    b0 = all0;
                    b1 = all1;
                } else if (has) {
                    const cert::Hit4X<cert::Pt> h = s_h[j0 + j];
                    float e0 = s_e0[slot][j], e1 = s_e1[slot][j], eps = s_eps[slot][j];
                    if (!(e0 < 1e30f) || !(e1 < 1e30f)) {   // the column's own bounds
                        Group4 own;
                        const cert::Pt *src = &m.xc;
#pragma unroll
                        for (int i = 0; i < 8; i++) own.m[i] = make_float2(src[i].v, src[i].v);
                        own.box[0] = make_float2(b.X_.lo, b.X_.hi);
                        own.box[1] = make_float2(b.Y_.lo, b.Y_.hi);
                        own.box[2] = make_float2(b.dR.lo, b.dR.hi);
                        const cert::Bound4 f0 = group_bound<K>(&own, s_zc[0], s_zc[half - 1], s_z[0].x, s_z[half - 1].y, s_h + j0 + j);
                        cert::Bound4 f1 = f0;
                        if (nz > 1)
                            f1 = group_bound<K>(&own, s_zc[half], s_zc[nz - 1], s_z[half].x, s_z[nz - 1].y, s_h + j0 + j);
                        e0 = f0.e;
                        e1 = f1.e;
                        eps = fmaxf(f0.eps, f1.eps);
                    }
#pragma unroll 1
                    for (int iz = 0; iz < nz; iz++) {
                        const uint32_t bit = 1u << iz;
                        const float e = iz < half ? e0 : e1;
                        bool bad = true;
                        cert::Pt dx, dy;
                        cert::wire4x(m, cert::Pt{s_zc[iz]}, h, dx, dy);
                        cert::Pre4X<cert::Pt> pre = cert::prefix4x(dx, dy, h);
                        pre.psi = cert::psi4(m, dx, dy, pre.iRA, eps, bad);
                        pre.Rpsi = cert::mul(m.R, pre.psi);
                        if (bad || !(e < 1e30f)) {
                            u0 |= all0 & bit;
                            u1 |= all1 & bit;
                            continue;
                        }
                        const float2 z = s_z[iz];
                        const cert::X<0> A2 = cert::a2_4x<0, cert::Pt>(b, cert::X<0>{z.x, z.y, 0.f}, h);
                        const cert::Delta4<cert::Pt> d0 = cert::delta4x(pre, m.R, m.aL, h.d, h),
                                                     d1 = cert::delta4x(pre, m.R, m.aL, cert::neg(h.d), h);
#pragma unroll 1
                        for (int s = 0; s < 2; s++) {
                            if (sign_only == 1 - s) continue;
                            const float f = s ? 1.f : -1.f;
                            const cert::Pt dl[2] = {{fmaf(f, d0.v.v, d0.u.v)}, {fmaf(f, d1.v.v, d1.u.v)}};
                            const int v = cert::vote4x(pre, m, cert::Pt{-f * m.aL.v}, h, A2, b.dR, e, dl);
                            const uint32_t y = v == cert::kYes ? bit : 0u, u = v == cert::kUnknown ? bit : 0u;
                            if (s) { b1 |= y; u1 |= u; } else { b0 |= y; u0 |= u; }
                        }
                    }
                }
                add_votes(0, b0);
                add_votes(1, b1);
                const unsigned um = __ballot_sync(0xffffffffu, (u0 | u1) != 0u);
                if (u0 | u1) {
                    const int i = nq + __popc(um & ((1u << lane) - 1u));   // below 64: drained from 32 on
                    q.id[i] = (uint32_t)lane | ((uint32_t)(j0 + j) << 8);
                    q.b0[i] = u0;
                    q.b1[i] = u1;
                }
                nq += __popc(um);
                if (nq >= 32 || (nq && j0 + j + 1 == na)) {
                    __syncwarp();
                    for (int i = lane; i < nq; i += 32) {
                        const int ot = (tid & ~31) + (int)(q.id[i] & 255u);
                        int ox, oy, oR;
                        tile_column(8 * s_grp[g0 + (ot >> 3)] + (ot & 7), x0, y0, r0, ox, oy, oR);
                        const uint2 y = resolve4<T>(it, le, rf, ox, oy, oR, hde + s_i[q.id[i] >> 8], q.b0[i], q.b1[i]);
                        q.b0[i] = y.x;
                        q.b1[i] = y.y;
                    }
                    __syncwarp();
                    for (int i = 0; i < nq; i++)
                        if ((int)(q.id[i] & 255u) == lane) {
                            add_votes(0, q.b0[i]);
                            add_votes(1, q.b1[i]);
                        }
                    __syncwarp();
                    nq = 0;
                }
            }
        }
        const long long col = ix + (long long)it.n[0] * (iy + (long long)it.n[1] * iR);
        for (int s = 0; s < 2 && has; s++) {
            if (sign_only >= 0 && s != sign_only) continue;
            for (int iz = 0; iz < nz; iz++) {
                int v = 0;
#pragma unroll
                for (int i = 0; i < 9; i++) v |= (int)((pl[s][i] >> iz) & 1u) << i;
                vo[(long long)s * it.nvox + col + it.ncol * iz] = v;
                mx[s] = v > mx[s] ? v : mx[s];
            }
        }
    }
    if (mx[0] > 0) atomicMax(&s_vmax[0], mx[0]);
    if (mx[1] > 0) atomicMax(&s_vmax[1], mx[1]);
    __syncthreads();
    if (tid < 2 && s_vmax[tid] > 0) atomicMax(&vmax[(long long)e * 2 + tid], s_vmax[tid]);
}

// Statistics of the maximum-vote voxels of the accumulator with the larger maximum (force
// >= 0: of that sign's accumulator).
__global__ void __launch_bounds__(256)
k4_stats(Iter4 it, int ev0, const int32_t *votes, const int32_t *vmax, Stats4 *st, int force) {
    __shared__ unsigned long long s_cnt, s_sum[4];
    __shared__ int s_mn[4], s_mx[4];
    const int el = blockIdx.y, e = ev0 + el, tid = threadIdx.x;
    if (tid == 0) {
        s_cnt = 0;
        for (int a = 0; a < 4; a++) { s_sum[a] = 0; s_mn[a] = 1 << 30; s_mx[a] = -1; }
    }
    __syncthreads();
    const int s = force >= 0 ? force : (vmax[(long long)e * 2] >= vmax[(long long)e * 2 + 1] ? 0 : 1);
    const int vm = vmax[(long long)e * 2 + s];
    const int32_t *vo = votes + ((long long)el * 2 + s) * it.nvox;
    unsigned long long cnt = 0, sum[4] = {0, 0, 0, 0};
    int mn[4] = {1 << 30, 1 << 30, 1 << 30, 1 << 30}, mx[4] = {-1, -1, -1, -1};
    for (long long j = (long long)blockIdx.x * blockDim.x + tid; j < it.nvox; j += (long long)gridDim.x * blockDim.x) {
        if (__ldcs(vo + j) != vm) continue;
        long long r = j;
        int idx[4];
        for (int a = 0; a < 4; a++) { idx[a] = (int)(r % it.n[a]); r /= it.n[a]; }
        cnt++;
        for (int a = 0; a < 4; a++) {
            sum[a] += (unsigned long long)idx[a];
            mn[a] = idx[a] < mn[a] ? idx[a] : mn[a];
            mx[a] = idx[a] > mx[a] ? idx[a] : mx[a];
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        cnt += __shfl_down_sync(0xffffffffu, cnt, o);
        for (int a = 0; a < 4; a++) {
            sum[a] += __shfl_down_sync(0xffffffffu, sum[a], o);
            const int a1 = __shfl_down_sync(0xffffffffu, mn[a], o), b1 = __shfl_down_sync(0xffffffffu, mx[a], o);
            mn[a] = a1 < mn[a] ? a1 : mn[a];
            mx[a] = b1 > mx[a] ? b1 : mx[a];
        }
    }
    if ((tid & 31) == 0 && cnt) {
        atomicAdd(&s_cnt, cnt);
        for (int a = 0; a < 4; a++) {
            atomicAdd(&s_sum[a], sum[a]);
            atomicMin(&s_mn[a], mn[a]);
            atomicMax(&s_mx[a], mx[a]);
        }
    }
    __syncthreads();
    if (tid == 0 && s_cnt) {
        Stats4 &g = st[e];
        atomicAdd(&g.cnt, s_cnt);
        for (int a = 0; a < 4; a++) {
            atomicAdd(&g.sum[a], s_sum[a]);
            atomicMin(&g.mn[a], s_mn[a]);
            atomicMax(&g.mx[a], s_mx[a]);
        }
    }
}

// Active-hit bits from one byte per hit (CSR order), restricted to the staged valid hits.
__global__ void k4_active_bytes(const int32_t *offsets, const int32_t *n_hits, const uint8_t *in,
                                uint32_t *active) {
    const int e = blockIdx.x, wd = threadIdx.x;
    if (wd >= 8) return;
    const int n = n_hits[e] < 0 ? 0 : n_hits[e], a0 = offsets[e];
    uint32_t m = 0u;
    for (int b = 0; b < 32; b++) {
        const int i = 32 * wd + b;
        if (i < n && in[a0 + i]) m |= 1u << b;
    }
    active[(long long)e * 8 + wd] &= m;
}

__global__ void k4_reset_stats(int n, Stats4 *st, int32_t *vmax) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    Stats4 &g = st[e];
    g.cnt = 0;
    for (int a = 0; a < 4; a++) { g.sum[a] = 0; g.mn[a] = 1 << 30; g.mx[a] = -1; }
    if (vmax) vmax[2 * e] = vmax[2 * e + 1] = 0;
}

// Iteration 1 state: the global corner and the origin as reference point.
__global__ void k4_init(int n, double g0, double g1, double g2, double g3, double *lo, double *ref) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    lo[4 * e + 0] = g0; lo[4 * e + 1] = g1; lo[4 * e + 2] = g2; lo[4 * e + 3] = g3;
    ref[2 * e] = ref[2 * e + 1] = 0.0;
}

// Estimate, hit finding, and the next iteration's reference point and grid corner.
// One block per event.  k: this iteration; nxt (null after the last): the next one's
// shape; glo: the global corner.  Per-sign iteration 3 (lo2 / ref2 / active2: sign-major
// state of ne events):
//   force = s >= 0 (after iteration 2): the estimate of sign s's accumulator (st holds its
//     statistics), its hit finding into active2, its next reference point and corner into
//     ref2 / lo2; no record, no selection;
//   force < 0 with lo2 set (iteration 3): this iteration's corner and reference point are
//     those of the chosen sign in lo2 / ref2.
template <typename T>
__global__ void __launch_bounds__(256)
k4_finish(Iter4 it, int k, int n_iter, bool has_next, Iter4 nxt, double g0, double g1, double g2, double g3,
          const int32_t *offsets, const int32_t *n_hits, const HitRecD *hd, const int32_t *vmax,
          const Stats4 *st, double *lo, double *ref, uint32_t *active, apo4_iter *out, uint8_t *selected,
          int force, int ne, double *lo2, double *ref2, uint32_t *active2) {
    __shared__ double s_val[4], s_err[4];
    __shared__ int s_sign, s_cnt;
    __shared__ uint32_t s_act[8];
    __shared__ apo4_iter s_rec;   // the record of a forced-sign pass (not stored)
    const int e = blockIdx.x, tid = threadIdx.x;
    const int nh_raw = n_hits[e];
    const int nh = nh_raw < 0 ? 0 : nh_raw;
    const int sc = force >= 0 ? force : (vmax[2 * e] >= vmax[2 * e + 1] ? 0 : 1);
    const long long es = (long long)sc * ne + e;   // sign-major index
    apo4_iter &o = force >= 0 ? s_rec : out[(long long)e * n_iter + k];
    const double *le = (force < 0 && lo2) ? lo2 + es * 4 : lo + (long long)e * 4;
    const double *rf = (force < 0 && lo2) ? ref2 + es * 2 : ref + (long long)e * 2;
    double *le_out = force >= 0 ? lo2 + es * 4 : lo + (long long)e * 4;
    double *rf_out = force >= 0 ? ref2 + es * 2 : ref + (long long)e * 2;
    uint32_t *act_out = force >= 0 ? active2 + es * 8 : active + (long long)e * 8;
    if (force >= 0) selected = nullptr;
    if (tid == 0) {
        const int s = sc;
        const Stats4 g = st[e];
        const double m = (double)g.cnt;
        for (int a = 0; a < 4; a++) {
            const double mu = __ddiv_rn((double)g.sum[a], m);
            s_val[a] = __dadd_rn(le[a], __dmul_rn(it.w[a], __dadd_rn(mu, 0.5)));
            s_err[a] = __dmul_rn(__dmul_rn(it.w[a], (double)(g.mx[a] + 1 - g.mn[a])), 0.5);
            o.value[a] = s_val[a];
            o.err[a] = s_err[a];
        }
        o.ref[0] = rf[0];
        o.ref[1] = rf[1];
        s_sign = s == 0 ? 1 : -1;
        o.sign = s_sign;
        o.vmax = nh_raw < 0 ? nh_raw : vmax[2 * e + s];
        o.n_max = (int)g.cnt;
        s_cnt = 0;
    }
    if (tid < 8) s_act[tid] = 0u;
    __syncthreads();
    // hit finding on value +- hit_factor * error, every hit of the event
    double blo[4], bhi[4], c[4];
    for (int a = 0; a < 4; a++) {
        const double r = __dmul_rn(it.hit_factor, s_err[a]);
        blo[a] = __dsub_rn(s_val[a], r);
        bhi[a] = __dadd_rn(s_val[a], r);
        c[a] = mid4(blo[a], bhi[a]);
    }
    const Ctr4<T> m = centre4<T>(rn<T>(c[0]), rn<T>(c[1]), rn<T>(c[2]), rn<T>(it.p_gev), rn<T>(it.b_tesla),
                                 rn<T>(rf[0]), rn<T>(rf[1]));
    const IV<T> X = box_iv<T>(blo[0], bhi[0]), Y = box_iv<T>(blo[1], bhi[1]), Rv = box_iv<T>(blo[2], bhi[2]);
    const IV<T> Z = box_iv<T>(blo[3], bhi[3]);
    const int a0 = offsets[e], nseg = offsets[e + 1] - a0;
    for (int i = tid; i < nh; i += blockDim.x) {
        const HitRecD r = hd[(long long)e * kHitCap + i];
        bool v = false;
        if (m.valid) {
            const HitP<T> h = hit_point<T>(r);
            const Pre4<T> pre = prefix4<T>(m, rn<T>(c[3]), h);
            v = pre.guard || pair4<T>(m, pre, s_sign, h, a2_4<T>(X, Y, Z, hit_iv<T>(r)), Rv);
        }
        if (v) {
            atomicOr(&s_act[i >> 5], 1u << (i & 31));
            atomicAdd(&s_cnt, 1);
        }
        if (selected && !has_next) selected[a0 + i] = v ? 1 : 0;
    }
    if (selected && !has_next && nh_raw < 0 && a0 >= 0 && nseg >= 0 && nseg <= kHitCap)
        for (int i = tid; i < nseg; i += blockDim.x) selected[a0 + i] = 0;
    __syncthreads();
    if (tid < 8) act_out[tid] = s_act[tid];
    if (tid != 0) return;
    o.n_sel = s_cnt;
    if (!has_next) return;
    // next reference point: the selected hit's waist point nearest to the found circle
    double r0 = rf[0], r1 = rf[1], best = __longlong_as_double(0x7ff0000000000000LL);   // +inf
    for (int i = 0; i < nh; i++) {
        if (!((s_act[i >> 5] >> (i & 31)) & 1u)) continue;
        const HitRecD &r = hd[(long long)e * kHitCap + i];
        const double dx = __dsub_rn(r.v[0], s_val[0]), dy = __dsub_rn(r.v[1], s_val[1]);
        const double dist = fabs(__dsub_rn(__dsqrt_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy))), s_val[2]));
        if (dist < best) { best = dist; r0 = r.v[0]; r1 = r.v[1]; }
    }
    if (k + 1 == 1) {
        le_out[0] = g0; le_out[1] = g1; le_out[2] = g2; le_out[3] = g3;
    } else {
        // z0 moved from the old reference point to the new one: z0 + tan(lambda) R dpsi,
        // dpsi the difference of their phases from the direction of the origin
        const double xc = s_val[0], yc = s_val[1], R = s_val[2];
        const double ox = -xc, oy = -yc;
        const double on = __dsqrt_rn(__dadd_rn(__dmul_rn(ox, ox), __dmul_rn(oy, oy)));
        bool bad = !(on > 0.0);
        const double ax = __dsub_rn(rf[0], xc), ay = __dsub_rn(rf[1], yc);
        const double bx = __dsub_rn(r0, xc), by = __dsub_rn(r1, yc);
        const double pa = bad ? 0.0 : phase4<double>(ox, oy, on, ax, ay,
                                                     __dsqrt_rn(__dadd_rn(__dmul_rn(ax, ax), __dmul_rn(ay, ay))), bad);
        const double pb = bad ? 0.0 : phase4<double>(ox, oy, on, bx, by,
                                                     __dsqrt_rn(__dadd_rn(__dmul_rn(bx, bx), __dmul_rn(by, by))), bad);
        const double dpsi = bad ? 0.0 : __dsub_rn(pb, pa);
        const double ratio = __ddiv_rn(it.p_gev, __dmul_rn(__dmul_rn(0.3, it.b_tesla), R));
        const double aL = ratio > 1.0 ? __dsqrt_rn(__dsub_rn(__dmul_rn(ratio, ratio), 1.0)) : 0.0;
        const double L = s_sign > 0 ? aL : -aL;
        const double c3 = __dadd_rn(s_val[3], __dmul_rn(L, __dmul_rn(R, dpsi)));
        const double cc[4] = {s_val[0], s_val[1], s_val[2], c3};
        for (int a = 0; a < 4; a++)
            le_out[a] = __dsub_rn(cc[a], __dmul_rn(__dmul_rn((double)nxt.n[a], nxt.w[a]), 0.5));
    }
    rf_out[0] = r0;
    rf_out[1] = r1;
}

}  // namespace apo

namespace {

template <typename T>
void launch_vote4(const Iter4 &it, int ev0, int n, const int32_t *nh, const HitRecD *hd,
                  const uint32_t *active, const double *lo, const double *ref, int32_t *votes,
                  int32_t *vmax, cudaStream_t s, int sign_only = -1) {
    auto tiles = [&](int depth) {
        auto side = [&](int a, int s) { return (long long)((it.n[a] + s - 1) / s); };
        return side(0, k4Side) * side(1, k4Side) * side(2, depth);
    };
    int depth = k4Side;   // four waves of four blocks on 152 SMs
    while (depth > 2 && tiles(depth) * n < 4 * 4 * 152) depth /= 2;
    dim3 grid((unsigned)tiles(depth), n);
    k4_vote<T><<<grid, k4Threads, 0, s>>>(it, ev0, nh, hd, active, lo, ref, votes, vmax, sign_only, depth);
}

void launch_stats4(const Iter4 &it, int ev0, int n, const int32_t *votes, const int32_t *vmax,
                   Stats4 *st, cudaStream_t s, int force = -1) {
    long long b = (it.nvox + 256LL * 8 - 1) / (256LL * 8);
    dim3 grid((unsigned)(b < 1 ? 1 : (b > 1024 ? 1024 : b)), n);
    k4_stats<<<grid, 256, 0, s>>>(it, ev0, votes, vmax, st, force);
}

template <typename T>
void launch_finish4(const Iter4 &it, int k, const apo4_opts *o, bool has_next, const Iter4 &nxt,
                    const apo_hits *hits, const int32_t *nh, const HitRecD *hd, const int32_t *vmax,
                    const Stats4 *st, double *lo, double *ref, uint32_t *active, apo4_iter *out,
                    uint8_t *selected, int force, int ne, double *lo2, double *ref2, uint32_t *active2,
                    cudaStream_t s) {
    k4_finish<T><<<ne, 256, 0, s>>>(it, k, o->n_iter, has_next, nxt, o->glo[0], o->glo[1], o->glo[2], o->glo[3],
                                    hits->offsets, nh, hd, vmax, st, lo, ref, active, out, selected, force, ne,
                                    lo2, ref2, active2);
}

int check_hits4(const apo_hits *h) {
    if (!h) return fail4(APO_EINVAL, "hits is NULL");
    if (h->n_events < 0) return fail4(APO_EINVAL, "n_events < 0");
    if (h->n_events > 0 && (!h->offsets || !h->wire_id || !h->drift))
        return fail4(APO_EINVAL, "hits arrays must be non-NULL");
    return APO_OK;
}

int check_chamber(const apo4_chamber *c) {
    if (!c) return fail4(APO_EINVAL, "chamber is NULL");
    int dev = -1;
    CU4(cudaGetDevice(&dev));
    if (dev != c->device) return fail4(APO_EINVAL, "chamber lives on device %d, current is %d", c->device, dev);
    return APO_OK;
}

int check_ws4(const apo4_opts *o, int ne, void *ws, size_t bytes, Layout4 &L) {
    L = layout4(o, ne);
    if (!ws) return fail4(APO_EINVAL, "workspace is NULL");
    if (reinterpret_cast<uintptr_t>(ws) % 256) return fail4(APO_EINVAL, "workspace must be 256-byte aligned");
    if (bytes < L.end) return fail4(APO_ENOMEM, "workspace too small: %zu < %zu bytes", bytes, L.end);
    return APO_OK;
}

template <typename P> P *at4(void *ws, size_t off) { return reinterpret_cast<P *>(static_cast<unsigned char *>(ws) + off); }

}  // namespace

extern "C" {

void apo4_opts_default(apo4_opts *o) {
    if (!o) return;
    std::memset(o, 0, sizeof(*o));
    o->p_gev = 0.105;
    o->b_tesla = 1.0;
    o->disk_radius = 0.10;
    o->hit_factor = 5.0;
    const double glo[4] = {-0.45, -0.45, 0.225, -0.75};
    const double w[3][4] = {{0.018, 0.018, 0.00375, 0.075}, {0.010, 0.010, 0.00375, 0.075},
                            {0.001, 0.001, 0.001, 0.040}};
    const int n[3][4] = {{50, 50, 40, 20}, {90, 90, 40, 20}, {50, 50, 50, 20}};
    for (int a = 0; a < 4; a++) o->glo[a] = glo[a];
    for (int k = 0; k < 3; k++)
        for (int a = 0; a < 4; a++) { o->w[k][a] = w[k][a]; o->n[k][a] = n[k][a]; }
    o->precision = APO_F64;
    o->n_iter = 3;
    o->per_sign = 1;
}

int apo4_chamber_create(const apo_wires *w, apo4_chamber **out) {
    if (!out) return fail4(APO_EINVAL, "out is NULL");
    *out = nullptr;
    if (!w || w->n_wires <= 0) return fail4(APO_EINVAL, "wires missing");
    const double *wa[8] = {w->x0, w->y0, w->sin_phis, w->cos_phis, w->tan_tau, w->sphi_t, w->cphi_t, w->t2};
    for (int i = 0; i < 8; i++)
        if (!wa[i]) return fail4(APO_EINVAL, "wire array %d is NULL", i);
    apo4_chamber *c = new apo4_chamber();
    std::memset(&c->dg, 0, sizeof(c->dg));
    CU4(cudaGetDevice(&c->device));
    c->dg.n_wires = w->n_wires;
    for (int i = 0; i < 8; i++) {
        void *p = nullptr;
        cudaError_t e = cudaMalloc(&p, sizeof(double) * (size_t)w->n_wires);
        if (e == cudaSuccess) {
            c->allocs.push_back(p);
            e = cudaMemcpy(p, wa[i], sizeof(double) * (size_t)w->n_wires, cudaMemcpyHostToDevice);
        }
        if (e != cudaSuccess) {
            apo4_chamber_destroy(c);
            return fail4(APO_ECUDA, "wire upload: %s", cudaGetErrorString(e));
        }
        c->dg.wire[i] = static_cast<const double *>(p);
    }
    *out = c;
    return APO_OK;
}

void apo4_chamber_destroy(apo4_chamber *c) {
    if (!c) return;
    for (void *p : c->allocs) cudaFree(p);
    delete c;
}

int apo4_workspace_bytes(const apo4_chamber *c, int32_t n_events, const apo4_opts *o, size_t *bytes) {
    int rc;
    if (!c || !bytes) return fail4(APO_EINVAL, "NULL argument");
    if ((rc = check_opts(o))) return rc;
    if (n_events < 0) return fail4(APO_EINVAL, "n_events < 0");
    *bytes = layout4(o, n_events).end;
    return APO_OK;
}

int apo4_solve_batch(const apo4_chamber *c, const apo_hits *hits, const apo4_opts *o, apo4_iter *out,
                     uint8_t *selected, void *ws, size_t ws_bytes, void *stream) {
    int rc;
    if ((rc = check_chamber(c)) || (rc = check_hits4(hits)) || (rc = check_opts(o))) return rc;
    const int ne = hits->n_events;
    if (ne > 0 && !out) return fail4(APO_EINVAL, "out is NULL");
    Layout4 L;
    if ((rc = check_ws4(o, ne, ws, ws_bytes, L))) return rc;
    if (ne == 0) return APO_OK;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    unsigned *status = at4<unsigned>(ws, L.status);
    int32_t *nh = at4<int32_t>(ws, L.nh);
    HitRecD *hd = at4<HitRecD>(ws, L.hd);
    HitRecF *hf = at4<HitRecF>(ws, L.hf);
    uint32_t *active = at4<uint32_t>(ws, L.active);
    int32_t *done = at4<int32_t>(ws, L.done);
    double *lo = at4<double>(ws, L.lo);
    double *ref = at4<double>(ws, L.ref);
    int32_t *vmax = at4<int32_t>(ws, L.vmax);
    Stats4 *st = at4<Stats4>(ws, L.stats);
    double *lo2 = at4<double>(ws, L.lo2);
    double *ref2 = at4<double>(ws, L.ref2);
    uint32_t *active2 = at4<uint32_t>(ws, L.active2);
    Stats4 *st2 = at4<Stats4>(ws, L.stats2);
    int32_t *votes = at4<int32_t>(ws, L.votes);
    // per-sign iteration 3: after iteration 2 each sign's accumulator gets its own estimate,
    // hit finding, reference point and box; iteration 3 votes sign s on box s
    const bool ps = o->per_sign && o->n_iter == 3;
    const bool f32 = o->precision == APO_F32;
    CU4(cudaMemsetAsync(status, 0, 256, s));
    launch_stage(c->dg, ne, hits->offsets, hits->wire_id, hits->drift, hd, hf, nh, active, done, status, s);
    k4_init<<<(ne + 127) / 128, 128, 0, s>>>(ne, o->glo[0], o->glo[1], o->glo[2], o->glo[3], lo, ref);
    CU4(cudaGetLastError());
    for (int k = 0; k < o->n_iter; k++) {
        const Iter4 it = iter4(o, k);
        const bool has_next = k + 1 < o->n_iter;
        const Iter4 nxt = has_next ? iter4(o, k + 1) : it;
        const bool split_stats = ps && k == 1, split_vote = ps && k == 2;
        k4_reset_stats<<<(ne + 127) / 128, 128, 0, s>>>(ne, st, vmax);
        if (split_stats) k4_reset_stats<<<(2 * ne + 127) / 128, 128, 0, s>>>(2 * ne, st2, nullptr);
        for (int e0 = 0; e0 < ne; e0 += L.chunk) {
            const int n = ne - e0 < L.chunk ? ne - e0 : L.chunk;
            for (int sg = split_vote ? 0 : -1; sg < (split_vote ? 2 : 0); sg++) {
                const uint32_t *ac = sg < 0 ? active : active2 + (size_t)sg * ne * 8;
                const double *lc = sg < 0 ? lo : lo2 + (size_t)sg * ne * 4;
                const double *rc = sg < 0 ? ref : ref2 + (size_t)sg * ne * 2;
                if (f32) launch_vote4<float>(it, e0, n, nh, hd, ac, lc, rc, votes, vmax, s, sg);
                else launch_vote4<double>(it, e0, n, nh, hd, ac, lc, rc, votes, vmax, s, sg);
            }
            launch_stats4(it, e0, n, votes, vmax, st, s);
            if (split_stats)
                for (int sg = 0; sg < 2; sg++) launch_stats4(it, e0, n, votes, vmax, st2 + (size_t)sg * ne, s, sg);
        }
        if (split_stats)   // before the chosen sign's pass, which moves lo / ref on
            for (int sg = 0; sg < 2; sg++) {
                if (f32)
                    launch_finish4<float>(it, k, o, has_next, nxt, hits, nh, hd, vmax, st2 + (size_t)sg * ne, lo, ref,
                                          active, out, nullptr, sg, ne, lo2, ref2, active2, s);
                else
                    launch_finish4<double>(it, k, o, has_next, nxt, hits, nh, hd, vmax, st2 + (size_t)sg * ne, lo,
                                           ref, active, out, nullptr, sg, ne, lo2, ref2, active2, s);
            }
        if (f32)
            launch_finish4<float>(it, k, o, has_next, nxt, hits, nh, hd, vmax, st, lo, ref, active, out, selected, -1,
                                  ne, split_vote ? lo2 : nullptr, split_vote ? ref2 : nullptr, active2, s);
        else
            launch_finish4<double>(it, k, o, has_next, nxt, hits, nh, hd, vmax, st, lo, ref, active, out, selected,
                                   -1, ne, split_vote ? lo2 : nullptr, split_vote ? ref2 : nullptr, active2, s);
        CU4(cudaGetLastError());
    }
    return APO_OK;
}

int apo4_vote(const apo4_chamber *c, const apo_hits *hits, const apo4_opts *o, int32_t iter, const double *lo,
              const double *ref, const uint8_t *active_in, int32_t *votes_out, void *ws, size_t ws_bytes,
              void *stream) {
    int rc;
    if ((rc = check_chamber(c)) || (rc = check_hits4(hits)) || (rc = check_opts(o))) return rc;
    if (iter < 0 || iter >= o->n_iter) return fail4(APO_EINVAL, "iter out of range");
    const int ne = hits->n_events;
    if (ne > 0 && (!lo || !ref || !votes_out)) return fail4(APO_EINVAL, "lo, ref and votes must be non-NULL");
    Layout4 L;
    if ((rc = check_ws4(o, ne, ws, ws_bytes, L))) return rc;
    if (ne == 0) return APO_OK;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    unsigned *status = at4<unsigned>(ws, L.status);
    int32_t *nh = at4<int32_t>(ws, L.nh);
    HitRecD *hd = at4<HitRecD>(ws, L.hd);
    HitRecF *hf = at4<HitRecF>(ws, L.hf);
    uint32_t *active = at4<uint32_t>(ws, L.active);
    int32_t *done = at4<int32_t>(ws, L.done);
    int32_t *vmax = at4<int32_t>(ws, L.vmax);
    Stats4 *st = at4<Stats4>(ws, L.stats);
    CU4(cudaMemsetAsync(status, 0, 256, s));
    launch_stage(c->dg, ne, hits->offsets, hits->wire_id, hits->drift, hd, hf, nh, active, done, status, s);
    if (active_in) k4_active_bytes<<<ne, 32, 0, s>>>(hits->offsets, nh, active_in, active);
    k4_reset_stats<<<(ne + 127) / 128, 128, 0, s>>>(ne, st, vmax);
    const Iter4 it = iter4(o, iter);
    // the caller's array holds every event: vote all of them in one launch
    if (o->precision == APO_F32) launch_vote4<float>(it, 0, ne, nh, hd, active, lo, ref, votes_out, vmax, s);
    else launch_vote4<double>(it, 0, ne, nh, hd, active, lo, ref, votes_out, vmax, s);
    CU4(cudaGetLastError());
    return APO_OK;
}

}  // extern "C"

// own.cu -- block-owned layout of the analytic Schur product (pcg_own_kernel).
//
// The sliced point order (sell.cu) is dealt to blocks, one per CTA of the PCG
// kernel: slice i belongs to block i mod nblk.  A block owns its points, so
// b_j = C~_j^-1 sum u never leaves the CTA, and the camera side of the product
// runs over the block's own observations, grouped by camera: a run is the
// observations of one camera in one block.  Runs are laid out like the point
// slices, sorted by decreasing length, G lanes per run: round k of a run slice
// is 32 consecutive slots, a run's nine sums stay in its lanes, and each run
// ends in one store to the block's row of the partial sums, which the camera's
// owner adds in block order.  Cameras with long runs (few cameras) are split
// into parts, each with its own row.
//
// G is one number for most slices (OwnPlan).  A slice whose first (longest) run
// would take more than kRunRounds rounds takes more lanes per run, up to a whole
// warp: a camera that sees far more points than the others would otherwise pad
// its 32 / G - 1 neighbours to its own length and keep one warp busy long after
// the others (see own_cameras for the times).
#include <algorithm>

#include "mba_internal.cuh"

namespace mba {

namespace {

__global__ void point_blocks_kernel(const int4 *__restrict__ slice, int32_t n_slices, int32_t nblk,
                                    int2 *__restrict__ sp_bl) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_slices; i += gridDim.x * blockDim.x) {
        const int4 s = slice[i];
        const int count = s.y & 0xff, base = s.y >> 8;
        for (int p = 0; p < count; ++p) sp_bl[s.x + p] = make_int2(i % nblk, base + p);
    }
}

__global__ void obs_block_kernel(const int32_t *__restrict__ cm_sp, const int2 *__restrict__ sp_bl, int64_t n,
                                 int32_t *__restrict__ key) {
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n; s += (int64_t)gridDim.x * blockDim.x)
        key[s] = sp_bl[cm_sp[s]].x;
}

// run index block * nc + camera of every observation, in (block, camera) order
__global__ void run_key_kernel(const int32_t *__restrict__ ord, const int32_t *__restrict__ key,
                               const int32_t *__restrict__ cam_ptr, int32_t nc, int64_t n, int32_t *__restrict__ run,
                               int32_t *__restrict__ count) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
        const int s = ord[t];
        int lo = 0, hi = nc - 1;  // last camera with cam_ptr <= s
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (cam_ptr[mid] <= s) lo = mid;
            else hi = mid - 1;
        }
        const int r = key[s] * nc + lo;
        run[t] = r;
        atomicAdd(count + r, 1);
    }
}

__global__ void fill_runs_kernel(Prob P, const int32_t *__restrict__ ord, const int32_t *__restrict__ run,
                                 const int32_t *__restrict__ run_ptr, const int2 *__restrict__ base, int parts,
                                 const int2 *__restrict__ sp_bl, int32_t *__restrict__ orig2r,
                                 const int32_t *__restrict__ flag) {
    if (*flag & 2) return;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < P.n; t += (int64_t)gridDim.x * blockDim.x) {
        const int s = ord[t], r = run[t], k = (int)(t - run_ptr[r]);
        const int part = k % parts, kk = k / parts;
        const int2 at = base[(int64_t)r * parts + part];  // first slot, log2 G
        const int slot = at.x + 32 * (kk >> at.y) + (kk & ((1 << at.y) - 1));
        if (P.fp32) P.cm2r[s] = slot;
        else orig2r[P.cm_orig[s]] = slot;
        const int sp = P.cm_sp[s];
        if (P.r_pt16) P.r_pt16[slot] = (uint16_t)sp_bl[sp].y;
        else P.r_pt[slot] = sp;
    }
}

// slot -> observation in the input order (fill_slots_kernel) -> run slot
__global__ void slot_runs_kernel(Prob P, const int32_t *__restrict__ orig2r, const int32_t *__restrict__ flag) {
    if (*flag & 2) return;
    for (int64_t o = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; o < P.nslots; o += (int64_t)gridDim.x * blockDim.x)
        if (P.sl_cam[o] >= 0) P.sl2r[o] = orig2r[P.sl2r[o]];
}

// part of a run of l observations: those k with k mod parts equal to it
__device__ __forceinline__ int part_len(int l, int parts, int part) { return (l + parts - 1 - part) / parts; }

// rounds of a slice whose longest run has len observations, G = 2^lg lanes per run
__host__ __device__ __forceinline__ int run_rounds(int len, int lg) { return (len + (1 << lg) - 1) >> lg; }

// One CTA per block: its (camera, part) pairs by decreasing length, then index
// (bitonic sort of m = 2^k keys in shared memory), and their slices: (first pair,
// K | log2 G << kRunLg).  info: slices, rounds, slices of more than kRunRounds rounds.
__global__ void __launch_bounds__(512) sort_runs_kernel(const int32_t *__restrict__ len, int nc, int parts, int lg0,
                                                        int m, unsigned long long *__restrict__ sorted,
                                                        int2 *__restrict__ cut, int4 *info) {
    extern __shared__ unsigned long long key[];
    __shared__ int s_used, s_rounds, s_slices, s_from, s_long;
    const int items = nc * parts, per0 = 32 >> lg0;
    const int32_t *l = len + (int64_t)blockIdx.x * nc;
    if (threadIdx.x == 0) s_used = 0, s_rounds = 0;
    for (int i = threadIdx.x; i < m; i += blockDim.x)
        key[i] = i < items ? ((unsigned long long)(unsigned)~part_len(l[i / parts], parts, i % parts) << 32) | (unsigned)i
                           : ~0ull;
    for (int k = 2; k <= m; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            __syncthreads();
            for (int t = threadIdx.x; t < m / 2; t += blockDim.x) {
                const int i = 2 * t - (t & (j - 1)), o = i + j;
                const unsigned long long a = key[i], b = key[o];
                if ((a > b) == ((i & k) == 0)) key[i] = b, key[o] = a;
            }
        }
    __syncthreads();
    int used = 0;
    for (int i = threadIdx.x; i < items; i += blockDim.x) {
        const unsigned long long a = key[i];
        sorted[(int64_t)blockIdx.x * items + i] = a;
        if ((int)~(unsigned)(a >> 32) > 0) ++used;
    }
    atomicAdd(&s_used, used);
    __syncthreads();
    // the long runs first, slice by slice, then the others, 2^lg0 lanes each
    int2 *out = cut + (int64_t)blockIdx.x * items;
    if (threadIdx.x == 0) {
        int q = 0, j = 0, rounds = 0, longs = 0;
        while (q < s_used) {
            const int n = (int)~(unsigned)(key[q] >> 32);
            int lg = lg0;
            while (lg < 5 && run_rounds(n, lg) > kRunRounds) ++lg;
            if (lg == lg0) break;
            const int K = run_rounds(n, lg);
            out[j++] = make_int2(q, K | (lg << kRunLg));
            rounds += K;
            longs += K > kRunRounds;
            q += 32 >> lg;
        }
        s_from = q;
        s_slices = j;
        s_rounds = rounds;
        s_long = longs;
    }
    __syncthreads();
    const int from = s_from, rest = from < s_used ? (s_used - from + per0 - 1) / per0 : 0;
    int rounds = 0;
    for (int j = threadIdx.x; j < rest; j += blockDim.x) {
        const int q = from + j * per0, K = run_rounds((int)~(unsigned)(key[q] >> 32), lg0);
        out[s_slices + j] = make_int2(q, K | (lg0 << kRunLg));
        rounds += K;
    }
    atomicAdd(&s_rounds, rounds);
    __syncthreads();
    if (threadIdx.x == 0) info[blockIdx.x] = make_int4(s_slices + rest, s_rounds, s_long, 0);
}

// The run slices of a block (from slice first[b], round round0[b]): first slot and
// rounds, the (camera, row of the partial sums) of every lane, and the first slot
// and lanes of every (camera, part).
constexpr int kBlockSlices = 4096;  // a block has no more (camera, part) pairs
__global__ void __launch_bounds__(256) run_slices_kernel(Prob P, const unsigned long long *__restrict__ sorted,
                                                         const int2 *__restrict__ cut,
                                                         const int32_t *__restrict__ round0, int parts,
                                                         int2 *__restrict__ base, const int32_t *__restrict__ flag) {
    __shared__ int s_start[kBlockSlices];
    if (*flag & 2) return;
    const int b = blockIdx.x, items = P.nc * parts;
    const int first = P.blk_run[b].x, nsl = P.blk_run[b].z - first;
    const unsigned long long *key = sorted + (int64_t)b * items;
    cut += (int64_t)b * items;
    for (int j = threadIdx.x; j < nsl; j += blockDim.x) s_start[j] = cut[j].y & kRunMask;
    __syncthreads();
    if (threadIdx.x == 0) {
        int r = round0[b];
        for (int j = 0; j < nsl; ++j) {
            const int K = s_start[j];
            s_start[j] = r;
            r += K;
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 32 * nsl; i += blockDim.x) {
        const int j = i >> 5, lane = i & 31;
        const int2 c = cut[j];
        const int lg = c.y >> kRunLg, q = c.x + (lane >> lg);
        if (lane == 0) P.rslice[first + j] = make_int2(32 * s_start[j], c.y);
        int2 ln = make_int2(-1, 0);
        const unsigned long long a = q < items ? key[q] : ~0ull;
        if ((int)~(unsigned)(a >> 32) > 0) {
            const int it = (int)(a & 0xffffffffu), cam = it / parts, part = it % parts;
            ln = make_int2(cam, b * parts + part);
            if ((lane & ((1 << lg) - 1)) == 0)
                base[((int64_t)b * P.nc + cam) * parts + part] = make_int2(32 * s_start[j] + lane, lg);
        }
        P.rlane[32 * (int64_t)first + i] = ln;
    }
}

inline unsigned grid_for(int64_t n) {
    int64_t g = (n + kBlock - 1) / kBlock;
    if (g > 152 * 16) g = 152 * 16;
    return (unsigned)(g < 1 ? 1 : g);
}

size_t al256(size_t v) { return (v + 255) & ~size_t(255); }

// First slice and round of every block (one CTA, any number of blocks).  flag: bit 0
// some slice has more than kRunRounds rounds, bit 1 the arrays are too small (their
// size is a bound, so this does not happen; nothing is written then).
__global__ void __launch_bounds__(1024) run_offsets_kernel(const int4 *__restrict__ info, int nblk, int64_t cap_slices,
                                                           int64_t cap_slots, int4 *__restrict__ blk_run,
                                                           int32_t *__restrict__ round0, int32_t *flag) {
    __shared__ int2 s[1024];
    __shared__ int s_long;
    const int t = threadIdx.x;
    if (t == 0) s_long = 0;
    int2 carry = make_int2(0, 0);
    for (int b0 = 0; b0 < nblk; b0 += 1024) {
        const int4 v = b0 + t < nblk ? info[b0 + t] : make_int4(0, 0, 0, 0);
        __syncthreads();
        s[t] = make_int2(v.x, v.y);
        if (v.z > 0) s_long = 1;
        for (int d = 1; d < 1024; d <<= 1) {
            __syncthreads();
            const int2 a = s[t], b = t >= d ? s[t - d] : make_int2(0, 0);
            __syncthreads();
            s[t] = make_int2(a.x + b.x, a.y + b.y);
        }
        __syncthreads();
        const int first = carry.x + s[t].x - v.x;
        if (b0 + t < nblk) {
            blk_run[b0 + t] = make_int4(first, first + v.z, first + v.x, 0);
            round0[b0 + t] = carry.y + s[t].y - v.y;
        }
        carry.x += s[1023].x;
        carry.y += s[1023].y;
    }
    __syncthreads();
    if (t == 0) *flag = s_long | (carry.x > cap_slices || 32ll * carry.y > cap_slots ? 2 : 0);
}

// How the runs of nblk blocks are laid out, and how large that can get.
struct OwnPlan {
    int64_t nblk;
    int parts, lg;           // parts of a camera's run, log2 of the lanes per run
    int64_t slices, slots;   // run slices and slots, at most
};
OwnPlan own_plan(const Prob &P, int64_t nblk) {
    OwnPlan pl{};
    pl.nblk = nblk;
    // few cameras: split their runs until a block has work for a few hundred lanes
    const double mean = (double)P.n / ((double)nblk * P.nc);
    pl.parts = 1;
    while (pl.parts < kMaxParts && (int64_t)P.nc * pl.parts < 128 && mean / pl.parts > 16.0) pl.parts *= 2;
    // lanes per run, no more than the mean run fills.  FP32: a few rounds of the
    // CTA's warps.  FP64: two where the runs then still fit its 512 lanes twice,
    // more only to give the FP64 pipe a handful of warps (the reduction of nine
    // values over a run's lanes takes a third of a round's pipe time per level)
    const int64_t items = (int64_t)P.nc * pl.parts;
    while (pl.lg < 3 && (2 << pl.lg) <= mean / pl.parts &&
           (items << (pl.lg + 1)) <= (P.fp32 ? 4096 : (pl.lg == 0 ? 1024 : 256)))
        ++pl.lg;
    // Slots.  A slice that follows one with as many lanes per run takes, per run, no
    // more than a run of the slice before it, rounded up to G: together n and the
    // rounding.  A slice whose runs have a warp each pads only to 32.  That leaves
    // the first slice of each number of lanes in a block, at most kRunRounds rounds;
    // one with 2^c lanes, more than usual, holds a run of more than kRunRounds 2^(c-1).
    const int64_t G = int64_t(1) << pl.lg, per = 32 / G, n = P.n;
    const int64_t used = items * nblk < n ? items * nblk : n, longs = n / (kRunRounds * G);
    const int64_t usual = used / per + nblk;  // slices of the usual number of lanes
    pl.slices = usual + longs;
    pl.slots = n + (G - 1) * per * usual + 31 * longs + std::min<int64_t>(32 * kRunRounds * nblk, 32 * (n / G + nblk));
    for (int c = pl.lg + 1; c < 5; ++c)
        pl.slots += 32 * kRunRounds * std::min<int64_t>(nblk, n / (kRunRounds << (c - 1)));
    pl.slots = (pl.slots + 31) / 32 * 32;
    return pl;
}

// The arrays of a plan in a piece of memory (base NULL: only their size).
size_t own_arrays(Prob &P, const OwnPlan &pl, char *base) {
    size_t off = 0;
    auto arr = [&](size_t bytes) -> void * {
        void *p = base ? base + off : nullptr;
        off += al256(bytes ? bytes : 1);
        return p;
    };
    const size_t ns = (size_t)pl.slots;
    P.rslot_cap = pl.slots;
    P.rslice = (int2 *)arr(8 * (size_t)pl.slices);
    P.rlane = (int2 *)arr(32 * 8 * (size_t)pl.slices);
    P.blk_run = (int4 *)arr(16 * (size_t)pl.nblk);
    P.cm2r = P.fp32 ? (int32_t *)arr(4 * (size_t)P.n) : nullptr;
    P.c_part = arr((size_t)pl.nblk * pl.parts * P.nc * (P.fp32 ? kPartF * 4 : kPartD * 8));
    if (P.fp32) {
        P.r_rx = (float4 *)arr(16 * ns);
        P.r_pt16 = (uint16_t *)arr(2 * ns);
        P.r_w = P.loss != MBA_LOSS_NONE ? (float *)arr(4 * ns) : nullptr;
    } else {
        P.r_pt = (int32_t *)arr(4 * ns);
        P.r_hg = (double2 *)arr(80 * ns);
    }
    return off;
}

// Blocks per CTA with which b of a block's points is sure to fit in shared memory,
// kMaxBlocks if none is (FP64 keeps b in global memory: one block per CTA fits).
int own_blocks(const Prob &P, int grid) {
    int m = 1;
    Prob Q = P;
    while (m < kMaxBlocks && !own_fits(Q, grid, m, sell_block_points(P.n, P.np, (int64_t)grid * m))) ++m;
    return m;
}

}  // namespace

// Shared memory of the block-owned PCG kernel with m blocks per CTA of at most pb
// points: camera rows; b of a block's points (FP32) or the owner's group sums over
// all blocks; dot products and the owner's six vectors.
bool own_fits(Prob &P, int grid, int m, int64_t pb) {
    const int64_t rows = ((int64_t)P.nc * (P.fp32 ? kRowS * 4 : kRowD * 8) + 127) / 128 * 128;
    const int64_t cams = (P.nc + grid - 1) / grid;  // cameras of an owner, at most
    const int64_t dots = (3 + 6) * 9 * cams * 8;
    const int64_t vblk = (int64_t)grid * m * (P.nc >= 128 ? 1 : kMaxParts);
    int64_t region = (vblk + 7) / 8 * 9 * cams * 8;
    if (P.fp32 && pb * 12 > region) region = pb * 12;
    region = (region + 127) / 128 * 128;
    if (rows + region + dots > kOwnSmem || (P.fp32 && pb > 65000)) return false;
    P.nblk = grid * m;
    P.own_pb = (int32_t)pb;
    P.own_off_b = (int32_t)rows;
    P.own_off_dots = (int32_t)(rows + region);
    P.pcg_smem = (int32_t)(rows + region + dots);
    return true;
}

// The block-owned product is used where the camera rows leave room in shared
// memory and where the runs are long enough that the partial sums (written and
// read once per product) cost less than the gathers of b they replace: at least
// kMinRun observations on average, or partial sums of a few MB, which stay in L2.
constexpr double kMinRun = 4.0;
constexpr int64_t kSmallParts = 16 << 20;
bool own_wanted(const Prob &P, int grid) {
    const int64_t rows = (int64_t)P.nc * (P.fp32 ? kRowS * 4 : kRowD * 8);
    const int64_t parts = (int64_t)grid * P.nc * (P.fp32 ? kPartF * 4 : kPartD * 8);
    if (rows + 40 * 1024 > kOwnSmem || ((double)P.n < kMinRun * (double)grid * P.nc && parts > kSmallParts)) return false;
    Prob Q = P;
    if (!P.fp32 && !own_fits(Q, grid, 1, 0)) return false;  // no other form to fall back to
    for (int m = 1; m <= kMaxBlocks; ++m)
        if (own_plan(P, (int64_t)grid * m).slots >= (int64_t(1) << 31) - 64) return false;
    return true;
}

// Memory of the layout, whatever the slices turn out to be: the largest over the
// numbers of blocks that may be taken and, where none is sure to fit (FP32), the
// gathered product's arrays.
size_t own_pool_bytes(const Prob &P, int grid) {
    Prob Q = P;
    if (!P.own) return P.fact ? gathered_arrays(Q, nullptr) : 0;
    const int most = P.fp32 ? own_blocks(P, grid) : 1;
    size_t bytes = 0;
    for (int m = 1; m <= most; ++m) bytes = std::max(bytes, own_arrays(Q, own_plan(P, (int64_t)grid * m), nullptr));
    if (P.fp32 && most == kMaxBlocks) bytes = std::max(bytes, gathered_arrays(Q, nullptr));
    return bytes;
}

// The gathered FP32 product's arrays in a piece of memory (base NULL: only their size).
size_t gathered_arrays(Prob &P, char *base) {
    size_t off = 0;
    auto arr = [&](size_t bytes) -> void * {
        void *p = base ? base + off : nullptr;
        off += al256(bytes);
        return p;
    };
    P.RXcm = (float4 *)arr(16 * (size_t)P.n);
    P.sp_b = (float4 *)arr(16 * (size_t)P.np);
    P.cm_w = P.loss != MBA_LOSS_NONE ? (float *)arr(4 * (size_t)P.n) : nullptr;
    return off;
}

size_t own_tmp_bytes(const Prob &P, int grid) {
    const int64_t nblk = (int64_t)grid * (P.fp32 ? own_blocks(P, grid) : 1);
    return al256(8 * (size_t)P.np) + 3 * al256(4 * (size_t)P.n) + 2 * al256(4 * ((size_t)nblk * P.nc + 2)) +
           3 * al256(8 * (size_t)nblk * P.nc * (P.nc < 128 ? kMaxParts : 1)) + al256(16 * (size_t)nblk) +
           al256(4 * (size_t)nblk) + al256(4 * (size_t)exclusive_scan_tmp_ints(nblk * P.nc + 2)) +
           stable_sort_tmp_bytes(P.n, (int32_t)nblk + 1);
}

// Builds the run layout in `pool` (own_pool_bytes), on the device alone: with its
// sizes read back and its arrays allocated here, the creation of 2,000 points took
// 0.83 instead of 0.76 ms, of 50k points (FP32) 1.12 instead of 0.99.  *flag: see
// run_offsets_kernel.
cudaError_t build_own(Prob &P, void *tmp, size_t tmp_bytes, void *pool, size_t pool_bytes, int32_t *flag, cudaStream_t s) {
    const OwnPlan pl = own_plan(P, P.nblk);
    const int64_t nblk = P.nblk, nruns = nblk * P.nc;
    if (own_arrays(P, pl, (char *)pool) > pool_bytes) return cudaErrorInvalidValue;
    P.n_vblk = (int32_t)(nblk * pl.parts);
    char *t = (char *)tmp;
    auto take = [&](size_t bytes) {
        char *p = t;
        t += al256(bytes);
        return p;
    };
    int2 *sp_bl = (int2 *)take(8 * (size_t)P.np);
    int32_t *key = (int32_t *)take(4 * (size_t)P.n), *ord = (int32_t *)take(4 * (size_t)P.n),
            *run = (int32_t *)take(4 * (size_t)P.n);
    int32_t *count = (int32_t *)take(4 * ((size_t)nruns + 2)), *run_ptr = (int32_t *)take(4 * ((size_t)nruns + 2));
    const size_t pairs = 8 * (size_t)nruns * (P.nc < 128 ? kMaxParts : 1);
    int2 *base_d = (int2 *)take(pairs), *cut = (int2 *)take(pairs);
    auto *sorted = (unsigned long long *)take(pairs);
    int4 *info_d = (int4 *)take(16 * (size_t)nblk);
    int32_t *round0_d = (int32_t *)take(4 * (size_t)nblk);
    int32_t *scan_tmp = (int32_t *)take(4 * (size_t)exclusive_scan_tmp_ints(nruns + 2));
    const size_t sort_bytes = stable_sort_tmp_bytes(P.n, (int32_t)nblk + 1);
    if ((size_t)(t - (char *)tmp) + sort_bytes > tmp_bytes) return cudaErrorInvalidValue;

    point_blocks_kernel<<<grid_for(P.n_slices), kBlock, 0, s>>>(P.slice, P.n_slices, P.nblk, sp_bl);
    obs_block_kernel<<<grid_for(P.n), kBlock, 0, s>>>(P.cm_sp, sp_bl, P.n, key);
    cudaError_t e = stable_sort_by_key(key, P.n, (int32_t)nblk, ord, nullptr, t, sort_bytes, s);
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(count, 0, 4 * ((size_t)nruns + 2), s);
    if (e != cudaSuccess) return e;
    run_key_kernel<<<grid_for(P.n), kBlock, 0, s>>>(ord, key, P.cam_ptr, P.nc, P.n, run, count);
    e = exclusive_scan_i32(count, run_ptr, nruns + 1, scan_tmp, s);
    if (e != cudaSuccess) return e;
    int m = 2;
    while (m < P.nc * pl.parts) m *= 2;
    if (m > kBlockSlices) return cudaErrorInvalidValue;
    sort_runs_kernel<<<(unsigned)nblk, 512, 8 * (size_t)m, s>>>(count, P.nc, pl.parts, pl.lg, m, sorted, cut, info_d);
    run_offsets_kernel<<<1, 1024, 0, s>>>(info_d, (int)nblk, pl.slices, pl.slots, P.blk_run, round0_d, flag);
    e = cudaMemsetAsync(P.c_part, 0, (size_t)P.n_vblk * P.nc * (P.fp32 ? kPartF * 4 : kPartD * 8), s);
    if (e == cudaSuccess)
        e = P.fp32 ? cudaMemsetAsync(P.r_pt16, 0xff, 2 * (size_t)pl.slots, s)
                   : cudaMemsetAsync(P.r_pt, 0xff, 4 * (size_t)pl.slots, s);
    if (e != cudaSuccess) return e;
    run_slices_kernel<<<(unsigned)nblk, 256, 0, s>>>(P, sorted, cut, round0_d, pl.parts, base_d, flag);
    fill_runs_kernel<<<grid_for(P.n), kBlock, 0, s>>>(P, ord, run, run_ptr, base_d, pl.parts, sp_bl, key, flag);
    if (!P.fp32) slot_runs_kernel<<<grid_for(P.nslots), kBlock, 0, s>>>(P, key, flag);
    return cudaGetLastError();
}

}  // namespace mba

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
// G is one number for most slices (lg in build_own).  A slice whose first (longest) run
// would take more than kRunRounds rounds takes more lanes per run, up to a whole
// warp: a camera that sees far more points than the others would otherwise pad
// its 32 / G - 1 neighbours to its own length and keep one warp busy long after
// the others.  600 cameras, 500k observations, 5 % of them in one camera:
// see own_cameras for the times.
#include <algorithm>
#include <vector>

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
                                 const int2 *__restrict__ sp_bl) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < P.n; t += (int64_t)gridDim.x * blockDim.x) {
        const int s = ord[t], r = run[t], k = (int)(t - run_ptr[r]);
        const int part = k % parts, kk = k / parts;
        const int2 at = base[(int64_t)r * parts + part];  // first slot, log2 G
        const int slot = at.x + 32 * (kk >> at.y) + (kk & ((1 << at.y) - 1));
        P.cm2r[s] = slot;
        const int sp = P.cm_sp[s];
        if (P.r_pt16) P.r_pt16[slot] = (uint16_t)sp_bl[sp].y;
        else P.r_pt[slot] = sp;
    }
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
                                                         int2 *__restrict__ base) {
    __shared__ int s_start[kBlockSlices];
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

}  // namespace

// The block-owned product is used where the camera rows leave room in shared
// memory and where the runs are long enough that the partial sums (written and
// read once per product) cost less than the gathers of b they replace: at least
// kMinRun observations on average, or partial sums of a few MB, which stay in L2.
constexpr double kMinRun = 4.0;
constexpr int64_t kSmallParts = 16 << 20;
bool own_wanted(const Prob &P, int grid) {
    const int64_t rows = (int64_t)P.nc * (P.fp32 ? kRowS * 4 : kRowD * 8);
    const int64_t parts = (int64_t)grid * P.nc * (P.fp32 ? kPartF * 4 : kPartD * 8);
    return rows + 40 * 1024 <= kOwnSmem && ((double)P.n >= kMinRun * (double)grid * P.nc || parts <= kSmallParts);
}

size_t own_tmp_bytes(const Prob &P, int64_t nblk) {
    return al256(8 * (size_t)P.np) + 3 * al256(4 * (size_t)P.n) + 2 * al256(4 * ((size_t)nblk * P.nc + 2)) +
           3 * al256(8 * (size_t)nblk * P.nc * (P.nc < 128 ? kMaxParts : 1)) + 2 * al256(16 * (size_t)nblk) + 4 * (size_t)exclusive_scan_tmp_ints(nblk * P.nc + 2) + 1024 +
           stable_sort_tmp_bytes(P.n, (int32_t)nblk + 1);
}

// Builds the run layout; allocates its arrays (OwnArrays, freed with the problem).
cudaError_t build_own(Prob &P, void *tmp, size_t tmp_bytes, void **pool, size_t *pool_bytes, cudaStream_t s) {
    const int64_t nblk = P.nblk, nruns = nblk * P.nc;
    if (tmp_bytes < own_tmp_bytes(P, nblk)) return cudaErrorInvalidValue;
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

    point_blocks_kernel<<<grid_for(P.n_slices), kBlock, 0, s>>>(P.slice, P.n_slices, P.nblk, sp_bl);
    obs_block_kernel<<<grid_for(P.n), kBlock, 0, s>>>(P.cm_sp, sp_bl, P.n, key);
    cudaError_t e = stable_sort_by_key(key, P.n, (int32_t)nblk, ord, nullptr, t, sort_bytes, s);
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(count, 0, 4 * ((size_t)nruns + 2), s);
    if (e != cudaSuccess) return e;
    run_key_kernel<<<grid_for(P.n), kBlock, 0, s>>>(ord, key, P.cam_ptr, P.nc, P.n, run, count);
    e = exclusive_scan_i32(count, run_ptr, nruns + 1, scan_tmp, s);
    if (e != cudaSuccess) return e;

    // few cameras: split their runs until a block has work for a few hundred lanes
    const double mean = (double)P.n / (double)nruns;
    int parts = 1;
    while (parts < kMaxParts && (int64_t)P.nc * parts < 128 && mean / parts > 16.0) parts *= 2;
    P.n_vblk = (int32_t)(nblk * parts);
    // shared memory: camera rows, b of a block's points (FP32) or the owner's
    // group sums over them, dot products
    // lanes per run, no more than the mean run fills.  FP32: a few rounds of the
    // CTA's warps.  FP64: two where the runs then still fit its 512 lanes twice,
    // more only to give the FP64 pipe a handful of warps (the reduction of nine
    // values over a run's lanes takes a third of a round's pipe time per level)
    int lg = 0;
    const int64_t items_blk = (int64_t)P.nc * parts;
    while (lg < 3 && (2 << lg) <= mean / parts &&
           (items_blk << (lg + 1)) <= (P.fp32 ? 4096 : (lg == 0 ? 1024 : 256)))
        ++lg;

    // sort on the device, offsets of the blocks here, then the slices on the device:
    // laid out on the host (counts read back, tables of 32 lanes a slice sent), the
    // creation of 1.0M points and 5.0M observations took 8.6 ms instead of 3.5, of
    // 50k points and 250k observations 1.77 instead of 1.01
    int m = 2;
    while (m < items_blk) m *= 2;
    if (m > 4096) return cudaErrorInvalidValue;
    sort_runs_kernel<<<(unsigned)nblk, 512, 8 * (size_t)m, s>>>(count, P.nc, parts, lg, m, sorted, cut, info_d);
    std::vector<int4> info((size_t)nblk);
    e = cudaMemcpyAsync(info.data(), info_d, 16 * (size_t)nblk, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return e;
    std::vector<int4> blk((size_t)nblk);
    std::vector<int32_t> round0((size_t)nblk);
    int64_t slots = 0;
    int32_t nrs = 0;
    for (int64_t b = 0; b < nblk; ++b) {
        blk[b] = make_int4(nrs, nrs + info[b].z, nrs + info[b].x, 0);
        nrs += info[b].x;
        if (info[b].z > 0) P.long_runs = 1;
        round0[b] = (int32_t)(slots / 32);
        slots += 32 * (int64_t)info[b].y;
        if (slots > 2000000000ll) return cudaErrorInvalidValue;
    }
    P.rslot_cap = (slots + 31) / 32 * 32;

    // arrays
    const bool loss = P.loss != MBA_LOSS_NONE;
    const size_t ns = (size_t)P.rslot_cap, part_vals = (size_t)P.n_vblk * P.nc * (P.fp32 ? kPartF : kPartD);
    for (int pass = 0; pass < 2; ++pass) {
        char *q = (char *)*pool;
        size_t off = 0;
        auto arr = [&](size_t bytes) -> void * {
            void *p = pass ? q + off : nullptr;
            off += al256(bytes ? bytes : 1);
            return p;
        };
        P.rslice = (int2 *)arr(8 * (size_t)nrs);
        P.rlane = (int2 *)arr(32 * 8 * (size_t)nrs);
        P.blk_run = (int4 *)arr(16 * blk.size());
        P.cm2r = (int32_t *)arr(4 * (size_t)P.n);
        P.c_part = arr(part_vals * (P.fp32 ? 4 : 8));
        if (P.fp32) {
            P.r_rx = (float4 *)arr(16 * ns);
            P.r_pt16 = (uint16_t *)arr(2 * ns);
            P.r_w = loss ? (float *)arr(4 * ns) : nullptr;
        } else {
            P.r_pt = (int32_t *)arr(4 * ns);
            P.r_hg = (double2 *)arr(80 * ns);
        }
        if (pass == 0) {
            *pool_bytes = off;
            if (over_memory_limit(off)) return cudaErrorMemoryAllocation;
            e = cudaMalloc(pool, off);
            if (e != cudaSuccess) return e;
        }
    }
    e = cudaMemcpyAsync(P.blk_run, blk.data(), 16 * blk.size(), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(round0_d, round0.data(), 4 * round0.size(), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(P.c_part, 0, part_vals * (P.fp32 ? 4 : 8), s);
    if (e == cudaSuccess)
        e = P.fp32 ? cudaMemsetAsync(P.r_pt16, 0xff, 2 * ns, s) : cudaMemsetAsync(P.r_pt, 0xff, 4 * ns, s);
    if (e != cudaSuccess) return e;
    run_slices_kernel<<<(unsigned)nblk, 256, 0, s>>>(P, sorted, cut, round0_d, parts, base_d);
    fill_runs_kernel<<<grid_for(P.n), kBlock, 0, s>>>(P, ord, run, run_ptr, base_d, parts, sp_bl);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);  // the host vectors go out of scope
    return e;
}

}  // namespace mba

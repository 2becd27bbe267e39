// sell.cu -- the sliced point order of the point-side passes.
//
// Points are sorted by decreasing track length (stable) and cut into slices of
// one warp each.  A slice holds 32 / G points of one length, G lanes per point
// and K = ceil(length / G) rounds; the observation k of a point sits in round
// k / G at lane k mod G of the point's group, i.e. at slot
//   base + 32 (k / G) + G (point in slice) + k mod G.
// Every stream over the slots is then coalesced, a point's sums stay in its
// lanes' registers (log2 G shuffles join them) and slices of equal length keep a
// warp's lanes in step.  G is 1 where the slices alone fill the GPU's warps.
// Smaller problems take more lanes per point, long tracks take enough that a
// slice has at most kMaxRounds rounds (32 lanes at most), and a class of few
// points takes as many as fill its slice.
#include <vector>

#include "mba_internal.cuh"

namespace mba {

namespace {

constexpr int kMaxRounds = 16;
// warps that fill the GPU: one wave of the FP32 PCG kernel; in FP64 one and a half
// waves of its 16 warps per SM (more lanes per point repeat the point's C~^-1
// product and add reductions, which the FP64 pipe pays for)
constexpr int kFillWarps = 152 * 32, kFillWarps64 = 152 * 24;

// lanes per point of every class in a problem of np points: a power of two,
// as many (up to 8) as leave no more slices than that many warps
int base_lg(int32_t np, bool fp32) {
    int lg = 0;
    while (lg < 3 && ((int64_t)np << (lg + 1)) <= 32ll * (fp32 ? kFillWarps : kFillWarps64)) ++lg;
    return lg;
}

int class_lg(int len, int64_t count, int lg0) {
    int full = 0;  // 2^full >= len
    while (full < 5 && (1 << full) < len) ++full;
    int lg = lg0 < full ? lg0 : full;
    while (lg < full && ((len + (1 << lg) - 1) >> lg) > kMaxRounds) ++lg;
    while (lg < full && (count << lg) < 32) ++lg;
    return lg;
}

__global__ void length_key_kernel(const int32_t *__restrict__ pt_ptr, int32_t np, int32_t longest, int32_t *key) {
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < np; j += gridDim.x * blockDim.x)
        key[j] = longest - (pt_ptr[j + 1] - pt_ptr[j]);
}

__global__ void invert_kernel(const int32_t *__restrict__ perm, int32_t n, int32_t *inv) {
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) inv[perm[j]] = j;
}

// cls[length]: (first sorted point, first slot, log2 G, K)
__global__ void fill_slots_kernel(Prob P, const int32_t *__restrict__ pt_sp, const int4 *__restrict__ cls) {
    for (int64_t o = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; o < P.n; o += (int64_t)gridDim.x * blockDim.x) {
        const int pt = P.pm_pt[o], b = P.pt_ptr[pt], k = (int)(o - b);
        const int4 c = cls[P.pt_ptr[pt + 1] - b];
        const int q = pt_sp[pt] - c.x, per = 32 >> c.z, sl = q / per;
        const int64_t slot =
            c.y + (int64_t)sl * 32 * c.w + 32 * (k >> c.z) + ((q - sl * per) << c.z) + (k & ((1 << c.z) - 1));
        P.sl_cam[slot] = P.pm_cam[o];
        const double2 uv = P.pm_uv[o];
        P.sl_uv[slot] = uv;
        if (P.sl2r) P.sl2r[slot] = P.pm_orig[o];  // until build_own
        if (P.sl_uv32) P.sl_uv32[slot] = make_float2((float)uv.x, (float)uv.y);
    }
}

__global__ void cm_sorted_kernel(const int32_t *__restrict__ cm_pt, const int32_t *__restrict__ pt_sp, int64_t n,
                                 int32_t *__restrict__ cm_sp) {
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n; s += (int64_t)gridDim.x * blockDim.x)
        cm_sp[s] = pt_sp[cm_pt[s]];
}

inline unsigned grid_for(int64_t n) {
    int64_t g = (n + kBlock - 1) / kBlock;
    if (g > 152 * 16) g = 152 * 16;
    return (unsigned)(g < 1 ? 1 : g);
}

// distinct track lengths a problem can have: at most kMaxTrack, and their sum is at most n
int64_t class_bound(int64_t n) {
    int64_t c = 1;
    while (c < kMaxTrack && c * (c + 1) / 2 <= n) ++c;
    return c;
}

}  // namespace

// Slots: a class's lanes are more than half used (G < 2 length), or within
// 1/8 of full where G only bounds the rounds; each class may leave one slice
// of at most 32 kMaxRounds slots (32 x 32 for the longest tracks) partly empty.
int64_t sell_slot_bound(int64_t n, int32_t np) {
    return (base_lg(np, true) == 0 ? n + n / 8 : 2 * n) + class_bound(n) * 32 * kMaxRounds + 1024;
}
int64_t sell_slice_bound(int64_t n, int32_t np) { return sell_slot_bound(n, np) / 32 + 1; }

// Points of a block at most, slices dealt to nblk blocks in turn.  Full slices hold
// more points the shorter their tracks are, so that a block's slices hold at most as
// many as an equal share and one slice (32) more.  A class's last slice may be
// partly empty, and a class of few points has its own number of lanes: up to 62
// points per class that other blocks do not have.
int64_t sell_block_points(int64_t n, int32_t np, int64_t nblk) {
    return (np / nblk + 33 + 62 * class_bound(n) / nblk + 31) / 32 * 32;
}

// Scratch (tmp): the sort's, then keys and inverse (np each), the class offsets
// (kMaxTrack + 2) and the class table (kMaxTrack + 1 int4).
size_t sell_tmp_bytes(int32_t np) {
    return stable_sort_tmp_bytes(np, kMaxTrack + 1) + 2 * (((size_t)np * 4 + 255) & ~size_t(255)) +
           4 * (kMaxTrack + 64) + 16 * (kMaxTrack + 64);
}

cudaError_t build_slices(Prob &P, int grid, int max_track, void *tmp, size_t tmp_bytes, cudaStream_t s) {
    if (tmp_bytes < sell_tmp_bytes(P.np)) return cudaErrorInvalidValue;
    const size_t sort_bytes = stable_sort_tmp_bytes(P.np, kMaxTrack + 1);
    const size_t row = ((size_t)P.np * 4 + 255) & ~size_t(255);
    int32_t *key = (int32_t *)((char *)tmp + sort_bytes);
    int32_t *pt_sp = (int32_t *)((char *)key + row);
    int4 *cls_d = (int4 *)((char *)pt_sp + row);
    int32_t *off_d = (int32_t *)(cls_d + kMaxTrack + 64);

    length_key_kernel<<<grid_for(P.np), kBlock, 0, s>>>(P.pt_ptr, P.np, max_track, key);
    cudaError_t e = stable_sort_by_key(key, P.np, max_track + 1, P.sp_pt, off_d, tmp, sort_bytes, s);
    if (e != cudaSuccess) return e;
    invert_kernel<<<grid_for(P.np), kBlock, 0, s>>>(P.sp_pt, P.np, pt_sp);
    std::vector<int32_t> off((size_t)max_track + 2);
    e = cudaMemcpyAsync(off.data(), off_d, 4 * off.size(), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return e;

    const int lg0 = base_lg(P.np, P.fp32 != 0);
    std::vector<int4> slices, cls((size_t)max_track + 1, make_int4(0, 0, 0, 0));
    int64_t slots = 0;
    for (int k = 0; k < max_track; ++k) {  // key k: points of length max_track - k
        const int len = max_track - k;
        const int32_t first = off[k], count = off[k + 1] - off[k];
        if (count == 0) continue;
        const int lg = class_lg(len, count, lg0), K = (len + (1 << lg) - 1) >> lg, per = 32 >> lg;
        if (slots + ((int64_t)count / per + 1) * 32 * K > P.slot_cap) return cudaErrorInvalidValue;
        cls[len] = make_int4(first, (int32_t)slots, lg, K);
        for (int32_t p = 0; p < count; p += per) {
            slices.push_back(make_int4(first + p, count - p < per ? count - p : per, (int32_t)slots, K | (lg << 16)));
            slots += 32 * K;
        }
    }
    P.n_slices = (int32_t)slices.size();
    P.nslots = slots;
    // the blocks of the block-owned product: slice i belongs to block i mod nblk, a
    // block's points are numbered in slice order; as few blocks per CTA as let b of
    // a block's points fit in shared memory beside the camera rows (FP32)
    if (P.own) {
        std::vector<int32_t> used;
        P.own = 0;
        for (int m = 1; m <= kMaxBlocks && !P.own; ++m) {
            used.assign((size_t)grid * m, 0);
            for (size_t i = 0; i < slices.size(); ++i) used[i % used.size()] += slices[i].y;
            int32_t most = 0;
            for (int32_t u : used) most = u > most ? u : most;
            P.own = own_fits(P, grid, m, (most + 31) / 32 * 32) ? 1 : 0;
        }
    }
    if (P.own) {
        std::vector<int32_t> used;
        used.assign((size_t)P.nblk, 0);
        for (size_t i = 0; i < slices.size(); ++i) {
            const int32_t count = slices[i].y;
            slices[i].y |= used[i % P.nblk] << 8;
            used[i % P.nblk] += count;
        }
    }
    e = cudaMemcpyAsync(P.slice, slices.data(), sizeof(int4) * slices.size(), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(cls_d, cls.data(), sizeof(int4) * cls.size(), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(P.sl_cam, 0xff, 4 * (size_t)slots, s);
    if (e != cudaSuccess) return e;
    fill_slots_kernel<<<grid_for(P.n), kBlock, 0, s>>>(P, pt_sp, cls_d);
    cm_sorted_kernel<<<grid_for(P.n), kBlock, 0, s>>>(P.cm_pt, pt_sp, P.n, P.cm_sp);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);  // the host vectors go out of scope
    return e;
}

}  // namespace mba

// Update step of SIVF (Algorithm 5, Section 4.2) on sm_103a, plus the
// set-up kernels (CSR validation, seed centroids).
//
// Pipeline for iteration r (lambda = lambda^[r] from the assignment), in the
// default dense form:
//  u1  per-cluster member counts from the labels.
//  u2  an int64 fixed-point accumulator row of the instance's D terms per
//      cluster, kept across iterations: every object whose label changed
//      moves its q(x) = ceil(x 2^shift) values from its old cluster's row to
//      the new one with integer atomics (k_acc_scatter). Integer sums are
//      exact, so each entry is the sum over the current members whatever the
//      history, and the result is deterministic.
//  u3  pass 1 (k_acc_rows1): new row sizes, ||s_j|| from the exact 128-bit
//      sum of the squared integer sums (one rounding to FP64), and the
//      objective pieces <s_j, mu_j^[r-1]> the same way; pass 2 (k_acc_rows2): the row
//      compacted in ascending term order, u = S (2^-shift / ||s_j||) in FP32.
//      Dividing by |C_j| first cancels exactly and is skipped.
//  u4  invariant and empty clusters keep their centroid row (copied).
//  u5  the scan structures of the structured inverted file, counted per term
//      and part (k_if_count) and written in one scatter pass over the
//      centroid entries (k_scan_fill): the scan order (moving
//      clusters first), the dense head rows and the sparse scan copy, whose
//      lists hold the moving centroids first and the invariant ones after
//      (Algorithm 5, lines 1-14 and 21-30). The canonical sorted file (ids
//      ascending in each part) is built by a stable radix sort only when a
//      getter asks for it.
// The sort form replaces u1-u3 by a stable radix sort of (label, object id),
// an expansion of the recomputed clusters' members' (term, value) pairs sorted
// by (cluster rank, term) and reduced sequentially in FP64, in ascending
// object id, the order of the plain definition (Algorithm 5, lines 17-20).
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>

#include "bf16_rows.cuh"
#include "sivf_internal.cuh"

namespace sivf {
namespace {

constexpr int TPB = 256;

inline unsigned blocks_for(int64_t n, int tpb = TPB) {
    int64_t b = (n + tpb - 1) / tpb;
    if (b < 1) b = 1;
    if (b > 0x7FFFFFFF) b = 0x7FFFFFFF;
    return (unsigned)b;
}

// Grid of a grid-stride kernel: enough blocks to fill the GPU a few times
// over, not one per element, so that a launch bounded by a capacity (with the
// live count on the device) costs no empty blocks.
constexpr unsigned GS_MAX_BLOCKS = 4096;
inline unsigned blocks_gs(int64_t n, int tpb = TPB) {
    const unsigned b = blocks_for(n, tpb);
    return b < GS_MAX_BLOCKS ? b : GS_MAX_BLOCKS;
}

// ---------------- validation and set-up ----------------

// bad bits: 1 row_ptr, 2 idx range/order, 4 value, 8 norm
__global__ void k_validate(int64_t N, int32_t D, int64_t nnz, const int64_t *row_ptr, const int32_t *idx,
                           const float *val, float *sumv, int *bad) {
    const int lane = threadIdx.x & 31;
    const int64_t wid = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i = wid; i < N; i += nw) {
        const int64_t b = row_ptr[i], e = row_ptr[i + 1];
        int flags = 0;
        if (b < 0 || e < b || e > nnz) flags |= 1;
        double ss = 0.0, sv = 0.0;
        if (!(flags & 1)) {
            for (int64_t h = b + lane; h < e; h += 32) {
                const int t = idx[h];
                const float v = val[h];
                if (t < 0 || t >= D) flags |= 2;
                if (h > b && idx[h - 1] >= t) flags |= 2;
                if (!(v > 0.0f) || !isfinite(v)) flags |= 4;
                ss += (double)v * (double)v;
                sv += (double)v;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            ss += __shfl_xor_sync(0xffffffffu, ss, o);
            sv += __shfl_xor_sync(0xffffffffu, sv, o);
            flags |= __shfl_xor_sync(0xffffffffu, flags, o);
        }
        if (lane == 0) {
            if (!(flags & 1) && e > b && fabs(sqrt(ss) - 1.0) > 1e-4) flags |= 8;
            sumv[i] = (float)(sv * (1.0 + 1e-6));  // rounded up: the bound needs S >= sum v
            if (flags) atomicOr(bad, flags);
        }
    }
}

// Live entries of buffers that hold cap: none when the count says more (the
// rows were then not written; the count's own kernel reports it).
__device__ __forceinline__ int64_t live_entries(const int64_t *n_dev, int64_t cap) {
    const int64_t n = *n_dev;
    return n <= cap ? n : 0;
}

// State before the first assignment: no labels, no own scores, nothing added
// to the accumulator, every cluster moving, no sums behind the centroids; and
// the sizes of the seed rows. A row whose offsets are not in the CSR any more
// (the borrowed arrays changed) is given a size that no buffer holds.
__global__ void k_reset(int64_t N, int32_t k, int32_t *labels, int32_t *labels_prev, uint32_t *own, int32_t *acc_lab,
                        uint8_t *lam, uint8_t *lam_prev, uint8_t *moving, double *snorm, const int32_t *init_ids,
                        const int64_t *row_ptr, int64_t nnz, int64_t cap, int64_t *sz, DevCounters *ctr) {
    const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, st = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = g; i < N; i += st) {
        labels[i] = -1;
        labels_prev[i] = -1;
        own[i] = OWN_INVALID;
        if (acc_lab) acc_lab[i] = -1;
    }
    for (int64_t j = g; j < k; j += st) {
        lam[j] = 0;
        lam_prev[j] = 0;
        moving[j] = 1;
        snorm[j] = 0.0;
        const int64_t d = init_ids[j], b = row_ptr[d], e = row_ptr[d + 1];
        sz[j] = b >= 0 && b <= e && e <= nnz ? e - b : cap + 1;
    }
    if (g == 0) *ctr = DevCounters{};
}

// The seed rows, one warp each; their total is left in the counters. Rows that
// the buffers do not hold are not written, and reported.
__global__ void k_seed_rows(int32_t k, const int32_t *init_ids, const int64_t *row_ptr, const int32_t *idx,
                            const float *val, const int64_t *coff, int64_t cap, int32_t *cterm, float *cval,
                            int32_t *cclu, DevCounters *ctr) {
    const int lane = threadIdx.x & 31;
    const int64_t wid = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (wid >= k) return;
    if (coff[k] > cap) {
        if (wid == 0 && lane == 0) ctr->error = ERR_CAPACITY;
        return;
    }
    const int j = (int)wid;
    const int64_t d = init_ids[j];
    const int64_t b = row_ptr[d], e = row_ptr[d + 1], o = coff[j];
    for (int64_t h = b + lane; h < e; h += 32) {
        cterm[o + (h - b)] = idx[h];
        cval[o + (h - b)] = val[h];
        cclu[o + (h - b)] = j;
    }
    if (wid == 0 && lane == 0) ctr->c_nnz = coff[k];
}

// Replace a^[r] by src. lambda^[r] is recomputed against a^[r-1] (every
// cluster moving before the second assignment), whose centroids the stored own
// scores belong to. Where the centroids have been rebuilt since (rebuilt = 1:
// they belong to the labels replaced here, not to a^[r-1]), a cluster that loses
// or gains a member against those labels is moving as well: its row would
// otherwise stay that of the replaced labels. An object whose label changes
// loses its stored own-cluster score.
__global__ void k_set_labels(int64_t N, const int32_t *src, int32_t *labels, const int32_t *labels_prev, int rebuilt,
                             uint32_t *own, uint8_t *moving) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t a = src[i], old = labels[i], prev = labels_prev[i];
        if (old != a) {
            labels[i] = a;
            own[i] = OWN_INVALID;
        }
        const bool moved = rebuilt && old != a;
        if (a != prev || moved) moving[a] = 1;
        if (a != prev && prev >= 0) moving[prev] = 1;
        if (moved && old >= 0 && old != prev) moving[old] = 1;  // a store per object and cluster, not two
    }
}

__global__ void k_check_labels(int64_t N, int32_t k, const int32_t *src, int *bad) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t a = src[i];
        if (a < 0 || a >= k) atomicOr(bad, 1);
    }
}

// ---------------- u1: group objects by label ----------------

__global__ void k_label_keys(int64_t N, const int32_t *labels, uint32_t *keys, uint32_t *vals, int64_t *cnt) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t a = labels[i];
        keys[i] = (uint32_t)a;
        vals[i] = (uint32_t)i;
        atomicAdd(reinterpret_cast<unsigned long long *>(cnt + a), 1ull);
    }
}

// recompute flag: moving (lambda = 0) and non-empty
__global__ void k_recompute_flags(int32_t k, const uint8_t *lam, const int64_t *cnt, int64_t *flag) {
    int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < k) flag[j] = (lam[j] == 0 && cnt[j] > 0) ? 1 : 0;
}

// ---------------- u2: cluster sums ----------------

__global__ void k_member_tuples(int64_t N, const uint32_t *perm, const int32_t *labels, const int64_t *flag,
                                const int64_t *row_ptr, int64_t *tc) {
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < N; p += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = perm[p];
        tc[p] = flag[labels[i]] ? row_ptr[i + 1] - row_ptr[i] : 0;
    }
}

// One warp per member (in cluster, then object order): its (term, value)
// pairs become tuples t = toff[p] + h with the cluster's rank.
__global__ void k_expand(int64_t N, const uint32_t *perm, const int32_t *labels, const int64_t *rrank,
                         const int64_t *tc, const int64_t *toff, const int64_t *row_ptr, const int32_t *idx,
                         const float *val, uint32_t *kterm, uint32_t *vtup, uint32_t *tterm, float *tval,
                         uint32_t *trank) {
    const int lane = threadIdx.x & 31;
    const int64_t wid = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t p = wid; p < N; p += nw) {
        if (tc[p] == 0) continue;
        const int64_t i = perm[p];
        const uint32_t rk = (uint32_t)rrank[labels[i]];
        const int64_t b = row_ptr[i], e = row_ptr[i + 1], o = toff[p];
        for (int64_t h = b + lane; h < e; h += 32) {
            const uint32_t t = (uint32_t)(o + (h - b));
            kterm[t] = (uint32_t)idx[h];
            vtup[t] = t;
            tterm[t] = (uint32_t)idx[h];
            tval[t] = val[h];
            trank[t] = rk;
        }
    }
}

// One 32-bit key per tuple when it fits: (cluster rank, instance-local term),
// with the value's bits as the payload.
__global__ void k_expand_packed(int64_t N, const uint32_t *perm, const int32_t *labels, const int64_t *rrank,
                                const int64_t *tc, const int64_t *toff, const int64_t *row_ptr, const int32_t *idx,
                                const float *val, const int32_t *clu_doff, int bits_tl, uint32_t *key,
                                uint32_t *vbits) {
    const int lane = threadIdx.x & 31;
    const int64_t wid = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t p = wid; p < N; p += nw) {
        if (tc[p] == 0) continue;
        const int64_t i = perm[p];
        const int32_t j = labels[i];
        const uint32_t hi = (uint32_t)rrank[j] << bits_tl;
        const int32_t doff = clu_doff[j];
        const int64_t b = row_ptr[i], e = row_ptr[i + 1], o = toff[p];
        for (int64_t h = b + lane; h < e; h += 32) {
            key[o + (h - b)] = hi | (uint32_t)(idx[h] - doff);
            vbits[o + (h - b)] = __float_as_uint(val[h]);
        }
    }
}

// packed keys back to (rank << 32 | global term) and float values
__global__ void k_unpack(int64_t nmax, const int64_t *n_dev, const uint32_t *key, const uint32_t *vbits,
                         int bits_tl, const int32_t *rank2clu, const int32_t *clu_doff, unsigned long long *key64,
                         float *sval) {
    const int64_t n = *n_dev;
    const uint32_t tmask = (1u << bits_tl) - 1u;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t kk = key[q];
        const uint32_t r = kk >> bits_tl;
        const uint32_t t = (kk & tmask) + (uint32_t)clu_doff[rank2clu[r]];
        key64[q] = ((unsigned long long)r << 32) | (unsigned long long)t;
        sval[q] = __uint_as_float(vbits[q]);
    }
}

// cluster of each rank (inverse of rrank on the recomputed clusters)
__global__ void k_rank2clu(int32_t k, const int64_t *flag, const int64_t *rrank, int32_t *rank2clu) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < k && flag[j]) rank2clu[rrank[j]] = j;
}

// after the stable sort by term: rank keys for the stable sort by rank
__global__ void k_rank_keys(int64_t nmax, const int64_t *n_dev, const uint32_t *vtup_sorted, const uint32_t *trank,
                            uint32_t *krank, uint32_t *vrank) {
    const int64_t n = *n_dev;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t t = vtup_sorted[q];
        krank[q] = trank[t];
        vrank[q] = t;
    }
}

// tuples in (rank, term, object) order: composite key and value
__global__ void k_compose(int64_t nmax, const int64_t *n_dev, const uint32_t *krank, const uint32_t *vtup,
                          const uint32_t *tterm, const float *tval, unsigned long long *key64, float *sval) {
    const int64_t n = *n_dev;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t t = vtup[q];
        key64[q] = ((unsigned long long)krank[q] << 32) | (unsigned long long)tterm[t];
        sval[q] = tval[t];
    }
}

__global__ void k_heads(int64_t nmax, const int64_t *n_dev, const unsigned long long *key, uint32_t *head) {
    const int64_t n = *n_dev;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
        head[e] = (e == 0 || key[e] != key[e - 1]) ? 1u : 0u;
}

// position of each run of equal keys: hpos[u] = first element of run u
__global__ void k_head_pos(int64_t nmax, const int64_t *n_dev, const uint32_t *head, const uint32_t *uidx,
                           uint32_t *hpos) {
    const int64_t n = *n_dev;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
        if (head[e]) hpos[uidx[e]] = (uint32_t)e;
}

// FP64 sum of each run of equal keys (a (cluster, term) pair), in two passes
// with a fixed order (reproducible bit for bit):
//  1. each warp takes 32 consecutive elements and forms, by a segmented
//     inclusive scan over the lanes, the sum of every run piece inside those
//     32 elements, stored at the piece's last element;
//  2. one thread per run adds its pieces in ascending position.
__global__ void k_seg_pieces(int64_t nmax, const int64_t *n_dev, const unsigned long long *keys, const float *vals,
                             double *part) {
    const int64_t n = *n_dev;
    const int lane = threadIdx.x & 31;
    const int64_t wid = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t base = wid * 32; base < n; base += nw * 32) {
        const int64_t e = base + lane;
        const bool valid = e < n;
        const unsigned long long key = valid ? keys[e] : ~0ull;
        double x = valid ? (double)vals[e] : 0.0;
        const unsigned long long prev = __shfl_up_sync(0xffffffffu, key, 1);
        bool flag = lane == 0 || prev != key;  // a piece starts here
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double y = __shfl_up_sync(0xffffffffu, x, o);
            const bool f = __shfl_up_sync(0xffffffffu, flag, o);
            if (lane >= o && !flag) x = y + x;
            if (lane >= o) flag = flag || f;
        }
        const unsigned long long next = __shfl_down_sync(0xffffffffu, key, 1);
        const bool last = valid && (lane == 31 || e == n - 1 || next != key);
        if (last) part[e] = x;
    }
}

// Runs arrive sorted by (cluster rank, term): the first and the last run of
// each cluster record where its unique entries begin and end (no atomics).
__global__ void k_seg_runs(int64_t nmax, const int64_t *n_dev, const uint32_t *U_dev,
                           const unsigned long long *keys, const uint32_t *hpos, const double *part, int32_t *uterm,
                           double *usum, int64_t *ubeg, int64_t *uend) {
    const int64_t n = *n_dev;
    const int64_t U = n > 0 ? (int64_t)*U_dev : 0;
    for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < U; u += (int64_t)gridDim.x * blockDim.x) {
        const int64_t b = hpos[u];
        const int64_t e = (u + 1 < U) ? (int64_t)hpos[u + 1] : n;
        double acc = 0.0;
        for (int64_t c = b >> 5; c <= ((e - 1) >> 5); ++c) {
            const int64_t end = ((c + 1) << 5) < e ? ((c + 1) << 5) : e;
            acc += part[end - 1];
        }
        const unsigned long long key = keys[b];
        const uint32_t r = (uint32_t)(key >> 32);
        uterm[u] = (int32_t)(key & 0xFFFFFFFFull);
        usum[u] = acc;
        if (u == 0 || (uint32_t)(keys[hpos[u - 1]] >> 32) != r) ubeg[r] = u;
        if (u + 1 == U || (uint32_t)(keys[e] >> 32) != r) uend[r] = u + 1;
    }
}

// ---------------- u3 / u4: new centroid rows ----------------

__global__ void k_new_sizes(int32_t k, const int64_t *flag, const int64_t *rrank, const int64_t *supoff,
                            const int64_t *supend, const int64_t *coff_old, int64_t *sz) {
    int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < k) sz[j] = flag[j] ? supend[rrank[j]] - supoff[rrank[j]] : coff_old[j + 1] - coff_old[j];
}

// One CTA (WR_THREADS) per cluster. Recomputed clusters: ||s|| in FP64 with
// strided per-thread sums and a fixed tree, u = s / ||s|| as FP32, and
// <s_j, mu_j^[r-1]> by binary search of each term in the previous row.
// Other clusters copy their previous row.
constexpr int WR_THREADS = 256;

__device__ __forceinline__ double block_sum_fixed(double x, double *sh) {
    sh[threadIdx.x] = x;
    __syncthreads();
    for (int s = WR_THREADS / 2; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
        __syncthreads();
    }
    const double r = sh[0];
    __syncthreads();
    return r;
}

__global__ void __launch_bounds__(WR_THREADS) k_write_rows(
    int32_t k, const int64_t *flag, const int64_t *rrank, const int64_t *supoff, const int64_t *supend,
    const int32_t *uterm, const double *usum, const int64_t *cnt, const int64_t *coff_old, const int32_t *cterm_old,
    const float *cval_old, const double *snorm_old, const int64_t *coff_new, int32_t *cterm_new, float *cval_new,
    int32_t *cclu_new, double *snorm_new, double *jA, double *jU, int64_t cap, unsigned long long *error) {
    __shared__ double sh[WR_THREADS];
    const int j = blockIdx.x;
    if (j >= k) return;
    const int64_t o = coff_new[j];
    const int64_t cb = coff_old[j], ce = coff_old[j + 1];
    if (coff_new[k] > cap) {  // more centroid entries than the buffers hold: write nothing, report
        if (j == 0 && threadIdx.x == 0) atomicOr(error, ERR_CAPACITY);
        return;
    }
    if (flag[j]) {
        const int64_t r = rrank[j];
        const int64_t ub = supoff[r], n = supend[r] - supoff[r];
        double ss = 0.0;
        for (int64_t q = threadIdx.x; q < n; q += WR_THREADS) ss += usum[ub + q] * usum[ub + q];
        const double nrm = sqrt(block_sum_fixed(ss, sh));
        double dot = 0.0;
        for (int64_t q = threadIdx.x; q < n; q += WR_THREADS) {
            const int32_t t = uterm[ub + q];
            const double sv = usum[ub + q];
            cterm_new[o + q] = t;
            cval_new[o + q] = (float)(sv / nrm);
            cclu_new[o + q] = j;
            int64_t lo = cb, hi = ce;
            while (lo < hi) {
                const int64_t mid = (lo + hi) >> 1;
                if (cterm_old[mid] < t) lo = mid + 1; else hi = mid;
            }
            if (lo < ce && cterm_old[lo] == t) dot += sv * (double)cval_old[lo];
        }
        dot = block_sum_fixed(dot, sh);
        if (threadIdx.x == 0) {
            snorm_new[j] = nrm;
            jA[j] = dot;
            jU[j] = nrm;
        }
    } else {
        for (int64_t q = cb + threadIdx.x; q < ce; q += WR_THREADS) {
            cterm_new[o + (q - cb)] = cterm_old[q];
            cval_new[o + (q - cb)] = cval_old[q];
            cclu_new[o + (q - cb)] = j;
        }
        if (threadIdx.x == 0) {
            const double sn = cnt[j] > 0 ? snorm_old[j] : 0.0;
            snorm_new[j] = sn;
            jA[j] = sn;  // unchanged members: <s_j, s_j / ||s_j||> = ||s_j||
            jU[j] = sn;
        }
    }
}

// Last kernel of the centroid step. Blocks below n_inst: the objective sums of
// an instance, in a fixed order (per-thread strided partial sums, then a
// tree). The others copy the new rows back over the current ones (fixed
// buffers for graph replay). Block 0 leaves the step's counts. New rows that
// outgrew the buffers were not written: the current ones stay, whole and within
// the buffers, for the file that is built next.
__global__ void __launch_bounds__(1024) k_finish_rows(int32_t k, int64_t cap, int32_t n_inst, const int32_t *inst_k,
                                                      const double *jA, const double *jU, double *out,
                                                      const int64_t *coff_src, const int32_t *term_src,
                                                      const float *val_src, const double *sn_src, int64_t *coff_dst,
                                                      int32_t *term_dst, float *val_dst, double *sn_dst,
                                                      const int64_t *moved, DevCounters *ctr) {
    if ((int)blockIdx.x < n_inst) {
        __shared__ double sa[1024], sb[1024];
        const int m = blockIdx.x;
        const int j0 = inst_k[m], j1 = inst_k[m + 1];
        double x = 0.0, y = 0.0;
        for (int j = j0 + threadIdx.x; j < j1; j += 1024) {
            x += jA[j];
            y += jU[j];
        }
        sa[threadIdx.x] = x;
        sb[threadIdx.x] = y;
        __syncthreads();
        for (int s = 512; s > 0; s >>= 1) {
            if ((int)threadIdx.x < s) {
                sa[threadIdx.x] += sa[threadIdx.x + s];
                sb[threadIdx.x] += sb[threadIdx.x + s];
            }
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            out[2 * m] = sa[0];
            out[2 * m + 1] = sb[0];
            if (m == 0) {
                ctr->moved = *moved;
                ctr->c_nnz = coff_src[k];
            }
        }
        return;
    }
    const int64_t n = coff_src[k];
    if (n > cap) return;
    const int64_t g = (blockIdx.x - n_inst) * (int64_t)blockDim.x + threadIdx.x;
    const int64_t st = (int64_t)(gridDim.x - n_inst) * blockDim.x;
    for (int64_t e = g; e < n; e += st) {
        term_dst[e] = term_src[e];
        val_dst[e] = val_src[e];
    }
    for (int64_t j = g; j <= k; j += st) coff_dst[j] = coff_src[j];
    for (int64_t j = g; j < k; j += st) sn_dst[j] = sn_src[j];
}

// Offsets of the new rows: exclusive sums of sz[0..k) into coff[0..k], one CTA.
__global__ void __launch_bounds__(1024) k_row_offsets(int32_t k, const int64_t *sz, int64_t *coff) {
    constexpr int PER = 4;
    __shared__ int64_t warp_s[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t carry = 0;
    for (int64_t b = 0; b < k; b += 1024 * PER) {
        const int64_t j0 = b + (int64_t)threadIdx.x * PER;
        int64_t v[PER], sum = 0;
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            v[q] = j0 + q < k ? sz[j0 + q] : 0;
            sum += v[q];
        }
        int64_t inc = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        if (lane == 31) warp_s[warp] = inc;
        __syncthreads();
        int64_t w = warp_s[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        const int64_t total = __shfl_sync(0xffffffffu, w, 31);
        const int64_t before = __shfl_sync(0xffffffffu, w, (warp + 31) & 31);
        int64_t at = carry + (warp ? before : 0) + inc - sum;
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            if (j0 + q < k) coff[j0 + q] = at;
            at += v[q];
        }
        carry += total;
        __syncthreads();
    }
    if (threadIdx.x == 0) coff[k] = carry;
}

// ---------------- u2-u4, dense accumulator form ----------------
//
// Cluster sums in fixed point: every member value x contributes
// q(x) = ceil(x * 2^shift) to the cluster's accumulator entry of its term.
// The accumulator is kept across steps and updated incrementally: an object
// whose label differs from the one it was last added under (acc_lab) has its
// q values subtracted from the old cluster and added to the new one, with
// integer atomics. Integer sums do not depend on the order of the adds, so
// every entry equals the sum of q over the cluster's current members exactly,
// whatever the history; it exceeds the exact sum by less than one unit
// 2^-shift per member. The clusters touched are exactly the moving ones; their
// rows are then read in ascending term order.

// Member counts of the labels, and the objects whose label changed since they
// were last added: a changed object's q values move from the old cluster's row
// to the new one's, and every entry added to has its bit set in the occupancy
// map (bits, 32 entries per word; null: no map). A warp looks at `per` (at
// most 32) objects at once and takes the changed ones of them one by one, all
// lanes on an object's entries: one warp per object, changed or not, spent
// most of its warps on finding nothing to do.
__global__ void k_acc_scatter(int64_t N, int per, const int32_t *labels, int32_t *acc_lab, const int64_t *row_ptr,
                              const int32_t *idx, const float *val, const int32_t *clu_doff, const int64_t *acc_off,
                              float fscale, int64_t *acc, uint32_t *bits, const int64_t *bit_off, int64_t *cnt,
                              int64_t *moved) {
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int64_t stride = (((int64_t)gridDim.x * blockDim.x) >> 5) * per;
    long long mv = 0;
    for (int64_t i0 = ((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5) * per; i0 < N; i0 += stride) {
        const int64_t i = i0 + lane;
        const bool valid = lane < per && i < N;
        const int32_t jn = valid ? labels[i] : -1, jo = valid ? acc_lab[i] : -1;
        if (valid) atomicAdd(reinterpret_cast<unsigned long long *>(cnt + jn), 1ull);
        const bool changed = valid && jn != jo;
        int64_t rb = 0, re = 0;
        if (changed) {
            rb = row_ptr[i];
            re = row_ptr[i + 1];
            acc_lab[i] = jn;
            mv += (re - rb) * (jo >= 0 ? 2 : 1);
        }
        for (unsigned todo = __ballot_sync(FULL, changed); todo; todo &= todo - 1) {
            const int src = __ffs(todo) - 1;
            const int32_t n = __shfl_sync(FULL, jn, src), o = __shfl_sync(FULL, jo, src);
            const int64_t b = __shfl_sync(FULL, rb, src), e = __shfl_sync(FULL, re, src);
            const int32_t dn = clu_doff[n];
            unsigned long long *rn = reinterpret_cast<unsigned long long *>(acc + acc_off[n] - dn);
            uint32_t *bn = bits ? bits + bit_off[n] : nullptr;
            unsigned long long *ro =
                o >= 0 ? reinterpret_cast<unsigned long long *>(acc + acc_off[o] - clu_doff[o]) : nullptr;
            for (int64_t h = b + lane; h < e; h += 32) {
                const unsigned long long q = (unsigned long long)__float2ll_ru(val[h] * fscale);
                const int32_t t = idx[h];
                atomicAdd(rn + t, q);
                if (ro) atomicAdd(ro + t, 0ull - q);  // two's complement: subtracts q
                const uint32_t bit = 1u << ((t - dn) & 31);
                if (bn && !(bn[(t - dn) >> 5] & bit)) atomicOr(bn + ((t - dn) >> 5), bit);
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mv += __shfl_xor_sync(FULL, mv, o);
    if (lane == 0 && mv) atomicAdd(reinterpret_cast<unsigned long long *>(moved), (unsigned long long)mv);
}

// Empties the accumulator through its occupancy map, one CTA per cluster:
// only the entries that a member has touched (0.6 % of them at k = 20,000
// over 140,000 terms) are written.
__global__ void k_acc_clear(int32_t k, const int64_t *acc_off, const int64_t *bit_off, int64_t *acc, uint32_t *bits) {
    for (int j = blockIdx.x; j < k; j += gridDim.x) {
        const int64_t wb = bit_off[j], nw = bit_off[j + 1] - wb;
        int64_t *row = acc + acc_off[j];
        for (int64_t w = threadIdx.x; w < nw; w += blockDim.x) {
            uint32_t b = bits[wb + w];
            if (!b) continue;
            bits[wb + w] = 0;
            for (; b; b &= b - 1) row[32 * w + __ffs(b) - 1] = 0;
        }
    }
}

// Whether row j's accumulator entries are read through the occupancy map: the
// row passes below read 16 bytes per lane in sequence otherwise, which is
// cheaper once a word of the map (32 entries, eight sectors) has a few bits.
// Measured per update, whole rows without a map / whole rows beside one / through
// it, ms, at a density of non-zero entries of 0.3 % 3.9 / 2.5 / 0.83, 0.6 % 1.50
// / 1.58 / 0.65, 2.4 % 0.77 / 0.87 / 0.55, 4.2 % 0.59 / 0.66 / 0.47, 6.7 % 0.43 /
// 0.46 / 0.39, 9.5 % 0.72 / 0.83 / 0.71, 11 % 0.34 / 0.37 / 0.34, 18 % 1.26 / 1.47
// / 1.44 (k = 10,000 to 400 over 61,000 to 140,000 terms, a tenth of the labels
// changed). The line is at 1/16, on the near side of where the two are equal,
// by the length of the previous row, or by a third of the members' entries
// (avg_len each) where the row has grown.
__device__ __forceinline__ bool through_map(const uint32_t *bits, int64_t old_len, int64_t members, int64_t avg_len,
                                            int64_t L) {
    return bits && max(old_len, members * avg_len / 3) * 16 <= L;
}

// Bits 0, 2, 4, ... of the result from the low 16 bits of x, the odd ones from
// those of y.
__device__ __forceinline__ uint32_t interleave16(uint32_t x, uint32_t y) {
    auto spread = [](uint32_t v) {
        v &= 0xffffu;
        v = (v | (v << 8)) & 0x00ff00ffu;
        v = (v | (v << 4)) & 0x0f0f0f0fu;
        v = (v | (v << 2)) & 0x33333333u;
        return (v | (v << 1)) & 0x55555555u;
    };
    return spread(x) | (spread(y) << 1);
}

// Words of row j's non-zero bits (entry t in bit t & 31 of word t >> 5), which
// pass 1 leaves for pass 2: the row's part of the occupancy map, or of scratch
// where there is no map (null: of neither).
__device__ __forceinline__ uint32_t *row_words(uint32_t *bits, const int64_t *bit_off, uint32_t *scratch, int64_t base,
                                               int j) {
    if (bits) return bits + bit_off[j];
    return scratch ? scratch + (base >> 5) + j : nullptr;  // rows of L entries lie (L >> 5) + 1 words apart or more
}

__device__ __forceinline__ long long block_sum_ll(long long x, long long *sh) {
    sh[threadIdx.x] = x;
    __syncthreads();
    for (int s = WR_THREADS / 2; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
        __syncthreads();
    }
    const long long r = sh[0];
    __syncthreads();
    return r;
}

// Sum of (hi, lo) 128-bit unsigned values over the block (fixed tree, exact);
// every thread receives the total.
__device__ __forceinline__ void block_sum_u128(unsigned long long &hi, unsigned long long &lo,
                                               unsigned long long (*sh)[WR_THREADS]) {
    sh[0][threadIdx.x] = hi;
    sh[1][threadIdx.x] = lo;
    __syncthreads();
    for (int s = WR_THREADS / 2; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s) {
            const unsigned long long l = sh[1][threadIdx.x] + sh[1][threadIdx.x + s];
            sh[0][threadIdx.x] += sh[0][threadIdx.x + s] + (l < sh[1][threadIdx.x] ? 1ull : 0ull);
            sh[1][threadIdx.x] = l;
        }
        __syncthreads();
    }
    hi = sh[0][0];
    lo = sh[1][0];
    __syncthreads();
}

// Loads in flight per thread in the loops of both row passes: a cluster is one
// CTA's, so a long row (tens of thousands of entries in a corpus of few
// clusters) is read at its latency; with one or two loads in flight such rows
// held up the passes of a batch for 0.26 and 0.15 ms.
constexpr int ILP = 4;

// (hi, lo) += a * b.
__device__ __forceinline__ void add_product(unsigned long long &hi, unsigned long long &lo, unsigned long long a,
                                            unsigned long long b) {
    const unsigned long long p = a * b;
    lo += p;
    hi += __umul64hi(a, b) + (lo < p ? 1ull : 0ull);
}

// x in [2^-40, 2) in units of 2^-63, exactly; 0 for smaller x >= 0, whose bits
// no unit of 2^-63 holds.
__device__ __forceinline__ unsigned long long fixed63(float x) {
    const uint32_t b = __float_as_uint(x), e = b >> 23;
    return e >= 87u ? (unsigned long long)((b & 0x7fffffu) | 0x800000u) << (e - 87u) : 0ull;
}

// Turns of a whole row's loop (ILP * WR_THREADS entry pairs each) after which
// the entries just read are used for the objective's product with the previous
// row, while they are in L2: 8192 entries, 80 MB for the CTAs of the chip. After
// the whole row, those entries came from HBM again: 1.68 against 1.13 GB read at
// 1000 rows of 100,000 entries, 1.38 against 1.31 ms for the update. Half or
// twice the turns make no difference of more than 1 %.
constexpr int DOT_TURNS = 4;
// Previous entries in flight per thread there. The loop waits for a term, then
// for its sum; two in flight took 1.52 ms, also with fewer row loads and spills.
constexpr int DOT_ILP = 4;

// Pass 1, one CTA per cluster: size of the new row, ||s_j|| (the squared
// integer sums added exactly in 128 bits, one rounding to FP64) and
// <s_j, mu_j^[r-1]> over the previous row, whose values are taken in units of
// 2^-63 and multiplied and added exactly in 128 bits as well: conversions and
// products in FP64 took longer than the reads (the pass 330 us against 273 at 1000
// rows of 100,000 entries, 17 % non-zero). By Cauchy-Schwarz that sum stays
// below 2^63 times 2^63. Values below 2^-40, which that unit would cut short,
// are multiplied and added in FP64, in a loop of their own. The row's words (row_words) are left with exactly its
// non-zero entries' bits: bits of entries that became zero are cleared where the
// row is read through its map, all words are written where it is read whole.
// Other clusters keep their row (sizes and objective pieces as in k_write_rows).
__global__ void __launch_bounds__(WR_THREADS, 8) k_acc_rows1(
    int32_t k, const uint8_t *lam, const int64_t *cnt, const int64_t *acc_off, const int32_t *clu_doff,
    const int64_t *acc, uint32_t *bits, const int64_t *bit_off, uint32_t *scratch, int64_t avg_len, double inv_scale,
    const int64_t *coff_old, const int32_t *cterm_old, const float *cval_old, const double *snorm_old, int64_t *sz, double *snorm_new,
    double *jA, double *jU) {
    __shared__ long long shl[WR_THREADS];
    __shared__ unsigned long long sh128[2][WR_THREADS];
    __shared__ int s_any;  // a previous value lies below 2^-40 (a register for it costs spills, 1 % of the update)
    const int j = blockIdx.x;
    if (j >= k) return;
    if (threadIdx.x == 0) s_any = 0;
    __syncthreads();
    const int64_t cb = coff_old[j], ce = coff_old[j + 1];
    if (lam[j] != 0 || cnt[j] == 0) {  // invariant or empty
        if (threadIdx.x == 0) {
            const double sn = cnt[j] > 0 ? snorm_old[j] : 0.0;
            sz[j] = ce - cb;
            snorm_new[j] = sn;
            jA[j] = sn;  // unchanged members: <s_j, s_j / ||s_j||> = ||s_j||
            jU[j] = sn;
        }
        return;
    }
    const int64_t base = acc_off[j], L = acc_off[j + 1] - base;
    // <s_j, mu_j^[r-1]> over the thread's entries of the previous row (every
    // WR_THREADS-th) whose terms lie below a bound, from where it stopped last
    const int32_t doff = clu_doff[j];
    unsigned long long dot_hi = 0ull, dot_lo = 0ull;
    const uint32_t old = (uint32_t)(ce - cb);  // a row has at most 2^31 entries
    uint32_t at = threadIdx.x;
    auto dot_upto = [&](uint32_t bound) {
        for (bool more = at < old; more;) {
            uint32_t t[DOT_ILP];
#pragma unroll
            for (int q = 0; q < DOT_ILP; ++q)
                t[q] = at + q * WR_THREADS < old ? (uint32_t)(cterm_old[cb + (at + q * WR_THREADS)] - doff) : ~0u;
            long long v[DOT_ILP];
            float u[DOT_ILP];
#pragma unroll
            for (int q = 0; q < DOT_ILP; ++q) {
                v[q] = t[q] < bound ? acc[base + t[q]] : 0;
                u[q] = t[q] < bound ? cval_old[cb + (at + q * WR_THREADS)] : 1.f;  // times 0
            }
            more = t[DOT_ILP - 1] < bound;
#pragma unroll
            for (int q = 0; q < DOT_ILP; ++q) {
                add_product(dot_hi, dot_lo, (unsigned long long)v[q], fixed63(u[q]));
                if (u[q] < 0x1p-40f) s_any = 1;
                at += t[q] < bound ? WR_THREADS : 0;
            }
        }
    };
    uint32_t own_nz = 0;  // a row has at most 2^31 entries
    // ||S||^2 of the integer sums, exactly, as a 128-bit integer: the FP64 pipe
    // of this GPU retires about one operation per clock and SM, the integer
    // pipe dozens. Entries are non-negative (sums of positive member values)
    // and ||S|| = ||s_j|| 2^shift <= |C_j| 2^shift < 2^63, so the sum of
    // squares stays below 2^126.
    unsigned long long ss_hi = 0ull, ss_lo = 0ull;
    auto take = [&](long long v) {
        if (v) {
            ++own_nz;
            add_product(ss_hi, ss_lo, (unsigned long long)v, (unsigned long long)v);
        }
    };
    if (through_map(bits, ce - cb, cnt[j], avg_len, L)) {
        uint32_t *map = bits + bit_off[j];
        const int64_t nw = (L + 31) >> 5;
        for (int64_t w0 = threadIdx.x; w0 < nw; w0 += ILP * WR_THREADS) {
            uint32_t all[ILP];
#pragma unroll
            for (int q = 0; q < ILP; ++q) {
                const int64_t w = w0 + q * WR_THREADS;
                all[q] = w < nw ? map[w] : 0u;
            }
#pragma unroll
            for (int q = 0; q < ILP; ++q) {
                const int64_t w = w0 + q * WR_THREADS;
                uint32_t keep = all[q];
                const int64_t *e = acc + base + 32 * w;
                for (uint32_t b = all[q]; b;) {  // two entries in flight
                    const uint32_t b0 = b & (0u - b);
                    b ^= b0;
                    const uint32_t b1 = b & (0u - b);
                    b ^= b1;
                    const long long v0 = e[__ffs(b0) - 1];
                    const long long v1 = b1 ? e[__ffs(b1) - 1] : 0;
                    take(v0);
                    take(v1);
                    if (!v0) keep ^= b0;
                    if (!v1) keep &= ~b1;
                }
                if (keep != all[q]) map[w] = keep;
            }
        }
    } else {
        // rows start at even entries and have even lengths: 16-byte loads
        const longlong2 *row = reinterpret_cast<const longlong2 *>(acc + base);
        constexpr unsigned FULL = 0xffffffffu, TURN = ILP * WR_THREADS;
        const uint32_t L2 = (uint32_t)(L >> 1), nw = (uint32_t)((L + 31) >> 5), lane = threadIdx.x & 31;
        uint32_t *words = row_words(bits, bit_off, scratch, base, j);
        for (uint32_t p0 = 0; p0 < L2; p0 += TURN) {
            longlong2 v[ILP];
#pragma unroll
            for (int q = 0; q < ILP; ++q) {
                const uint32_t p = p0 + q * WR_THREADS + threadIdx.x;
                v[q] = p < L2 ? row[p] : make_longlong2(0, 0);
            }
            if (words) {  // a load of the warp is 64 entries, two words: lanes 2q and 2q + 1 write those of load q
                uint32_t x = 0, y = 0;
#pragma unroll
                for (int q = 0; q < ILP; ++q) {
                    const uint32_t bx = __ballot_sync(FULL, v[q].x != 0), by = __ballot_sync(FULL, v[q].y != 0);
                    if (lane >> 1 == q) {
                        x = bx;
                        y = by;
                    }
                }
                const uint32_t w = ((p0 + (lane >> 1) * WR_THREADS + (threadIdx.x & ~31u)) >> 4) + (lane & 1);
                const uint32_t half = (lane & 1) << 4;
                if (lane < 2 * ILP && w < nw) words[w] = interleave16(x >> half, y >> half);
            }
#pragma unroll
            for (int q = 0; q < ILP; ++q) {
                take(v[q].x);
                take(v[q].y);
            }
            if ((p0 / TURN) % DOT_TURNS == DOT_TURNS - 1) dot_upto(min(2 * (p0 + TURN), (uint32_t)L));
        }
    }
    const long long nz = block_sum_ll(own_nz, shl);
    block_sum_u128(ss_hi, ss_lo, sh128);
    // the exact sum to FP64 (one rounding of each half), then the power-of-two scale
    const double nrm = sqrt(((double)ss_hi * 18446744073709551616.0 + (double)ss_lo) * (inv_scale * inv_scale));
    dot_upto((uint32_t)L);
    block_sum_u128(dot_hi, dot_lo, sh128);
    double dot = ((double)dot_hi * 18446744073709551616.0 + (double)dot_lo) * inv_scale * 0x1p-63;
    if (s_any) {  // the same for the whole block, behind the sums' barriers
        double small = 0.0;
        for (uint32_t q = threadIdx.x; q < old; q += WR_THREADS) {
            const float u = cval_old[cb + q];
            if (u < 0x1p-40f) small += (double)acc[base + (cterm_old[cb + q] - doff)] * (double)u;
        }
        dot += block_sum_fixed(small, reinterpret_cast<double *>(shl)) * inv_scale;
    }
    if (threadIdx.x == 0) {
        sz[j] = nz;
        snorm_new[j] = nrm;
        jA[j] = dot;
        jU[j] = nrm;
    }
}

// Pass 2, one CTA per cluster: the new row in ascending term order and
// u = s * (2^-shift / ||s||) as FP32. Other clusters copy their row. A row that
// pass 1 read whole is cut into one stretch per warp by the words it left: the
// warps count their bits, one barrier gives each its place, and only the sectors
// with non-zero entries are read again (without the words every chunk of 1024
// entries waited for the block's counts, and every entry was read again: 277 us
// for 1000 rows of 100,000 entries, 17 % non-zero, against 199).
__global__ void __launch_bounds__(WR_THREADS, 8) k_acc_rows2(
    int32_t k, const uint8_t *lam, const int64_t *cnt, const int64_t *acc_off, const int32_t *clu_doff,
    const int64_t *acc, uint32_t *bits, const int64_t *bit_off, uint32_t *scratch, int64_t avg_len, double inv_scale, const int64_t *coff_old, const int32_t *cterm_old,
    const float *cval_old, const double *snorm_new, const int64_t *coff_new, int32_t *cterm_new, float *cval_new,
    int32_t *cclu_new, int64_t cap, unsigned long long *error) {
    constexpr int PER = 2;  // whole rows: sub-chunks of WR_THREADS entry pairs per chunk
    constexpr int NWR = WR_THREADS / 32;
    __shared__ int warp_n[PER][NWR];
    const int j = blockIdx.x;
    if (j >= k) return;
    const bool over = coff_new[k] > cap;  // more entries than the buffers hold: write nothing, report
    if (over && j == 0 && threadIdx.x == 0) atomicOr(error, ERR_CAPACITY);
    if (over) return;
    const int64_t o0 = coff_new[j];
    const int64_t cb = coff_old[j], ce = coff_old[j + 1];
    if (lam[j] != 0 || cnt[j] == 0) {  // invariant or empty
        for (int64_t q0 = cb + threadIdx.x; q0 < ce; q0 += ILP * WR_THREADS) {
            int32_t t[ILP];
            float u[ILP];
#pragma unroll
            for (int q = 0; q < ILP; ++q) {
                const int64_t at = q0 + q * WR_THREADS;
                if (at < ce) {
                    t[q] = cterm_old[at];
                    u[q] = cval_old[at];
                }
            }
#pragma unroll
            for (int q = 0; q < ILP; ++q) {
                const int64_t at = q0 + q * WR_THREADS;
                if (at < ce) {
                    cterm_new[o0 + (at - cb)] = t[q];
                    cval_new[o0 + (at - cb)] = u[q];
                    cclu_new[o0 + (at - cb)] = j;
                }
            }
        }
        return;
    }
    const int64_t base = acc_off[j], L = acc_off[j + 1] - base;
    const int32_t doff = clu_doff[j];
    // u = S * (2^-shift / ||s_j||) in FP32 from the integer sum S (split in
    // 32-bit halves, each converted with one rounding): at most 4 roundings,
    // a relative error below 2.4e-7, with no FP64 operation per entry
    const float ff = (float)(inv_scale / snorm_new[j]);
    auto value = [&](long long v) {
        const unsigned long long u = (unsigned long long)v;
        const float fs = fmaf(__uint2float_rn((unsigned)(u >> 32)), 4294967296.0f, __uint2float_rn((unsigned)u));
        return fs * ff;
    };
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t o = o0;
    if (through_map(bits, ce - cb, cnt[j], avg_len, L)) {  // as pass 1 decided, which left the bits of the non-zero entries
        const uint32_t *map = bits + bit_off[j];
        const int64_t nw = (L + 31) >> 5;
        int turn = 0;
        for (int64_t w0 = 0; w0 < nw; w0 += WR_THREADS, turn ^= 1) {
            const int64_t w = w0 + threadIdx.x;
            uint32_t b = w < nw ? map[w] : 0u;
            const int64_t *e = acc + base + 32 * w;
            const int n = __popc(b);
            int inc = n;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, inc, d);
                if (lane >= d) inc += y;
            }
            if (lane == 31) warp_n[turn][warp] = inc;
            __syncthreads();  // the counts of the turn before the last are rewritten only behind this
            int pre = 0, total = 0;
#pragma unroll
            for (int v = 0; v < NWR; ++v) {
                const int c = warp_n[turn][v];
                if (v < warp) pre += c;
                total += c;
            }
            int64_t pos = o + pre + (inc - n);
            for (; b; b &= b - 1, ++pos) {
                const int t = __ffs(b) - 1;
                cterm_new[pos] = (int32_t)(32 * w + t) + doff;
                cval_new[pos] = value(e[t]);
                cclu_new[pos] = j;
            }
            o += total;
        }
        return;
    }
    if (const uint32_t *words = row_words(bits, bit_off, scratch, base, j)) {
        const int64_t nw = (L + 31) >> 5, per = (nw + NWR - 1) / NWR;
        const int64_t wb = min(nw, per * warp), we = min(nw, per * (warp + 1));
        int n = 0;
        for (int64_t w = wb + lane; w < we; w += 32) n += __popc(words[w]);
        n = __reduce_add_sync(0xffffffffu, n);
        if (lane == 0) warp_n[0][warp] = n;
        __syncthreads();
        for (int v = 0; v < warp; ++v) o += warp_n[0][v];
        const uint32_t below = (1u << lane) - 1u;
        for (int64_t w0 = wb; w0 < we; w0 += 32) {
            const uint32_t mine = w0 + lane < we ? words[w0 + lane] : 0u;
            for (unsigned todo = __ballot_sync(0xffffffffu, mine != 0); todo;) {  // the non-empty words, four at a time
                uint32_t m[ILP];
                int at[ILP];
                long long v[ILP];
#pragma unroll
                for (int q = 0; q < ILP; ++q) {
                    at[q] = todo ? __ffs(todo) - 1 : 0;
                    m[q] = __shfl_sync(0xffffffffu, mine, at[q]);
                    if (!todo) m[q] = 0;
                    todo &= todo - 1;
                    if (m[q] >> lane & 1u) v[q] = acc[base + 32 * (w0 + at[q]) + lane];
                }
#pragma unroll
                for (int q = 0; q < ILP; ++q) {
                    if (m[q] >> lane & 1u) {
                        const int64_t pos = o + __popc(m[q] & below);
                        cterm_new[pos] = (int32_t)(32 * (w0 + at[q]) + lane) + doff;
                        cval_new[pos] = value(v[q]);
                        cclu_new[pos] = j;
                    }
                    o += __popc(m[q]);
                }
            }
        }
        return;
    }
    const longlong2 *row = reinterpret_cast<const longlong2 *>(acc + base);
    const int64_t L2 = L >> 1;  // entry pairs (even rows)
    for (int64_t c0 = 0; c0 < L2; c0 += (int64_t)WR_THREADS * PER) {
        // sub-chunk m holds pairs c0 + m*WR_THREADS + tid (coalesced 16-byte loads);
        // entries keep their order: pair by pair, and x before y inside a pair
        longlong2 v[PER];
        int ex[PER];
#pragma unroll
        for (int m = 0; m < PER; ++m) {
            const int64_t p = c0 + (int64_t)m * WR_THREADS + threadIdx.x;
            v[m] = p < L2 ? row[p] : make_longlong2(0, 0);
            const int n = (v[m].x != 0) + (v[m].y != 0);
            int inc = n;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, inc, d);
                if (lane >= d) inc += y;
            }
            ex[m] = inc - n;
            if (lane == 31) warp_n[m][warp] = inc;
        }
        __syncthreads();
        int total = 0;
#pragma unroll
        for (int m = 0; m < PER; ++m)
#pragma unroll
            for (int w = 0; w < NWR; ++w) total += warp_n[m][w];
#pragma unroll
        for (int m = 0; m < PER; ++m) {
            if (v[m].x == 0 && v[m].y == 0) continue;
            int pre = 0;
            for (int mm = 0; mm < m; ++mm)
                for (int w = 0; w < NWR; ++w) pre += warp_n[mm][w];
            for (int w = 0; w < warp; ++w) pre += warp_n[m][w];
            int64_t pos = o + pre + ex[m];
            const int64_t t = 2 * (c0 + (int64_t)m * WR_THREADS + threadIdx.x);
            const long long pv[2] = {v[m].x, v[m].y};
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                if (!pv[e]) continue;
                cterm_new[pos] = (int32_t)(t + e) + doff;
                cval_new[pos] = value(pv[e]);
                cclu_new[pos] = j;
                ++pos;
            }
        }
        o += total;
        __syncthreads();  // warp_n is rewritten by the next chunk
    }
}

// ---------------- u5: structured inverted file ----------------

// key = term << 1 | part (0 = front, moving; 1 = back, invariant). The
// unstructured file of IVF-CBICP keeps every posting in part 0.
__global__ void k_if_keys(const int64_t *n_dev, int64_t cap, const int32_t *cterm, const int32_t *cclu,
                          const uint8_t *lam, int structured, uint32_t *keys, uint32_t *vals, uint32_t *cnt2) {
    const int64_t n = live_entries(n_dev, cap);
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t key = ((uint32_t)cterm[e] << 1) | (uint32_t)(structured && lam[cclu[e]] ? 1 : 0);
        keys[e] = key;
        vals[e] = (uint32_t)e;
        atomicAdd(cnt2 + key, 1u);
    }
}

// Canonical arrays (if_cid: global cluster ids, if_val) in sorted order.
__global__ void k_if_fill(const int64_t *n_dev, int64_t cap, const uint32_t *order, const int32_t *cclu,
                          const float *cval, int32_t *if_cid, float *if_val) {
    const int64_t n = live_entries(n_dev, cap);
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t e = order[q];
        if_cid[q] = cclu[e];
        if_val[q] = cval[e];
    }
}

// ---------------- scan order and dense head rows ----------------

constexpr int DENSE_BINS = 64;      // list length / k in steps of 1/64
constexpr int DENSE_MIN_LEN = 32;   // shorter lists stay sparse whatever k

// instance of term t, its k, and the 1/64 bin of its list length
__device__ __forceinline__ void term_bin(int32_t t, int32_t n_inst, const int32_t *inst_d, const int32_t *inst_k,
                                         int64_t L, int32_t *kin, int *bin) {
    int lo = 0, hi = n_inst - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (inst_d[mid] <= t) lo = mid; else hi = mid - 1;
    }
    const int32_t km = inst_k[lo + 1] - inst_k[lo];
    *kin = km;
    const int64_t q = (L * DENSE_BINS) / (km > 0 ? km : 1);
    *bin = (int)(q < DENSE_BINS ? q : DENSE_BINS);
}

// First pass over the terms of the build: list lengths and front lengths from
// the per-part counts, the slot cursors cleared, and the histogram of the
// dense-row entries each length bin would take (lists of at least min_len
// postings; formed per block, then added). The scan position of every cluster
// is found beside it: within its instance, the moving clusters of lambda^[r]
// (mov_list, ascending) take positions 0 .. n_mov - 1 and the invariant ones
// follow in ascending id; id_order (IVF-CBICP) keeps the ids. lambda is kept as
// the canonical file's, which may be asked for after it has changed.
__global__ void __launch_bounds__(TPB) k_if_lists(int32_t D, int32_t k, int32_t n_inst, const int32_t *inst_d,
                                                  const int32_t *inst_k, const uint32_t *cnt2, int64_t min_len,
                                                  int dense, int64_t *len, int32_t *mf0, uint32_t *cursor,
                                                  unsigned long long *hist, const uint8_t *lam,
                                                  const int32_t *mov_list, const int32_t *mov_beg, int id_order,
                                                  int32_t *clu_pos, int32_t *pos_clu, uint8_t *lam_file,
                                                  DevCounters *ctr) {
    __shared__ unsigned long long sh[DENSE_BINS + 1];
    for (int b = threadIdx.x; b <= DENSE_BINS; b += TPB) sh[b] = 0ull;
    if (blockIdx.x == 0 && threadIdx.x == 0) ctr->dense_terms = 0;
    __syncthreads();
    const int64_t g0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, st = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = g0; t < D; t += st) {
        const uint32_t f = cnt2[2 * t], b = cnt2[2 * t + 1];
        const int64_t L = (int64_t)f + (int64_t)b;
        len[t] = L;
        mf0[t] = (int32_t)f;
        cursor[2 * t] = 0u;
        cursor[2 * t + 1] = 0u;
        if (dense && L >= min_len) {
            int32_t km;
            int bin;
            term_bin((int32_t)t, n_inst, inst_d, inst_k, L, &km, &bin);
            atomicAdd(sh + bin, (unsigned long long)((km + 7) & ~7));
        }
    }
    for (int64_t g = g0; g < k; g += st) {
        const int32_t j = (int32_t)g;
        int lo = 0, hi = n_inst - 1;  // instance: largest m with inst_k[m] <= j
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (inst_k[mid] <= j) lo = mid; else hi = mid - 1;
        }
        const int32_t koff = inst_k[lo], jl = j - koff;
        int32_t p = jl;
        if (!id_order) {
            const int32_t b = mov_beg[lo], e = mov_beg[lo + 1];
            int32_t a = b, z = e;  // first moving id >= j
            while (a < z) {
                const int32_t mid = (a + z) >> 1;
                if (mov_list[mid] < j) a = mid + 1; else z = mid;
            }
            p = lam[j] == 0 ? a - b : (e - b) + (jl - (a - b));
        }
        clu_pos[j] = p;
        pos_clu[koff + p] = jl;
        lam_file[j] = lam[j];
    }
    __syncthreads();
    for (int b = threadIdx.x; b <= DENSE_BINS; b += TPB)
        if (sh[b]) atomicAdd(hist + b, sh[b]);
}

// The terms in tiles of IF_TILE: second pass, the width of a dense row (in
// 8-entry units) or the room of a sparse list for every term, and each tile's
// sums of list lengths, sparse entries and row widths. Every block finds the
// dense threshold from the histogram: the smallest bin >= bmin whose rows
// (with every longer bin's) fit in cap entries; DENSE_BINS + 1 = no dense rows.
constexpr int IF_TILE = 4 * TPB;
// Up to this many tiles every block adds up the earlier ones for itself, above
// it, where that grows with their square, they are scanned in a launch of their
// own. ms per update (3000 documents, k = 50), added / scanned: 1954 tiles 0.312
// / 0.316, 3907 0.366 / 0.373, 15,625 0.754 / 0.691, 62,500 3.37 / 1.91, 125,000
// (128M terms) 9.91 / 3.49.
constexpr int64_t IF_TILES_ADDED = 4096;

struct IfSums {
    long long len, room, w8;
};

__device__ __forceinline__ IfSums if_add(IfSums a, IfSums b) {
    return {a.len + b.len, a.room + b.room, a.w8 + b.w8};
}

// inclusive scan over the block; total for every thread (two barriers)
__device__ __forceinline__ IfSums if_block_scan(IfSums v, IfSums *warp_s, IfSums &total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const IfSums y = {__shfl_up_sync(0xffffffffu, v.len, o), __shfl_up_sync(0xffffffffu, v.room, o),
                          __shfl_up_sync(0xffffffffu, v.w8, o)};
        if (lane >= o) v = if_add(v, y);
    }
    __syncthreads();
    if (lane == 31) warp_s[warp] = v;
    __syncthreads();
    IfSums before = {0, 0, 0};
    total = {0, 0, 0};
#pragma unroll
    for (int w = 0; w < TPB / 32; ++w) {
        if (w < warp) before = if_add(before, warp_s[w]);
        total = if_add(total, warp_s[w]);
    }
    return if_add(before, v);
}

__device__ __forceinline__ int64_t quads4(int64_t n) { return (n + 3) & ~(int64_t)3; }

__global__ void __launch_bounds__(TPB) k_if_tiles(int32_t D, int32_t n_inst, const int32_t *inst_d,
                                                  const int32_t *inst_k, const int64_t *len, const int32_t *mf0,
                                                  int64_t min_len, const unsigned long long *hist, int bmin,
                                                  unsigned long long cap, int32_t *thr, int32_t *w8, IfSums *tiles) {
    __shared__ IfSums warp_s[TPB / 32];
    __shared__ unsigned long long sh[DENSE_BINS + 1];
    __shared__ int s_thr;
    for (int b = threadIdx.x; b <= DENSE_BINS; b += TPB) sh[b] = hist[b];
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long acc = 0;
        int b = DENSE_BINS + 1;
        for (int q = DENSE_BINS; q >= bmin; --q) {
            acc += sh[q];
            if (acc > cap) break;
            b = q;
        }
        s_thr = b;
        if (blockIdx.x == 0) *thr = b;
    }
    __syncthreads();
    const int64_t n_tiles = ((int64_t)D + IF_TILE - 1) / IF_TILE;
    for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
        IfSums v = {0, 0, 0};
#pragma unroll
        for (int q = 0; q < IF_TILE / TPB; ++q) {
            const int64_t t = tile * IF_TILE + (int64_t)q * TPB + threadIdx.x;
            if (t >= D) break;
            const int64_t L = len[t];
            int64_t w = 0;
            if (L >= min_len && s_thr <= DENSE_BINS) {
                int32_t km;
                int bin;
                term_bin((int32_t)t, n_inst, inst_d, inst_k, L, &km, &bin);
                if (bin >= s_thr) w = (km + 7) >> 3;
            }
            w8[t] = (int32_t)w;
            const int64_t f = mf0[t];
            v = if_add(v, {L, w ? 0 : quads4(f) + quads4(L - f), w});
        }
        IfSums total;
        if_block_scan(v, warp_s, total);
        if (threadIdx.x == 0) tiles[tile] = total;
    }
}

// The tiles' sums made sums of the earlier tiles, by one CTA of which a thread
// takes PER tiles a turn.
__global__ void __launch_bounds__(TPB) k_if_tile_scan(int64_t n_tiles, IfSums *tiles) {
    constexpr int PER = 4;
    __shared__ IfSums warp_s[TPB / 32];
    IfSums carry = {0, 0, 0};
    for (int64_t b = 0; b < n_tiles; b += TPB * PER) {
        const int64_t t0 = b + (int64_t)threadIdx.x * PER;
        IfSums v[PER], sum = {0, 0, 0};
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            v[q] = t0 + q < n_tiles ? tiles[t0 + q] : IfSums{0, 0, 0};
            sum = if_add(sum, v[q]);
        }
        IfSums total;
        const IfSums inc = if_block_scan(sum, warp_s, total);
        IfSums at = {carry.len + inc.len - sum.len, carry.room + inc.room - sum.room, carry.w8 + inc.w8 - sum.w8};
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            if (t0 + q < n_tiles) tiles[t0 + q] = at;
            at = if_add(at, v[q]);
        }
        carry = if_add(carry, total);
    }
}

// Third pass: the offsets (sums of the earlier tiles, then within the tile)
// and what the assignment reads about a term, in one 16-byte descriptor: the
// first quad of its list in the scan copy, its front and list lengths, and its
// dense row. The last quads of a sparse list's front and back are filled up
// with zero postings here (they add 0 to a score). tiles: sums of the earlier
// tiles (summed), or the tiles' own, of which every block adds up the earlier
// ones.
__global__ void __launch_bounds__(TPB) k_if_offsets(int32_t D, const int64_t *len, const int32_t *mf0,
                                                    const int32_t *w8, const IfSums *tiles, int summed, int64_t *if_off,
                                                    int4 *tdesc, uint16_t *sc_id16, int32_t *sc_id32, float *sc_val,
                                                    uint32_t *sc_pack, uint16_t *sc_lp, DevCounters *ctr) {
    __shared__ IfSums warp_s[TPB / 32];
    auto fill = [&](int64_t from, int64_t to) {
        for (int64_t p = from; p < to; ++p) {
            if (sc_id16) sc_id16[p] = 0;
            if (sc_id32) sc_id32[p] = 0;
            if (sc_val) sc_val[p] = 0.0f;
            if (sc_pack) sc_pack[p] = 0;
            if (sc_lp) sc_lp[p] = 0;
        }
    };
    const int64_t n_tiles = ((int64_t)D + IF_TILE - 1) / IF_TILE;
    long long n_dense = 0;
    for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
        IfSums base = {0, 0, 0};
        if (summed) {
            base = tiles[tile];
        } else {
            for (int64_t q = threadIdx.x; q < tile; q += TPB) base = if_add(base, tiles[q]);
            IfSums total;
            if_block_scan(base, warp_s, total);
            base = total;  // every earlier tile
        }
#pragma unroll
        for (int q = 0; q < IF_TILE / TPB; ++q) {
            const int64_t t = tile * IF_TILE + (int64_t)q * TPB + threadIdx.x;
            int64_t L = 0, f = 0, w = 0;
            if (t < D) {
                L = len[t];
                f = mf0[t];
                w = w8[t];
            }
            const IfSums v = {L, w ? 0 : quads4(f) + quads4(L - f), w};
            IfSums total;
            const IfSums inc = if_block_scan(v, warp_s, total);
            if (t < D) {
                const int64_t at = base.room + inc.room - v.room;
                if_off[t] = base.len + inc.len - L;
                tdesc[t] = make_int4((int)(at >> 2), (int)f, (int)L, w ? (int)(base.w8 + inc.w8 - w) : -1);
                if (w) {
                    ++n_dense;
                } else {
                    fill(at + f, at + quads4(f));
                    fill(at + quads4(f) + (L - f), at + v.room);
                }
            }
            base = if_add(base, total);
        }
        if (tile == n_tiles - 1 && threadIdx.x == 0) {
            if_off[D] = base.len;
            ctr->sparse_entries = base.room;
            ctr->dense_used = base.w8;
        }
    }
    if (n_dense) atomicAdd(reinterpret_cast<unsigned long long *>(&ctr->dense_terms), (unsigned long long)n_dense);
}

// zero the entries in use (16 bytes at a time; rows are multiples of 8 entries)
__global__ void k_dense_zero(const DevCounters *ctr, int esize, uint4 *dense) {
    const int64_t n16 = ctr->dense_used * 8 * esize / 16;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n16; q += (int64_t)gridDim.x * blockDim.x)
        dense[q] = make_uint4(0u, 0u, 0u, 0u);
}

// 16-bit stored value of a posting: BF16 (nearest, ties to even), or FP16 of
// u * 2^14 kept strictly positive
__device__ __forceinline__ uint16_t encode_lp(float u, int prec) {
    if (prec == SIVF_BF16) return __bfloat16_as_ushort(__float2bfloat16_rn(u));
    unsigned short h = __half_as_ushort(__float2half_rn(u * FP16_SCALE));
    if (h == 0 && u > 0.0f) h = 1;
    return h;
}

// per (term, part) posting counts of the current centroids
__global__ void k_if_count(const int64_t *n_dev, int64_t cap, const int32_t *cterm, const int32_t *cclu,
                           const uint8_t *lam, int structured, uint32_t *cnt2) {
    const int64_t n = live_entries(n_dev, cap);
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
        atomicAdd(cnt2 + (((uint32_t)cterm[e] << 1) | (uint32_t)(structured && lam[cclu[e]] ? 1 : 0)), 1u);
}

// The scan structures read by the assignment, straight from the cluster-major
// centroid entries (one pass, no sort): an entry of a term with a dense row
// goes to the row at its cluster's scan position; any other entry takes the
// next free slot of its term's front (moving cluster) or back (invariant
// cluster) in the scan copy, with the score slot of the cluster's scan position
// as its id. The order of the postings inside a segment follows the atomic
// cursor; no score depends on it (each posting is one integer add).
__global__ void k_scan_fill(const int64_t *n_dev, int64_t cap, const int32_t *cterm, const int32_t *cclu,
                            const float *cval, const uint8_t *lam, int structured, const int32_t *clu_pos,
                            const int4 *tdesc, uint32_t *cursor, int prec, void *dense, uint16_t *sc_id16,
                            int32_t *sc_id32, float *sc_val, uint32_t *sc_pack, uint16_t *sc_lp) {
    const int64_t n = live_entries(n_dev, cap);
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        const int32_t t = cterm[e], j = cclu[e];
        const float u = cval[e];
        const uint32_t p = (uint32_t)clu_pos[j];
        const int4 td = tdesc[t];
        if (td.w >= 0) {
            const int64_t d = (int64_t)td.w * 8 + p;
            if (prec == SIVF_FP32) static_cast<float *>(dense)[d] = u;
            else if (prec == SIVF_FP16 || !(p & 1u)) static_cast<uint16_t *>(dense)[d] = encode_lp(u, prec);
            continue;  // odd entries of BF16 rows: k_dense_odd
        }
        const uint32_t part = (structured && lam[j]) ? 1u : 0u;
        const int64_t pos = (int64_t)(unsigned)td.x * 4 + atomicAdd(cursor + (((uint32_t)t << 1) | part), 1u) +
                            (part ? (td.y + 3) & ~3 : 0);
        const uint32_t id = structured ? (uint32_t)score_slot((int)p) : p;  // IVF-CBICP keeps cluster ids
        if (sc_id16) sc_id16[pos] = (uint16_t)id;
        if (sc_id32) sc_id32[pos] = (int32_t)id;
        if (prec == SIVF_FP32) {
            sc_val[pos] = u;
            continue;
        }
        const uint16_t lp = encode_lp(u, prec);
        if (sc_pack) sc_pack[pos] = (id << 16) | (uint32_t)lp;
        else sc_lp[pos] = lp;
    }
}

// Odd entries of the BF16 dense rows, once the even ones are there: the scan
// reads a word (even entry below, odd entry above) as FP32 for the odd one.
__global__ void k_dense_odd(const int64_t *n_dev, int64_t cap, const int32_t *cterm, const int32_t *cclu,
                            const float *cval, const int32_t *clu_pos, const int4 *tdesc, uint16_t *dense) {
    const int64_t n = live_entries(n_dev, cap);
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        const int32_t p = clu_pos[cclu[e]];
        if (!(p & 1)) continue;
        const int32_t row = tdesc[cterm[e]].w;
        if (row < 0) continue;
        uint16_t *at = dense + (int64_t)row * 8 + p;
        *at = odd_upper_half(__float_as_uint(cval[e]), at[-1]);
    }
}

}  // namespace

cudaError_t validate_csr(sivf_ctx *c, int *bad_host) {
    int *bad = c->ws.take<int>(1);
    if (!bad) return cudaErrorMemoryAllocation;
    SIVF_CUDA_TRY(cudaMemsetAsync(bad, 0, sizeof(int), c->stream));
    k_validate<<<blocks_gs(c->N * 32), TPB, 0, c->stream>>>(c->N, c->D, c->nnz, c->row_ptr, c->idx, c->val,
                                                               c->sumv, bad);
    note_launch();
    SIVF_CUDA_TRY(cudaGetLastError());
    SIVF_CUDA_TRY(cudaMemcpyAsync(bad_host, bad, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
    SIVF_CUDA_TRY(cudaStreamSynchronize(c->stream));
    c->ws.reset();
    return cudaSuccess;
}

cudaError_t set_labels_dev(sivf_ctx *c, const int32_t *src) {
    // src must not live in the workspace region taken below
    int *bad = c->ws.take<int>(1);
    if (!bad) return cudaErrorMemoryAllocation;
    SIVF_CUDA_TRY(cudaMemsetAsync(bad, 0, sizeof(int), c->stream));
    k_check_labels<<<blocks_gs(c->N), TPB, 0, c->stream>>>(c->N, c->k, src, bad);
    note_launch();
    int bad_h = 0;
    SIVF_CUDA_TRY(cudaMemcpyAsync(&bad_h, bad, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
    SIVF_CUDA_TRY(cudaStreamSynchronize(c->stream));
    if (bad_h) return cudaErrorInvalidValue;
    // labels set twice without an update in between: the centroids belong to
    // those before the first call, so its marks stay
    const bool rebuilt = !c->assigned;
    if (!(rebuilt && c->needs_update)) SIVF_CUDA_TRY(cudaMemsetAsync(c->moving, 0, c->k, c->stream));
    k_set_labels<<<blocks_gs(c->N), TPB, 0, c->stream>>>(c->N, src, c->labels, c->labels_prev, rebuilt ? 1 : 0, c->own,
                                                         c->moving);
    note_launch();
    SIVF_CUDA_TRY(cudaGetLastError());
    if (c->iter == 0) c->iter = 1;  // first membership: every cluster is moving
    SIVF_CUDA_TRY(launch_finalize_assign(c));
    return cudaSuccess;
}

// Scan structures of the structured inverted file of the current centroids
// (count in coff[k], on the device) with the current lambda: list offsets and
// front lengths, the scan order, the dense head rows and the sparse scan copy.
// No host synchronisation. The canonical file (ascending ids in each part,
// for the getters) is built on demand by build_canonical_if.
cudaError_t build_inverted_file(sivf_ctx *c) {
    const int64_t cap = c->cap_c;
    const int cur = c->cur;
    const int64_t *n_dev = c->coff[cur] + c->k;
    const int32_t D = c->D;
    Workspace &ws = c->ws;
    size_t mark = ws.used;
    const int64_t n_tiles = ((int64_t)D + IF_TILE - 1) / IF_TILE;
    // the counts and the histogram are cleared together
    uint32_t *cnt2 = ws.take<uint32_t>((size_t)2 * D + 2 * (DENSE_BINS + 1));
    uint32_t *cursor = ws.take<uint32_t>((size_t)2 * D);
    int64_t *len = ws.take<int64_t>((size_t)D);
    int32_t *w8 = ws.take<int32_t>((size_t)D);
    IfSums *tiles = ws.take<IfSums>((size_t)n_tiles);
    if (!cnt2 || !cursor || !len || !w8 || !tiles) return cudaErrorMemoryAllocation;
    unsigned long long *hist = reinterpret_cast<unsigned long long *>(cnt2 + 2 * (size_t)D);
    cudaStream_t s = c->stream;
    const bool cb = c->cfg.icp == 2;
    c->canon_stale = true;
    SIVF_CUDA_TRY(cudaMemsetAsync(cnt2, 0, sizeof(uint32_t) * (2 * (size_t)D + 2 * (DENSE_BINS + 1)), s));
    k_if_count<<<blocks_gs(cap), TPB, 0, s>>>(n_dev, cap, c->cterm[cur], c->cclu, c->lam, cb ? 0 : 1, cnt2);
    // dense head rows: the longest lists (relative to their instance's k) that
    // fit in the row capacity, from dense_frac of k up; with dense_all every
    // list (the dense-mean variant: all of the centroids as dense rows)
    const bool all = c->cfg.dense_all != 0;
    const int bmin = all ? 0 : std::max(1, (int)ceilf(c->dense_frac * DENSE_BINS));
    const int64_t min_len = all ? 1 : DENSE_MIN_LEN;
    const bool dense = c->cap_dense > 0 && !cb && bmin <= DENSE_BINS;
    const unsigned tile_blocks = (unsigned)std::min<int64_t>(n_tiles, GS_MAX_BLOCKS);
    // (mov_list and mov_beg belong to the current lambda^[r])
    k_if_lists<<<(unsigned)std::min<int64_t>(blocks_for(std::max(D, c->k)), 1024), TPB, 0, s>>>(
        D, c->k, c->n_inst, c->inst_d, c->inst_k, cnt2, min_len, dense ? 1 : 0, len, c->if_mf0, cursor, hist, c->lam,
        c->mov_list, c->mov_beg, cb ? 1 : 0, c->clu_pos, c->pos_clu, c->lam_file, c->ctr);
    k_if_tiles<<<tile_blocks, TPB, 0, s>>>(D, c->n_inst, c->inst_d, c->inst_k, len, c->if_mf0, min_len, hist,
                                           dense ? bmin : DENSE_BINS + 1, (unsigned long long)c->cap_dense,
                                           c->dense_thr, w8, tiles);
    const bool summed = n_tiles > IF_TILES_ADDED;
    if (summed) {
        k_if_tile_scan<<<1, TPB, 0, s>>>(n_tiles, tiles);
        note_launch();
    }
    k_if_offsets<<<tile_blocks, TPB, 0, s>>>(D, len, c->if_mf0, w8, tiles, summed ? 1 : 0, c->if_off, c->tdesc, c->sc_id16, c->sc_id32,
                                             c->sc_val, c->sc_pack, c->sc_lp, c->ctr);
    note_launch(4);
    SIVF_CUDA_TRY(cudaGetLastError());
    if (dense) {
        const int esize = c->cfg.prec == SIVF_FP32 ? 4 : 2;
        k_dense_zero<<<blocks_gs(c->cap_dense * esize / 16), TPB, 0, s>>>(c->ctr, esize,
                                                                            static_cast<uint4 *>(c->dense_val));
        note_launch();
    }
    k_scan_fill<<<blocks_gs(cap), TPB, 0, s>>>(n_dev, cap, c->cterm[cur], c->cclu, c->cval[cur], c->lam, cb ? 0 : 1,
                                                c->clu_pos, c->tdesc, cursor, (int)c->cfg.prec, c->dense_val,
                                                c->sc_id16, c->sc_id32, c->sc_val, c->sc_pack, c->sc_lp);
    note_launch();
    if (dense && c->cfg.prec == SIVF_BF16) {
        k_dense_odd<<<blocks_gs(cap), TPB, 0, s>>>(n_dev, cap, c->cterm[cur], c->cclu, c->cval[cur], c->clu_pos,
                                                   c->tdesc, static_cast<uint16_t *>(c->dense_val));
        note_launch();
    }
    SIVF_CUDA_TRY(cudaGetLastError());
    ws.used = mark;
    return cudaSuccess;
}

// The canonical structured inverted file of the current centroids and the lambda
// of the last build (Algorithm 5: for every term, the moving centroids first and
// the invariant ones after, ascending ids in each part), with the offsets and
// front lengths of that build: a stable radix sort of the centroid entries by
// (term, part). It lies in the centroid buffer that is not current (terms:
// cluster ids, values), which nothing reads until the next update writes it.
// Used by the getters only; synchronises the stream.
cudaError_t build_canonical_if(sivf_ctx *c) {
    if (!c->canon_stale) return cudaSuccess;
    const int64_t cap = c->cap_c;
    const int cur = c->cur;
    const int64_t *n_dev = c->coff[cur] + c->k;
    Workspace &ws = c->ws;
    ws.reset();
    uint32_t *cnt2 = ws.take<uint32_t>((size_t)2 * c->D);
    uint32_t *k0 = ws.take<uint32_t>((size_t)cap + 1), *v0 = ws.take<uint32_t>((size_t)cap + 1);
    uint32_t *k1 = ws.take<uint32_t>((size_t)cap + 1), *v1 = ws.take<uint32_t>((size_t)cap + 1);
    if (!cnt2 || !k0 || !v0 || !k1 || !v1) return cudaErrorMemoryAllocation;
    cudaStream_t s = c->stream;
    SIVF_CUDA_TRY(cudaMemsetAsync(cnt2, 0, sizeof(uint32_t) * 2 * c->D, s));
    k_if_keys<<<blocks_gs(cap), TPB, 0, s>>>(n_dev, cap, c->cterm[cur], c->cclu, c->lam_file, c->cfg.icp == 2 ? 0 : 1,
                                              k0, v0, cnt2);
    note_launch();
    bool alt = false;
    SIVF_CUDA_TRY(radix_sort_pairs_dev(k0, v0, k1, v1, cap, n_dev, c->bits_t + 1, &alt, ws, s));
    k_if_fill<<<blocks_gs(cap), TPB, 0, s>>>(n_dev, cap, alt ? v1 : v0, c->cclu, c->cval[cur],
                                              c->cterm[1 - cur], c->cval[1 - cur]);
    note_launch();
    SIVF_CUDA_TRY(cudaGetLastError());
    SIVF_CUDA_TRY(cudaStreamSynchronize(s));
    ws.reset();
    c->canon_stale = false;
    return cudaSuccess;
}

namespace {

// coff of the new buffer from the row sizes
cudaError_t row_offsets(sivf_ctx *c, const int64_t *sz, int nw) {
    cudaStream_t s = c->stream;
    // one CTA, 4096 rows a turn, or a scan of two launches: ms per update, one /
    // two, at k = 4096 0.307 / 0.311, 16,384 0.509 / 0.505, 65,536 1.21 / 1.17,
    // 262,144 3.95 / 3.76
    if (c->k <= 8192) {
        k_row_offsets<<<1, 1024, 0, s>>>(c->k, sz, c->coff[nw]);
        note_launch();
        return cudaGetLastError();
    }
    return scan_exclusive_i64(sz, c->coff[nw], c->k, c->coff[nw] + c->k, c->ws, s);
}

// objective sums, rows into the current buffer, counts of the step
cudaError_t finish_rows(sivf_ctx *c, const double *jA, const double *jU, const int64_t *moved) {
    const int cur = c->cur, nw = 1 - c->cur;
    const unsigned copy = (unsigned)std::min<int64_t>((c->cap_c + 1023) / 1024, 1024);
    k_finish_rows<<<(unsigned)c->n_inst + copy, 1024, 0, c->stream>>>(
        c->k, c->cap_c, c->n_inst, c->inst_k, jA, jU, c->obj_dev, c->coff[nw], c->cterm[nw], c->cval[nw],
        c->snorm_new, c->coff[cur], c->cterm[cur], c->cval[cur], c->snorm, moved, c->ctr);
    note_launch();
    return cudaGetLastError();
}

}  // namespace

// Restart from new seeds: no labels, no own scores, every cluster moving,
// mu^[0] = seed rows (distinct documents: they fit the centroid buffers unless
// the borrowed CSR changed), first inverted file. No host synchronisation; the
// counts and a failed check are in the counters.
cudaError_t reseed_dev(sivf_ctx *c, const int32_t *init_ids_dev) {
    const int64_t N = c->N;
    const int32_t k = c->k;
    const int cur = c->cur;
    cudaStream_t s = c->stream;
    const size_t mark = c->ws.used;
    int64_t *sz = c->ws.take<int64_t>((size_t)k + 1);
    if (!sz) return cudaErrorMemoryAllocation;
    if (c->dense) {  // no member has been added yet
        if (c->acc_bits && c->acc_ready) {
            k_acc_clear<<<(unsigned)std::min<int32_t>(k, 65535), TPB, 0, s>>>(k, c->acc_off, c->acc_bit_off, c->acc,
                                                                              c->acc_bits);
            note_launch();
        } else {
            SIVF_CUDA_TRY(cudaMemsetAsync(c->acc, 0, sizeof(int64_t) * (size_t)c->acc_total, s));
            if (c->acc_bits)
                SIVF_CUDA_TRY(cudaMemsetAsync(c->acc_bits, 0, sizeof(uint32_t) * (size_t)c->acc_words, s));
            c->acc_ready = true;
        }
    }
    k_reset<<<blocks_gs(std::max<int64_t>(N, k)), TPB, 0, s>>>(N, k, c->labels, c->labels_prev, c->own,
                                                               c->dense ? c->acc_lab : nullptr, c->lam, c->lam_prev,
                                                               c->moving, c->snorm, init_ids_dev, c->row_ptr, c->nnz,
                                                               c->cap_c, sz, c->ctr);
    note_launch();
    c->iter = 1;  // finalize below marks every cluster moving
    SIVF_CUDA_TRY(launch_finalize_assign(c));
    c->iter = 0;
    SIVF_CUDA_TRY(row_offsets(c, sz, cur));
    k_seed_rows<<<blocks_for((int64_t)k * 32), TPB, 0, s>>>(k, init_ids_dev, c->row_ptr, c->idx, c->val, c->coff[cur],
                                                            c->cap_c, c->cterm[cur], c->cval[cur], c->cclu, c->ctr);
    note_launch();
    SIVF_CUDA_TRY(cudaGetLastError());
    SIVF_CUDA_TRY(build_inverted_file(c));
    c->ws.used = mark;
    c->needs_update = false;
    c->assigned = false;
    return cudaSuccess;
}

// Update step with the dense accumulator (u1: member counts only; u2-u4 as
// above; u5 as in the sort form).
cudaError_t run_update_dense(sivf_ctx *c) {
    cudaStream_t s = c->stream;
    Workspace &ws = c->ws;
    ws.reset();
    const int64_t N = c->N;
    const int32_t k = c->k;
    const int cur = c->cur, nw = 1 - c->cur;
    int64_t *cnt = ws.take<int64_t>((size_t)k + 1), *sz = ws.take<int64_t>((size_t)k + 1);
    double *jAd = ws.take<double>(k), *jUd = ws.take<double>(k);
    if (!cnt || !sz || !jAd || !jUd) return cudaErrorMemoryAllocation;
    int64_t *moved_d = cnt + k;  // cleared with the counts
    SIVF_CUDA_TRY(cudaMemsetAsync(cnt, 0, sizeof(int64_t) * ((size_t)k + 1), s));
    const float fscale = ldexpf(1.0f, c->acc_shift);
    const double inv_scale = ldexp(1.0, -c->acc_shift);
    const int64_t avg_len = c->nnz / N + 1;  // entries of an object
    int per = 1;  // objects a warp looks at together: as many as still leave every SM 64 warps
    while (per < 32 && N / (2 * per) >= (int64_t)c->num_sms * 64) per *= 2;
    k_acc_scatter<<<blocks_gs((N + per - 1) / per * 32), TPB, 0, s>>>(
        N, per, c->labels, c->acc_lab, c->row_ptr, c->idx, c->val, c->clu_doff, c->acc_off, fscale, c->acc,
        c->acc_bits, c->acc_bit_off, cnt, moved_d);
    // Without a map, the row passes' words lie in the workspace: it is sized for
    // sorting as many entries as the centroids can hold, far more than a bit
    // per accumulator entry wherever rows are too full for a map.
    const size_t n_words = (size_t)(c->acc_total / 32 + k + 1);
    uint32_t *words = !c->acc_bits && 4 * n_words <= ws.cap / 2 ? ws.take<uint32_t>(n_words) : nullptr;
    k_acc_rows1<<<(unsigned)k, WR_THREADS, 0, s>>>(k, c->lam, cnt, c->acc_off, c->clu_doff, c->acc, c->acc_bits,
                                                   c->acc_bit_off, words, avg_len, inv_scale, c->coff[cur], c->cterm[cur],
                                                   c->cval[cur], c->snorm, sz, c->snorm_new, jAd, jUd);
    SIVF_CUDA_TRY(row_offsets(c, sz, nw));
    k_acc_rows2<<<(unsigned)k, WR_THREADS, 0, s>>>(k, c->lam, cnt, c->acc_off, c->clu_doff, c->acc, c->acc_bits,
                                                   c->acc_bit_off, words, avg_len, inv_scale, c->coff[cur], c->cterm[cur],
                                                   c->cval[cur], c->snorm_new, c->coff[nw], c->cterm[nw], c->cval[nw],
                                                   c->cclu, c->cap_c, &c->ctr->error);
    note_launch(3);
    SIVF_CUDA_TRY(finish_rows(c, jAd, jUd, moved_d));
    ws.reset();
    SIVF_CUDA_TRY(build_inverted_file(c));
    ws.reset();
    return cudaSuccess;
}

// One update step (Algorithm 5). Every size that depends on the data stays on
// the device, so the whole step can be captured in a CUDA graph.
cudaError_t run_update(sivf_ctx *c) {
    cudaStream_t s = c->stream;
    Workspace &ws = c->ws;
    ws.reset();
    const int64_t N = c->N;
    const int32_t k = c->k;
    const int64_t Tmax = c->nnz > 0 ? c->nnz : 1;
    const int cur = c->cur, nw = 1 - c->cur;

    if (c->dense) return run_update_dense(c);

    // u1: members grouped by cluster, ascending object id
    uint32_t *lk0 = ws.take<uint32_t>(N), *lv0 = ws.take<uint32_t>(N);
    uint32_t *lk1 = ws.take<uint32_t>(N), *lv1 = ws.take<uint32_t>(N);
    int64_t *cnt = ws.take<int64_t>(k), *flag = ws.take<int64_t>(k), *rrank = ws.take<int64_t>(k);
    int64_t *nrec_d = ws.take<int64_t>(1), *T_d = ws.take<int64_t>(1);
    uint32_t *U_d = ws.take<uint32_t>(1);
    int64_t *sz = ws.take<int64_t>((size_t)k + 1);
    double *jAd = ws.take<double>(k), *jUd = ws.take<double>(k);
    int64_t *tc = ws.take<int64_t>(N), *toff = ws.take<int64_t>(N);
    int64_t *ubeg = ws.take<int64_t>((size_t)k + 1), *uend = ws.take<int64_t>((size_t)k + 1);
    if (!lk0 || !lv0 || !lk1 || !lv1 || !cnt || !flag || !rrank || !nrec_d || !T_d || !U_d || !sz ||
        !jAd || !jUd || !tc || !toff || !ubeg || !uend)
        return cudaErrorMemoryAllocation;
    SIVF_CUDA_TRY(cudaMemsetAsync(cnt, 0, sizeof(int64_t) * k, s));
    k_label_keys<<<blocks_gs(N), TPB, 0, s>>>(N, c->labels, lk0, lv0, cnt);
    note_launch();
    bool alt = false;
    SIVF_CUDA_TRY(radix_sort_pairs(lk0, lv0, lk1, lv1, N, bits_for((uint64_t)(k - 1)), &alt, ws, s));
    const uint32_t *perm = alt ? lv1 : lv0;
    k_recompute_flags<<<blocks_for(k), TPB, 0, s>>>(k, c->lam, cnt, flag);
    note_launch();
    SIVF_CUDA_TRY(scan_exclusive_i64(flag, rrank, k, nrec_d, ws, s));

    // u2: tuples of the recomputed clusters' members, in member order; a
    // stable sort by term then a stable sort by cluster rank leave them in
    // (rank, term, object) order; equal (rank, term) runs are summed in FP64
    k_member_tuples<<<blocks_gs(N), TPB, 0, s>>>(N, perm, c->labels, flag, c->row_ptr, tc);
    note_launch();
    SIVF_CUDA_TRY(scan_exclusive_i64(tc, toff, N, T_d, ws, s));
    uint32_t *sa_k = ws.take<uint32_t>(Tmax), *sa_v = ws.take<uint32_t>(Tmax);
    uint32_t *sb_k = ws.take<uint32_t>(Tmax), *sb_v = ws.take<uint32_t>(Tmax);
    double *part = ws.take<double>(Tmax);  // holds the tuples' terms and ranks before the piece sums
    uint32_t *tterm = reinterpret_cast<uint32_t *>(part), *trank = tterm + Tmax;
    float *tval = ws.take<float>(Tmax), *sval = ws.take<float>(Tmax);
    unsigned long long *key64 = ws.take<unsigned long long>(Tmax);
    int32_t *rank2clu = ws.take<int32_t>(k);
    int32_t *uterm = ws.take<int32_t>(Tmax);
    double *usum = ws.take<double>(Tmax);
    if (!sa_k || !sa_v || !sb_k || !sb_v || !part || !tval || !sval || !key64 || !rank2clu || !uterm || !usum)
        return cudaErrorMemoryAllocation;
    const int bits_r = bits_for((uint64_t)(k - 1));
    if (bits_r + c->bits_tl <= 32) {
        // one sort on (rank, local term) carrying the value bits
        k_rank2clu<<<blocks_for(k), TPB, 0, s>>>(k, flag, rrank, rank2clu);
        k_expand_packed<<<blocks_gs(N * 32), TPB, 0, s>>>(N, perm, c->labels, rrank, tc, toff, c->row_ptr, c->idx,
                                                            c->val, c->clu_doff, c->bits_tl, sa_k, sa_v);
        note_launch(2);
        bool a1 = false;
        SIVF_CUDA_TRY(radix_sort_pairs_dev(sa_k, sa_v, sb_k, sb_v, Tmax, T_d, bits_r + c->bits_tl, &a1, ws, s));
        k_unpack<<<blocks_gs(Tmax), TPB, 0, s>>>(Tmax, T_d, a1 ? sb_k : sa_k, a1 ? sb_v : sa_v, c->bits_tl, rank2clu,
                                                  c->clu_doff, key64, sval);
        note_launch();
    } else {
        // two stable sorts: by global term, then by rank
        k_expand<<<blocks_gs(N * 32), TPB, 0, s>>>(N, perm, c->labels, rrank, tc, toff, c->row_ptr, c->idx, c->val,
                                                     sa_k, sa_v, tterm, tval, trank);
        note_launch();
        bool a1 = false;
        SIVF_CUDA_TRY(radix_sort_pairs_dev(sa_k, sa_v, sb_k, sb_v, Tmax, T_d, c->bits_t, &a1, ws, s));
        uint32_t *x_v = a1 ? sb_v : sa_v;                           // tuple ids sorted by term
        uint32_t *y_k = a1 ? sa_k : sb_k, *y_v = a1 ? sa_v : sb_v;  // the free pair
        uint32_t *z_k = a1 ? sb_k : sa_k;                           // its ping-pong partner
        k_rank_keys<<<blocks_gs(Tmax), TPB, 0, s>>>(Tmax, T_d, x_v, trank, y_k, y_v);
        note_launch();
        bool a2 = false;
        SIVF_CUDA_TRY(radix_sort_pairs_dev(y_k, y_v, z_k, x_v, Tmax, T_d, bits_r, &a2, ws, s));
        const uint32_t *r_k = a2 ? z_k : y_k, *r_v = a2 ? x_v : y_v;
        k_compose<<<blocks_gs(Tmax), TPB, 0, s>>>(Tmax, T_d, r_k, r_v, tterm, tval, key64, sval);
        note_launch();
    }
    // the sort buffers are free again: run flags, run index, run position
    uint32_t *head = sa_k, *uidx = sa_v, *hpos = sb_k;
    k_heads<<<blocks_gs(Tmax), TPB, 0, s>>>(Tmax, T_d, key64, head);
    note_launch();
    SIVF_CUDA_TRY(scan_exclusive_u32_dev(head, uidx, Tmax, T_d, U_d, ws, s));
    SIVF_CUDA_TRY(cudaMemsetAsync(ubeg, 0, sizeof(int64_t) * (k + 1), s));  // empty-row clusters: no entries
    SIVF_CUDA_TRY(cudaMemsetAsync(uend, 0, sizeof(int64_t) * (k + 1), s));
    k_head_pos<<<blocks_gs(Tmax), TPB, 0, s>>>(Tmax, T_d, head, uidx, hpos);
    k_seg_pieces<<<blocks_gs((Tmax + 31) / 32 * 32), TPB, 0, s>>>(Tmax, T_d, key64, sval, part);
    k_seg_runs<<<blocks_gs(Tmax), TPB, 0, s>>>(Tmax, T_d, U_d, key64, hpos, part, uterm, usum, ubeg, uend);
    note_launch(3);
    SIVF_CUDA_TRY(cudaGetLastError());

    // u3/u4: new cluster-major rows (into the second buffer), copied back
    k_new_sizes<<<blocks_for(k), TPB, 0, s>>>(k, flag, rrank, ubeg, uend, c->coff[cur], sz);
    note_launch();
    SIVF_CUDA_TRY(row_offsets(c, sz, nw));
    k_write_rows<<<(unsigned)k, WR_THREADS, 0, s>>>(
        k, flag, rrank, ubeg, uend, uterm, usum, cnt, c->coff[cur], c->cterm[cur], c->cval[cur], c->snorm,
        c->coff[nw], c->cterm[nw], c->cval[nw], c->cclu, c->snorm_new, jAd, jUd, c->cap_c, &c->ctr->error);
    note_launch();
    SIVF_CUDA_TRY(finish_rows(c, jAd, jUd, T_d));
    ws.reset();

    // u5: rebuild the structured inverted file with lambda^[r]
    SIVF_CUDA_TRY(build_inverted_file(c));
    ws.reset();
    return cudaSuccess;
}
}  // namespace sivf

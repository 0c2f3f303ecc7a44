// Spatial ordering and packing of the sources for the near-field kernels.
//
// FP32C needs sources grouped into compact chunks so that float32 offsets from a
// per-chunk float64 origin keep the precision of close pairs.  The charges are
// ordered along the Hilbert curve of a 256^3 grid over the box (hilbert_key24) by a
// stable least-significant-digit radix sort (8-bit digits), then packed 128 at
// a time with the midpoint of each chunk's bounding box as its origin.
#include "launch.cuh"
#include "diffuse.cuh"

namespace psum {

constexpr int kSortThreads = 256;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kSortPerThread = 8;
constexpr int kSortTile = kSortThreads * kSortPerThread;   // 2048 keys per block
constexpr int kRadix = 256;

__global__ void k_curve_keys(const double* __restrict__ x, int64_t n, CurveBox box, uint32_t* __restrict__ keys) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) keys[i] = stored_key(x + 3 * i, box);
}

__global__ void __launch_bounds__(kSortThreads) k_sort_hist(const uint32_t* __restrict__ keys, int64_t n, int shift,
                                                            uint32_t* __restrict__ hist, int nblk) {
    __shared__ uint32_t cnt[kRadix];
    for (int d = threadIdx.x; d < kRadix; d += kSortThreads) cnt[d] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kSortTile;
    for (int k = 0; k < kSortPerThread; ++k) {
        const int64_t i = base + k * kSortThreads + threadIdx.x;
        if (i < n) atomicAdd(&cnt[(keys[i] >> shift) & (kRadix - 1)], 1u);
    }
    __syncthreads();
    for (int d = threadIdx.x; d < kRadix; d += kSortThreads) hist[(int64_t)d * nblk + blockIdx.x] = cnt[d];
}

// exclusive scan of `total` counts in place, one block of 1024 threads
__global__ void __launch_bounds__(1024) k_sort_scan(uint32_t* __restrict__ hist, int64_t total) {
    __shared__ uint32_t s[1024];
    const int64_t per = (total + 1023) / 1024;
    const int64_t b = threadIdx.x * per;
    const int64_t e = b + per < total ? b + per : total;
    uint32_t sum = 0;
    for (int64_t i = b; i < e; ++i) sum += hist[i];
    s[threadIdx.x] = sum;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {
        const uint32_t v = threadIdx.x >= o ? s[threadIdx.x - o] : 0u;
        __syncthreads();
        s[threadIdx.x] += v;
        __syncthreads();
    }
    uint32_t run = s[threadIdx.x] - sum;
    for (int64_t i = b; i < e; ++i) {
        const uint32_t v = hist[i];
        hist[i] = run;
        run += v;
    }
}

// Stable scatter: warp w of block b owns keys [b*T + w*256, +256) and walks them in
// order, 32 at a time; equal digits inside a step are ranked by lane.
__global__ void __launch_bounds__(kSortThreads) k_sort_scatter(const uint32_t* __restrict__ kin,
                                                               const uint32_t* __restrict__ vin, int64_t n, int shift,
                                                               const uint32_t* __restrict__ offs, int nblk,
                                                               uint32_t* __restrict__ kout,
                                                               uint32_t* __restrict__ vout) {
    __shared__ uint32_t wcnt[kSortWarps][kRadix];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < kSortWarps * kRadix; i += kSortThreads) (&wcnt[0][0])[i] = 0;
    __syncthreads();
    const int64_t wbase = (int64_t)blockIdx.x * kSortTile + w * (kSortPerThread * 32);
    for (int k = 0; k < kSortPerThread; ++k) {
        const int64_t i = wbase + k * 32 + lane;
        if (i < n) atomicAdd(&wcnt[w][(kin[i] >> shift) & (kRadix - 1)], 1u);
    }
    __syncthreads();
    for (int d = threadIdx.x; d < kRadix; d += kSortThreads) {
        uint32_t run = offs[(int64_t)d * nblk + blockIdx.x];
        for (int ww = 0; ww < kSortWarps; ++ww) {
            const uint32_t c = wcnt[ww][d];
            wcnt[ww][d] = run;
            run += c;
        }
    }
    __syncthreads();
    const uint32_t lt = (1u << lane) - 1u;
    for (int k = 0; k < kSortPerThread; ++k) {
        const int64_t i = wbase + k * 32 + lane;
        const bool valid = i < n;
        const uint32_t key = valid ? kin[i] : 0u;
        const uint32_t dig = valid ? ((key >> shift) & (kRadix - 1)) : (uint32_t)(kRadix + lane);
        const uint32_t peers = __match_any_sync(0xffffffffu, dig);
        const uint32_t rank = __popc(peers & lt);
        uint32_t pos = 0;
        if (valid) pos = wcnt[w][dig] + rank;
        __syncwarp();
        if (valid && rank == 0) wcnt[w][dig] += __popc(peers);
        __syncwarp();
        if (valid) {
            kout[pos] = key;
            vout[pos] = vin ? vin[i] : (uint32_t)i;     // no values: the input positions
        }
    }
}

// One block per group of kNearChunk sorted positions: the bounding-box midpoint is the
// float64 origin, stored with the group radius (largest distance of a point from it);
// each point's offset from the origin is split into a float32 hi part and the float32
// rounding remainder lo, packed two float4 each: (x,x,y,y),(z,z,q,q) and (xl,xl,yl,yl),(zl,zl,ql,ql)
// (ql = q - float(q), read only by the float-float kernels).
// Padding points (s >= n) get q = 0 and the origin: a far unit's targets all lie outside the group, off its
// origin (any other place may be a charge's in some box: 1/0 there, times 0, is no number), and a near unit
// takes K(0) = 0.  `ext` (optional) receives each group's bounding-box half extents about its origin.
// With a group table (batches) group g covers the sorted positions
// [grp_start[g], grp_start[g] + grp_count[g]); without one, [128 g, min(128 (g+1), n)).
//
// float32 charges carry the rounding error along the group (in sorted order): each charge absorbs
// the error carried so far, so the group's float32 charges sum to its float64 total up to one
// rounding; a non-neutral rounding residue would add the potential of a net charge over all images
// to every target.  The recurrence v = fl32(q - carry), carry += v - q is sequential; as a chain of
// five dependent float64 operations per charge it took 40-57 us whatever N was (GB300 issues one
// float64 warp instruction per scheduler in 64 cycles).  Here it runs in fixed point, as integers
// of 2^-61 of the group's largest power of two (exact for charges down to 2^-9 of the largest,
// rounded to 2^-62 of it below): the rounding position of each charge is taken from the charge
// itself, so a step is U = (Q + half) - c, c = half - (U & mask), three short 64-bit integer
// operations.  The whole warp then checks what the chain assumed: that no charge minus its carry
// left its binade and that no rounding was a tie (round-to-even would need one more bit); a group
// where it does not hold, or whose scale leaves float32's normal range, repeats the float64 chain.
// A group whose charges are all float32 numbers (+-1, say) needs no chain.
//
// A block of 128 threads packs one group, a point per thread: the offsets are some twenty operations
// a point on the float64 pipe, which the four schedulers of an SM then share (a warp per group took
// four times as long at small sizes).  Minima and maxima go over ordered integers.  Measured, a whole
// evaluation of 500 charges (+-1: no chain) and of 5001 (Gaussian): the chain in integers 106.4 -> 74.9 and
// 533 -> 492 us, a thread per point (with keys without division) 58.0 -> 51.5 and 419 -> 414 us.
__device__ __forceinline__ long long shfl_xor_ll(long long v, int off) {
    return (long long)__shfl_xor_sync(0xffffffffu, (unsigned long long)v, off);
}

constexpr int kPackThreads = kNearChunk;

__global__ void __launch_bounds__(kPackThreads) k_pack32(const double* __restrict__ x, const double* __restrict__ q,
                         const uint32_t* __restrict__ perm, int64_t n,
                         const int64_t* __restrict__ grp_start, const int* __restrict__ grp_count,
                         float4* __restrict__ pk_hi, float4* __restrict__ pk_lo, double* __restrict__ org,
                         double* __restrict__ xs, float4* __restrict__ ext) {
    constexpr int kWarps = kPackThreads / 32;
    __shared__ long long s_box[kWarps][7];          // lows, highs, then r^2
    __shared__ int s_emax[kWarps];
    __shared__ long long s_u[kNearChunk];           // Q + half
    __shared__ long long s_m[kNearChunk];           // mask, then the carry in
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    const int64_t grp = blockIdx.x;
    const int64_t s0 = grp_start ? grp_start[grp] : grp * kNearChunk;
    const int64_t s1 = grp_start ? s0 + grp_count[grp] : (grp + 1) * kNearChunk < n ? (grp + 1) * kNearChunk : n;
    const int cnt = s1 > s0 ? (int)(s1 - s0) : 0;
    const bool ok = tid < cnt;
    double px[3] = {0.0, 0.0, 0.0}, pq = 0.0;
    long long lo[3], hi[3];
    if (ok) {
        const int64_t i = perm ? (int64_t)perm[s0 + tid] : s0 + tid;
#pragma unroll
        for (int c = 0; c < 3; ++c) px[c] = x[3 * i + c];
        if (q) pq = q[i];                           // no charges: a pack of evaluation points
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const long long o = ordered_bits(__double_as_longlong(px[c]));
        lo[c] = ok ? o : 0x7fffffffffffffffll;
        hi[c] = ok ? o : -0x7fffffffffffffffll - 1;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const long long l2 = shfl_xor_ll(lo[c], off), h2 = shfl_xor_ll(hi[c], off);
            lo[c] = l2 < lo[c] ? l2 : lo[c];
            hi[c] = h2 > hi[c] ? h2 : hi[c];
        }
        if (lane == 0) {
            s_box[w][c] = lo[c];
            s_box[w][3 + c] = hi[c];
        }
    }
    const long long qb = __double_as_longlong(pq);
    const int e = exp_field(qb);
    {
        const int em = __reduce_max_sync(0xffffffffu, e);
        if (lane == 0) s_emax[w] = em;
    }
    // 24 significant bits and a normal float32 exponent, or zero
    const bool exact = pq == 0.0 || ((qb & 0x1fffffff) == 0 && e > 1023 - 126 && e < 1023 + 127);
    const bool chain = !__syncthreads_and(exact);   // also: s_box and s_emax are written
    double o[3], blo[3], bhi[3];
    int emax = 0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        lo[c] = s_box[0][c];
        hi[c] = s_box[0][3 + c];
#pragma unroll
        for (int k = 1; k < kWarps; ++k) {
            lo[c] = s_box[k][c] < lo[c] ? s_box[k][c] : lo[c];
            hi[c] = s_box[k][3 + c] > hi[c] ? s_box[k][3 + c] : hi[c];
        }
        blo[c] = __longlong_as_double(ordered_bits(lo[c]));
        bhi[c] = __longlong_as_double(ordered_bits(hi[c]));
        o[c] = cnt > 0 ? 0.5 * (blo[c] + bhi[c]) : 0.0;
    }
#pragma unroll
    for (int k = 0; k < kWarps; ++k) emax = s_emax[k] > emax ? s_emax[k] : emax;
    // the float32 charge (see above)
    float fq = (float)pq;
    if (chain) {
        bool held = emax >= kExpLo && emax <= kExpHi;        // uniform
        if (held) {
            const long long Q = fixed_charge(qb, emax);
            {
                const long long m = (1ll << dropped_bits(Q)) - 1;
                s_m[tid] = m;
                s_u[tid] = Q + ((m + 1) >> 1);
            }
            __syncthreads();
            if (tid == 0) {
                long long c = 0;
#pragma unroll 8
                for (int t = 0; t < kNearChunk; ++t) {       // past cnt: zero charges, not read back
                    const long long m = s_m[t];
                    s_m[t] = c;
                    c = diffuse_step(s_u[t], m, c);
                }
            }
            __syncthreads();
            bool fine;
            const long long V = diffuse_value(Q, s_m[tid], fine);
            fq = (float)((double)V * fixed_unit(emax));
            held = __syncthreads_and(fine || !ok);
        }
        if (!held) {
            double* s_q = reinterpret_cast<double*>(s_u);
            float* s_f = reinterpret_cast<float*>(s_m);
            s_q[tid] = pq;
            __syncthreads();
            if (tid == 0) {
                double carry = 0.0;
                for (int t = 0; t < cnt; ++t) {
                    const double qm = s_q[t];
                    const float v = (float)(qm - carry);
                    carry += (double)v - qm;
                    s_f[t] = v;
                }
            }
            __syncthreads();
            fq = s_f[tid];
        }
    }
    double r2 = 0.0;
    const int64_t s = grp * kNearChunk + tid;
    {
        float fx = 0.f, fy = 0.f, fz = 0.f, fc = 0.f, lx = 0.f, ly = 0.f, lz = 0.f, lq = 0.f;
        if (ok) {
            const double rx = px[0] - o[0], ry = px[1] - o[1], rz = px[2] - o[2];
            r2 = rx * rx + ry * ry + rz * rz;
            fx = (float)rx; fy = (float)ry; fz = (float)rz;
            lx = (float)(rx - (double)fx); ly = (float)(ry - (double)fy); lz = (float)(rz - (double)fz);
            fc = fq;
            lq = (float)(pq - (double)fq);        // the charge's float-float remainder (FF pair sums)
        }
        pk_hi[2 * s] = make_float4(fx, fx, fy, fy);
        pk_hi[2 * s + 1] = make_float4(fz, fz, fc, fc);
        pk_lo[2 * s] = make_float4(lx, lx, ly, ly);
        pk_lo[2 * s + 1] = make_float4(lz, lz, lq, lq);
    }
    if (xs) {
        xs[3 * s] = ok ? px[0] : 1.0e3;
        xs[3 * s + 1] = ok ? px[1] : 1.0e3;
        xs[3 * s + 2] = ok ? px[2] : 1.0e3;
    }
    // r^2 >= 0: its bits are in integer order too (a NaN, reported elsewhere, counts as 0)
    long long r2b = r2 >= 0.0 ? __double_as_longlong(r2) : 0ll;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const long long v = shfl_xor_ll(r2b, off);
        r2b = v > r2b ? v : r2b;
    }
    if (lane == 0) s_box[w][6] = r2b;
    __syncthreads();
    if (tid == 0) {
#pragma unroll
        for (int k = 1; k < kWarps; ++k) r2b = s_box[k][6] > r2b ? s_box[k][6] : r2b;
        org[4 * grp] = o[0]; org[4 * grp + 1] = o[1]; org[4 * grp + 2] = o[2];
        org[4 * grp + 3] = sqrt(__longlong_as_double(r2b));
    }
    if (ext && tid == 32) {
        // half extents of the bounding box about the origin, rounded up (never smaller)
        float h[3];
        for (int c = 0; c < 3; ++c) h[c] = cnt > 0 ? __double2float_ru(fmax(bhi[c] - o[c], o[c] - blo[c])) : 0.f;
        ext[grp] = make_float4(h[0], h[1], h[2], 0.f);
    }
}

__global__ void k_pack64(const double* __restrict__ x, const double* __restrict__ q, int64_t n, int64_t n_pad,
                         double4_32a* __restrict__ pk) {
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n_pad) return;
    if (s < n)
        pk[s] = make_double4_32a(x[3 * s], x[3 * s + 1], x[3 * s + 2], q ? q[s] : 0.0);
    else
        pk[s] = pad64(0.0);
}

// batches: packed point s of group g = s / 128 holds charge grp_start[g] + s % 128 if
// s % 128 < grp_count[g] (caller order inside each system), padding otherwise
__global__ void k_pack64_groups(const double* __restrict__ x, const double* __restrict__ q, int64_t n_pts,
                                const int64_t* __restrict__ grp_start, const int* __restrict__ grp_count,
                                double4_32a* __restrict__ pk) {
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n_pts) return;
    const int64_t g = s / kNearChunk;
    const int k = (int)(s - g * kNearChunk);
    if (k < grp_count[g]) {
        const int64_t i = grp_start[g] + k;
        pk[s] = make_double4_32a(x[3 * i], x[3 * i + 1], x[3 * i + 2], q[i]);
    } else {
        pk[s] = pad64(0.0);
    }
}

cudaError_t launch_pack64_groups(const double* x, const double* q, int64_t n_pts, const int64_t* grp_start,
                                 const int* grp_count, double4_32a* pk, cudaStream_t st) {
    k_pack64_groups<<<(unsigned)((n_pts + 255) / 256), 256, 0, st>>>(x, q, n_pts, grp_start, grp_count, pk);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
int sort_blocks(int64_t n) { return (int)((n + kSortTile - 1) / kSortTile); }

// Stable LSD radix sort of (key, value) pairs, 8 bits per pass over `passes` passes,
// ping-ponging (ka, va) -> (kb, vb) -> ...: the result ends in (ka, va) after an even
// number of passes and in (kb, vb) after an odd one; hist is scratch.  With va null the values are
// the input positions, and the passes after the first ping-pong between vb and `spare`.
cudaError_t launch_radix_sort(uint32_t* ka, uint32_t* va, uint32_t* kb, uint32_t* vb, uint32_t* hist, int64_t n,
                              int passes, cudaStream_t st, uint32_t* spare) {
    const int nblk = sort_blocks(n);
    uint32_t *ki = ka, *vi = va, *ko = kb, *vo = vb;
    for (int pass = 0; pass < passes; ++pass) {
        const int shift = 8 * pass;
        k_sort_hist<<<nblk, kSortThreads, 0, st>>>(ki, n, shift, hist, nblk);
        k_sort_scan<<<1, 1024, 0, st>>>(hist, (int64_t)kRadix * nblk);
        k_sort_scatter<<<nblk, kSortThreads, 0, st>>>(ki, vi, n, shift, hist, nblk, ko, vo);
        uint32_t* t = ki; ki = ko; ko = t;
        t = vi ? vi : spare;
        vi = vo;
        vo = t;
    }
    return cudaGetLastError();
}

// Small inputs by counting: a point's place is the number of points before it in (key, index)
// order, the order of the stable radix sort.  A block ranks 32 kPer points, kPer per lane; its 16
// warps count over every 16th block of four keys, which all lanes read as one 16-byte broadcast, and
// the warps' counts are added in shared memory.  The keys are stored as float32 numbers (24 bits,
// exact), so that a compare is a saturating subtraction, min(max(key - other, 0), 1), and its count
// another addition: two operations on the full-rate pipe, where integer compares and counts took
// seven cycles.  n^2 compares then stay below the radix sort's nine dependent launches (about 65 us
// at any size up to 1e5) until kRankMax points.
// A broadcast fills 32 lanes' registers, four cycles of an SM's load path for 16 bytes: with one
// point per lane that path bounds the kernel (20 000 points: 55 us).  A lane takes as many points as
// bring the launch to one block an SM or fewer: 157 blocks on 152 SMs take the time of two rounds
// (20 000 points with four per lane: 51 us).
constexpr int kRankWarps = 16;

// min(max(a - b, 0), 1) in one instruction
__device__ __forceinline__ float sub_sat(float a, float b) {
    float r;
    asm("sub.rn.sat.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}

template <int kPer>
__global__ void __launch_bounds__(32 * kRankWarps) k_rank_order(const float* __restrict__ keys, int n,
                                                                uint32_t* __restrict__ perm) {
    constexpr int kPoints = 32 * kPer;
    __shared__ int s_cnt[kRankWarps][kPoints];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int i0 = blockIdx.x * kPoints;
    const float4* k4 = reinterpret_cast<const float4*>(keys); // the key buffer starts on 256 bytes
    const int n4 = n >> 2, own = i0 >> 2;                     // whole blocks of four; the block's own
    float key[kPer], key1[kPer], c0[kPer], c1[kPer];          // counts below 2^24: exact
#pragma unroll
    for (int r = 0; r < kPer; ++r) {
        const int i = i0 + 32 * r + lane;
        key[r] = i < n ? keys[i] : 0.f;
        key1[r] = key[r] + 1.f;
        c0[r] = c1[r] = 0.f;
    }
    // points before the block's own: an equal key counts; after them: it does not
#pragma unroll 4
    for (int j = w; j < own; j += kRankWarps) {
        const float4 k = k4[j];
#pragma unroll
        for (int r = 0; r < kPer; ++r) {
            c0[r] += sub_sat(key1[r], k.x);
            c1[r] += sub_sat(key1[r], k.y);
            c0[r] += sub_sat(key1[r], k.z);
            c1[r] += sub_sat(key1[r], k.w);
        }
    }
#pragma unroll 4
    for (int j = own + kPoints / 4 + w; j < n4; j += kRankWarps) {
        const float4 k = k4[j];
#pragma unroll
        for (int r = 0; r < kPer; ++r) {
            c0[r] += sub_sat(key[r], k.x);
            c1[r] += sub_sat(key[r], k.y);
            c0[r] += sub_sat(key[r], k.z);
            c1[r] += sub_sat(key[r], k.w);
        }
    }
#pragma unroll
    for (int r = 0; r < kPer; ++r) {
        const int i = i0 + 32 * r + lane;
        int c = (int)(c0[r] + c1[r]);
        // the block's own points, each warp a share of them
        for (int j = i0 + w; j < i0 + kPoints && j < n; j += kRankWarps) c += keys[j] < key[r] || (keys[j] == key[r] && j < i);
        // keys past the last whole block of four, unless they are the block's own
        if (w == 0 && (n4 << 2) >= i0 + kPoints)
            for (int j = n4 << 2; j < n; ++j) c += keys[j] < key[r];
        s_cnt[w][32 * r + lane] = c;
    }
    __syncthreads();
    if (w < kPer) {
        const int i = i0 + 32 * w + lane;
        int r = 0;
#pragma unroll
        for (int k = 0; k < kRankWarps; ++k) r += s_cnt[k][32 * w + lane];
        if (i < n) perm[r] = (uint32_t)i;
    }
}

int curve_order_launches(int64_t n) { return n <= kRankMax ? 1 : 3 * 3; }

// The stable order of n points by their keys as stored_key wrote them to kb (which is overwritten):
// the permutation ends in va.
cudaError_t launch_curve_order(int64_t n, uint32_t* ka, uint32_t* va, uint32_t* kb, uint32_t* vb, uint32_t* hist,
                               cudaStream_t st) {
    if (n <= kRankMax) {
        const int per = (int)((n + 32 * kRankSms - 1) / (32 * kRankSms));
        const unsigned nb = (unsigned)((n + 32 * per - 1) / (32 * per));
        const float* keys = (const float*)kb;
        const auto kernel = per == 1 ? k_rank_order<1> : per == 2 ? k_rank_order<2> : per == 3 ? k_rank_order<3>
                                     : per == 4 ? k_rank_order<4> : k_rank_order<5>;
        kernel<<<nb, 32 * kRankWarps, 0, st>>>(keys, (int)n, va);
        return cudaGetLastError();
    }
    return launch_radix_sort(kb, nullptr, ka, va, hist, n, 3, st, vb);
}

// Keys and order of the points (callers whose keys do not come with the validation).
cudaError_t launch_curve_sort(const double* x, int64_t n, const double d[3], uint32_t* ka, uint32_t* va,
                               uint32_t* kb, uint32_t* vb, uint32_t* hist, cudaStream_t st) {
    const int bs = 256;
    k_curve_keys<<<(unsigned)((n + bs - 1) / bs), bs, 0, st>>>(x, n, curve_box(d, n), kb);
    return launch_curve_order(n, ka, va, kb, vb, hist, st);
}

cudaError_t launch_pack32(const double* x, const double* q, const uint32_t* perm, int64_t n, int64_t n_groups,
                          float4* pk_hi, float4* pk_lo, double* org, cudaStream_t st, double* xs, float4* ext) {
    k_pack32<<<(unsigned)n_groups, kPackThreads, 0, st>>>(x, q, perm, n, nullptr, nullptr, pk_hi, pk_lo, org, xs, ext);
    return cudaGetLastError();
}

cudaError_t launch_pack32_groups(const double* x, const double* q, const uint32_t* perm, int64_t n_groups,
                                 const int64_t* grp_start, const int* grp_count, float4* pk_hi, float4* pk_lo,
                                 double* org, cudaStream_t st, float4* ext) {
    k_pack32<<<(unsigned)n_groups, kPackThreads, 0, st>>>(x, q, perm, 0, grp_start, grp_count, pk_hi, pk_lo, org,
                                                          nullptr, ext);
    return cudaGetLastError();
}

cudaError_t launch_pack64(const double* x, const double* q, int64_t n, int64_t n_pad, double4_32a* pk, cudaStream_t st) {
    const int bs = 256;
    k_pack64<<<(unsigned)((n_pad + bs - 1) / bs), bs, 0, st>>>(x, q, n, n_pad, pk);
    return cudaGetLastError();
}

}  // namespace psum

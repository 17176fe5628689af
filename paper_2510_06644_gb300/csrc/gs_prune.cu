// A-9 gradient-reuse pruning (Sec. 4.1, Eq. 7), the change ratio of
// tile-Gaussian intersections, compaction, and A-10 keyframe-driven dynamic
// downsampling (Sec. 4.2) on sm_103a.
//
// Selection is a radix select on the unique 64-bit key (score bits << 32 |
// id): digits of 11, 11 and 10 bits settle the score, and 11-bit digits of the
// bits that ids below n have settle ties.  A pass needs only the histogram of
// the pass before it, which every CTA scans for itself, so no pass needs a
// pick launch or a host round trip.  Scores are non-negative, so their float
// bits order like their values.
#include "gs_internal.cuh"

namespace gs {

typedef unsigned long long u64;

#define PR_THREADS 256
#define SEL_THREADS 512
#define SEL_BINS 2048        // 11-bit digits
#define SEL_MAX_PASSES 6     // 3 of the score, at most 3 of the id
#define KEEP_PER_THREAD 8
#define KEEP_STEP (PR_THREADS * KEEP_PER_THREAD)
#define KEEP_MAX_CHUNKS 2048

__device__ __forceinline__ u64 score_key(float mu, float sig, int64_t k, float lam) {
    // Eq. 7 in float32: product rounded, then sum rounded (no fused multiply-add)
    const float s = __fadd_rn(mu, __fmul_rn(lam, sig));
    return ((u64)__float_as_uint(s) << 32) | (u64)(uint32_t)k;
}

// ---------------------------------------------------------------------------
// Selection
// ---------------------------------------------------------------------------
// One digit: `bits` wide, its lowest bit at `shift`.
struct Digit {
    int shift, bits;
};

struct SelPasses {
    Digit d[SEL_MAX_PASSES];
    int count;
};

// The digits for ids below n: bits that no id has are not passed over (1M ids:
// five passes, at most 2048 ids: four).
static SelPasses sel_passes(int64_t n) {
    SelPasses P;
    P.d[0] = {53, 11};
    P.d[1] = {42, 11};
    P.d[2] = {32, 10};
    P.count = 3;
    int top = 0;
    while (top < 32 && ((n - 1) >> top) > 0) ++top;
    while (top > 0) {
        const int w = top < 11 ? top : 11;
        top -= w;
        P.d[P.count++] = {top, w};
    }
    return P;
}

// What the passes so far have fixed: the key prefix, the rank that is left
// inside it, and whether the threshold is known.
enum { SEL_OPEN = 0, SEL_DONE = 1, SEL_NONE = 2 };
struct SelState {
    u64 prefix, remaining, status;
};

struct SelArgs {
    const float* terms;
    uint8_t* mask;
    int64_t n;
    float lam, frac;
    int64_t max_select;
    SelState* state;     // [pass]: before that pass
    unsigned int* hist;  // [pass][SEL_BINS]
    int pass;            // digits of this pass and of the one before it
    Digit d, prev;
    int vec;             // terms 16-byte and mask 4-byte aligned
};

// m = min(floor(frac * n_active), max_select): rank (1-based) of the largest
// selected key.
__device__ __forceinline__ u64 select_count(u64 n_active, float frac, int64_t max_select) {
    const double m = floor((double)frac * (double)n_active);
    u64 mm = (u64)m;
    if ((int64_t)mm > max_select) mm = (u64)(max_select < 0 ? 0 : max_select);
    return mm;
}

// The state before pass p, from the state before pass p - 1 and that pass's
// histogram: every CTA scans the 2048 counts (four a thread) and block 0 stores
// the result for the next launch.  The first histogram also counts the active
// Gaussians.  If all keys of the chosen bin are selected, the digits below
// cannot matter and the threshold is the bin's last key.
__device__ __forceinline__ SelState sel_advance(const SelArgs& A) {
    const int p = A.pass;
    __shared__ SelState s_new;
    __shared__ u64 s_warp[SEL_THREADS / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    SelState S = {0, 0, SEL_OPEN};
    if (p == 0) return S;
    if (p > 1) S = A.state[p - 1];
    if (S.status == SEL_OPEN) {
        const unsigned int* hp = A.hist + (size_t)(p - 1) * SEL_BINS + 4 * threadIdx.x;
        const uint4 h = make_uint4(hp[0], hp[1], hp[2], hp[3]);  // (a workspace may be 8-byte aligned)
        const u64 mine = (u64)h.x + h.y + h.z + h.w;
        u64 x = mine;
        for (int o = 1; o < 32; o <<= 1) {
            const u64 y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s_warp[wid] = x;
        __syncthreads();
        u64 before = 0, total = 0;
        for (int w = 0; w < SEL_THREADS / 32; ++w) {
            if (w < wid) before += s_warp[w];
            total += s_warp[w];
        }
        if (p == 1) {
            S.remaining = select_count(total, A.frac, A.max_select);
            if (S.remaining == 0) S.status = SEL_NONE;
            else if (S.remaining >= total) S = {~0ull, S.remaining, SEL_DONE};
        }
        if (S.status == SEL_OPEN) {
            u64 cum = before + x - mine;  // counts below this thread's bins
            if (cum < S.remaining && S.remaining <= cum + mine) {
                unsigned int c = h.x, j = 0;
                if (cum + c < S.remaining) { cum += c; c = h.y; j = 1; }
                if (j == 1 && cum + c < S.remaining) { cum += c; c = h.z; j = 2; }
                if (j == 2 && cum + c < S.remaining) { cum += c; c = h.w; j = 3; }
                SelState N = {S.prefix | ((u64)(threadIdx.x * 4 + j) << A.prev.shift), S.remaining - cum, SEL_OPEN};
                if (N.remaining == c) {
                    N.prefix |= (1ull << A.prev.shift) - 1ull;
                    N.status = SEL_DONE;
                }
                s_new = N;
            }
            __syncthreads();
            S = s_new;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) A.state[p] = S;
    return S;
}

// The keys of ids [4 q, 4 q + 4) and which of them are unmasked (bit j).
__device__ __forceinline__ unsigned int load_keys(const SelArgs& A, int64_t q, u64* key) {
    const int64_t k = 4 * q;
    unsigned int live = 0;
    if (A.vec && k + 4 <= A.n) {
        const uchar4 m = reinterpret_cast<const uchar4*>(A.mask)[q];
        const float4 a = __ldg(reinterpret_cast<const float4*>(A.terms) + 2 * q);
        const float4 b = __ldg(reinterpret_cast<const float4*>(A.terms) + 2 * q + 1);
        key[0] = score_key(a.x, a.y, k, A.lam);
        key[1] = score_key(a.z, a.w, k + 1, A.lam);
        key[2] = score_key(b.x, b.y, k + 2, A.lam);
        key[3] = score_key(b.z, b.w, k + 3, A.lam);
        live = (m.x ? 0u : 1u) | (m.y ? 0u : 2u) | (m.z ? 0u : 4u) | (m.w ? 0u : 8u);
    } else {
        for (int j = 0; j < 4; ++j) {
            key[j] = 0;
            if (k + j < A.n && A.mask[k + j] == 0) {
                key[j] = score_key(A.terms[2 * (k + j)], A.terms[2 * (k + j) + 1], k + j, A.lam);
                live |= 1u << j;
            }
        }
    }
    return live;
}

// Histogram of one digit over the unmasked keys under the prefix.  The scores
// come from L2 in every pass (8 bytes a Gaussian), so a pass is short and the
// launches count: eight 8-bit passes, each re-deriving the whole prefix by one
// thread, took 69 us with their count and mask launches at 1M Gaussians;
// these take 36.  Many scores are equal (zero where nothing was blended), so a warp
// adds its first key's bin once for all lanes that share it.
__global__ void __launch_bounds__(SEL_THREADS) k_select_pass(const __grid_constant__ SelArgs A) {
    __shared__ unsigned int sh[SEL_BINS];
    for (int i = threadIdx.x; i < SEL_BINS; i += SEL_THREADS) sh[i] = 0;
    const int p = A.pass;
    const SelState S = sel_advance(A);
    if (S.status != SEL_OPEN) return;  // the same in every thread of the grid
    __syncthreads();
    const Digit d = A.d;
    const unsigned int bin_mask = (1u << d.bits) - 1u;
    const int top = A.prev.shift;
    const int lane = threadIdx.x & 31;
    const int64_t nq = (A.n + 3) >> 2;
    const int64_t stride = (int64_t)gridDim.x * SEL_THREADS;
    for (int64_t q0 = (int64_t)blockIdx.x * SEL_THREADS + (threadIdx.x & ~31); q0 < nq; q0 += stride) {
        u64 key[4] = {0, 0, 0, 0};
        const unsigned int live = q0 + lane < nq ? load_keys(A, q0 + lane, key) : 0u;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const bool take = (live >> j & 1u) && (p == 0 || ((key[j] ^ S.prefix) >> top) == 0);
            const unsigned int any = __ballot_sync(0xffffffffu, take);
            if (any == 0) continue;
            const int first = __ffs(any) - 1;
            const unsigned int bin = (unsigned int)(key[j] >> d.shift) & bin_mask;
            const unsigned int b0 = __shfl_sync(0xffffffffu, bin, first);
            const unsigned int same = __ballot_sync(0xffffffffu, take && bin == b0);
            if (lane == first) atomicAdd(&sh[b0], (unsigned int)__popc(same));
            else if (take && bin != b0) atomicAdd(&sh[bin], 1u);
        }
    }
    __syncthreads();
    unsigned int* h = A.hist + (size_t)p * SEL_BINS;
    for (int i = threadIdx.x; i < SEL_BINS; i += SEL_THREADS)
        if (sh[i]) atomicAdd(h + i, sh[i]);
}

__global__ void __launch_bounds__(SEL_THREADS) k_select_mask(const __grid_constant__ SelArgs A) {
    const SelState S = sel_advance(A);
    if (S.status == SEL_NONE) return;
    const int64_t nq = (A.n + 3) >> 2;
    for (int64_t q = (int64_t)blockIdx.x * SEL_THREADS + threadIdx.x; q < nq; q += (int64_t)gridDim.x * SEL_THREADS) {
        u64 key[4];
        const unsigned int live = load_keys(A, q, key);
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if ((live >> j & 1u) && key[j] <= S.prefix) A.mask[4 * q + j] = 1;
    }
}

// ---------------------------------------------------------------------------
// Compaction map: exclusive scan of (mask == 0) in id order
// ---------------------------------------------------------------------------
// Bit j: id k + j exists and is kept.
__device__ __forceinline__ unsigned int keep_bits(const uint8_t* __restrict__ mask, int64_t k, int64_t n, bool vec) {
    unsigned int keep = 0;
    if (vec && k + KEEP_PER_THREAD <= n) {
        const uint2 m = __ldg(reinterpret_cast<const uint2*>(mask + k));
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            keep |= ((m.x >> (8 * j)) & 0xffu) ? 0u : 1u << j;
            keep |= ((m.y >> (8 * j)) & 0xffu) ? 0u : 16u << j;
        }
    } else {
        for (int j = 0; j < KEEP_PER_THREAD; ++j)
            if (k + j < n && mask[k + j] == 0) keep |= 1u << j;
    }
    return keep;
}

// Kept ids of each chunk.  A chunk is a multiple of 2048 ids such that there
// are at most 2048 chunks: few enough that k_keep_write sums those before its
// own itself, without a scan launch between the two.
__global__ void __launch_bounds__(PR_THREADS) k_keep_count(const uint8_t* __restrict__ mask, int64_t n, int64_t chunk,
                                                           bool vec, u64* __restrict__ partial) {
    __shared__ unsigned int s;
    if (threadIdx.x == 0) s = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * chunk;
    unsigned int c = 0;
    for (int64_t o = (int64_t)threadIdx.x * KEEP_PER_THREAD; o < chunk; o += KEEP_STEP)
        c += __popc(keep_bits(mask, base + o, n, vec));
    c = __reduce_add_sync(0xffffffffu, c);
    if ((threadIdx.x & 31) == 0) atomicAdd(&s, c);
    __syncthreads();
    if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

__global__ void __launch_bounds__(PR_THREADS) k_keep_write(const uint8_t* __restrict__ mask, int64_t n, int64_t chunk,
                                                           bool vec, bool vec_out, const u64* __restrict__ partial,
                                                           uint32_t* __restrict__ map, int64_t* __restrict__ n_kept) {
    __shared__ u64 s_before;
    __shared__ unsigned int s_warp[2][PR_THREADS / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_before = 0;
    __syncthreads();
    u64 part = 0;
    for (unsigned int b = threadIdx.x; b < blockIdx.x; b += PR_THREADS) part += partial[b];
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    if (lane == 0 && part) atomicAdd(&s_before, part);
    __syncthreads();
    u64 off = s_before;
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *n_kept = (int64_t)(off + partial[blockIdx.x]);
    const int64_t base = (int64_t)blockIdx.x * chunk;
    int buf = 0;
    for (int64_t o = 0; o < chunk && base + o < n; o += KEEP_STEP, buf ^= 1) {
        const int64_t k = base + o + (int64_t)threadIdx.x * KEEP_PER_THREAD;
        const unsigned int keep = keep_bits(mask, k, n, vec);
        const unsigned int mine = __popc(keep);
        unsigned int x = mine;
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned int y = __shfl_up_sync(0xffffffffu, x, d);
            if (lane >= d) x += y;
        }
        if (lane == 31) s_warp[buf][wid] = x;
        __syncthreads();  // the other buffer is read before the next barrier at the latest
        unsigned int before = 0, total = 0;
#pragma unroll
        for (int w = 0; w < PR_THREADS / 32; ++w) {
            const unsigned int t = s_warp[buf][w];
            before += w < wid ? t : 0u;
            total += t;
        }
        uint32_t to[KEEP_PER_THREAD], at = (uint32_t)off + before + x - mine;
#pragma unroll
        for (int j = 0; j < KEEP_PER_THREAD; ++j) to[j] = (keep >> j & 1u) ? at++ : 0xFFFFFFFFu;
        if (vec_out && k + KEEP_PER_THREAD <= n) {
            uint4* dst = reinterpret_cast<uint4*>(map + k);
            dst[0] = make_uint4(to[0], to[1], to[2], to[3]);
            dst[1] = make_uint4(to[4], to[5], to[6], to[7]);
        } else {
#pragma unroll
            for (int j = 0; j < KEEP_PER_THREAD; ++j)
                if (k + j < n) map[k + j] = to[j];
        }
        off += total;
    }
}

// ---------------------------------------------------------------------------
// Change ratio
// ---------------------------------------------------------------------------
// |rect_a| + |rect_b| - 2 |rect_a & rect_b| and |rect_a| summed over Gaussians.
template <int DT>
__global__ void __launch_bounds__(PR_THREADS) k_change(gs_camera cam, float alpha_min, const void* __restrict__ sa,
                                                       const void* __restrict__ sb, int64_t n, u64* __restrict__ acc,
                                                       float* __restrict__ out) {
    __shared__ u64 s_acc[2];
    if (threadIdx.x < 2) s_acc[threadIdx.x] = 0;
    __syncthreads();
    const Grid grid = make_grid(cam);
    u64 sym = 0, na = 0;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        int ax0, ax1, ay0, ay1, bx0, bx1, by0, by1;
        const int ca = tile_rect(grid, load_geom<DT>(sa, (uint32_t)k), alpha_min, ax0, ax1, ay0, ay1);
        const int cb = tile_rect(grid, load_geom<DT>(sb, (uint32_t)k), alpha_min, bx0, bx1, by0, by1);
        int inter = 0;
        if (ca > 0 && cb > 0) {
            const int ix = min(ax1, bx1) - max(ax0, bx0), iy = min(ay1, by1) - max(ay0, by0);
            if (ix > 0 && iy > 0) inter = ix * iy;
        }
        sym += (u64)(ca + cb - 2 * inter);
        na += (u64)ca;
    }
    for (int o = 16; o > 0; o >>= 1) {
        sym += __shfl_xor_sync(0xffffffffu, sym, o);
        na += __shfl_xor_sync(0xffffffffu, na, o);
    }
    if ((threadIdx.x & 31) == 0 && (sym | na)) {
        atomicAdd(&s_acc[0], sym);
        atomicAdd(&s_acc[1], na);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (s_acc[0]) atomicAdd(acc, s_acc[0]);
        if (s_acc[1]) atomicAdd(acc + 1, s_acc[1]);
        __threadfence();
        if (atomicAdd(acc + 2, 1ull) == gridDim.x - 1) {  // every block has added its share
            const u64 tot = atomicAdd(acc, 0ull);
            const double in_a = (double)atomicAdd(acc + 1, 0ull);
            *out = (float)((double)tot / (in_a > 1.0 ? in_a : 1.0));
        }
    }
}

__host__ __device__ constexpr int compact_rows(int w) { return w == 1 ? 1024 : w == 2 ? 512 : 256; }

// Rows of a parameter array to their places in the compacted one; W floats a
// row (1 to 4 as constants: 0 takes any width).  A block moves ROWS rows, so the
// row of an element is a 32-bit division by a constant and every load of the
// block is in flight at once, three or four elements a thread (1M rows of 3
// floats, a 64-bit division an element 8.5 us, now 5.5; 3M rows of 1, 256 rows a
// block 10.9, now 5.4).
template <int W>
__global__ void __launch_bounds__(256) k_compact(const float* __restrict__ src, int64_t n, int width,
                                                 const uint32_t* __restrict__ map, float* __restrict__ dst) {
    if (W == 0) {
        const int64_t total = n * (int64_t)width;
        for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < total;
             q += (int64_t)gridDim.x * blockDim.x) {
            const int64_t k = q / width;
            const uint32_t to = map[k];
            if (to != 0xFFFFFFFFu) dst[(int64_t)to * width + (q - k * width)] = src[q];
        }
        return;
    }
    constexpr int WC = W > 0 ? W : 1, ROWS = compact_rows(W), E = WC * ROWS / 256;
    for (int64_t r0 = (int64_t)blockIdx.x * ROWS; r0 < n; r0 += (int64_t)gridDim.x * ROWS) {
        const unsigned int rows = (unsigned int)(n - r0 < ROWS ? n - r0 : ROWS);
        uint32_t to[E];
        float v[E];
#pragma unroll
        for (int j = 0; j < E; ++j) {
            const unsigned int e = threadIdx.x + 256u * j;
            const bool in = e < rows * WC;
            to[j] = in ? __ldg(map + r0 + e / WC) : 0xFFFFFFFFu;
            v[j] = in ? __ldg(src + r0 * WC + e) : 0.f;
        }
#pragma unroll
        for (int j = 0; j < E; ++j)
            if (to[j] != 0xFFFFFFFFu) dst[(int64_t)to[j] * WC + (threadIdx.x + 256u * j) % WC] = v[j];
    }
}

__global__ void __launch_bounds__(256) k_gather(const float* __restrict__ full, int C, int W, int H, int sx, int sy,
                                                float* __restrict__ out) {
    const int Ws = (W + sx - 1) / sx, Hs = (H + sy - 1) / sy;
    const int64_t total = (int64_t)C * Ws * Hs;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < total; q += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(q % Ws);
        const int64_t r = q / Ws;
        const int j = (int)(r % Hs);
        const int c = (int)(r / Hs);
        out[q] = full[((int64_t)c * H + (int64_t)j * sy) * W + (int64_t)i * sx];
    }
}

static size_t a256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace gs

using namespace gs;

extern "C" int32_t gs_next_interval(const gs_config* cfg, int32_t K, float change_ratio) {
    if (!cfg || K < 1) return 1;
    int32_t nk = change_ratio > cfg->change_thr ? K / 2 : 2 * K;
    if (nk < 1) nk = 1;
    if (nk > cfg->k_max) nk = cfg->k_max;
    return nk;
}

extern "C" gs_status gs_prune(const gs_config* cfg, const float* score_terms, int64_t n, uint8_t* mask_inout,
                              int iter_in_interval, int* k_inout, float change_ratio, int64_t max_select,
                              uint32_t* compact_map_out, int64_t* n_kept_out, void* workspace,
                              size_t* workspace_bytes, gs_stream stream) {
    if (!cfg || !workspace_bytes || !k_inout) return set_error(GS_ERR_INVALID_ARG, "config, k_inout or workspace_bytes NULL");
    if (n < 0 || n > (int64_t)0xFFFFFFF0LL) return set_error(GS_ERR_INVALID_ARG, "bad Gaussian count");
    if (*k_inout < 1) return set_error(GS_ERR_INVALID_ARG, "interval K must be >= 1");
    const int64_t steps = (n + KEEP_STEP - 1) / KEEP_STEP;
    const int64_t chunk = KEEP_STEP * ((steps + KEEP_MAX_CHUNKS - 1) / KEEP_MAX_CHUNKS);
    const size_t hist_bytes = SEL_MAX_PASSES * SEL_BINS * sizeof(unsigned int);
    const size_t off_state = a256(hist_bytes);
    const size_t off_part = a256(off_state + (SEL_MAX_PASSES + 1) * sizeof(SelState));
    const size_t need = a256(off_part + sizeof(u64) * KEEP_MAX_CHUNKS);
    if (!workspace) { *workspace_bytes = need; return GS_OK; }
    if (*workspace_bytes < need) return set_error(GS_ERR_WORKSPACE, "workspace %zu < %zu", *workspace_bytes, need);
    cudaStream_t st = (cudaStream_t)stream;
    char* ws = (char*)workspace;
    gs_status s;
    if (iter_in_interval == 0) {
        if (n == 0) return GS_OK;
        if (!score_terms || !mask_inout) return set_error(GS_ERR_INVALID_ARG, "score_terms or mask NULL");
        SelArgs A;
        A.terms = score_terms;
        A.mask = mask_inout;
        A.n = n;
        A.lam = cfg->lambda_score;
        A.frac = cfg->prune_frac;
        A.max_select = max_select;
        A.state = (SelState*)(ws + off_state);
        A.hist = (unsigned int*)ws;
        A.vec = ((uintptr_t)score_terms & 15) == 0 && ((uintptr_t)mask_inout & 3) == 0;
        const SelPasses P = sel_passes(n);
        if (cudaMemsetAsync(ws, 0, P.count * SEL_BINS * sizeof(unsigned int), st) != cudaSuccess)
            return set_error(GS_ERR_CUDA, "memset prune state");
        // four ids a thread; two CTAs an SM at most, so that few histograms are merged
        const int sms = num_sms();
        const int64_t want = (n + 4 * SEL_THREADS - 1) / (4 * SEL_THREADS);
        const unsigned nb = (unsigned)(want < 2 * sms ? want : 2 * sms);
        A.prev = {0, 0};
        for (A.pass = 0; A.pass < P.count; ++A.pass) {
            A.d = P.d[A.pass];
            k_select_pass<<<nb, SEL_THREADS, 0, st>>>(A);
            if ((s = check_launch("k_select_pass")) != GS_OK) return s;
            A.prev = A.d;
        }
        k_select_mask<<<nb, SEL_THREADS, 0, st>>>(A);
        return check_launch("k_select_mask");
    }
    if (iter_in_interval == *k_inout) {
        if (!compact_map_out || !n_kept_out || (n > 0 && !mask_inout))
            return set_error(GS_ERR_INVALID_ARG, "compact map, n_kept or mask NULL");
        if (n == 0) {
            if (cudaMemsetAsync(n_kept_out, 0, sizeof(int64_t), st) != cudaSuccess) return set_error(GS_ERR_CUDA, "memset");
        } else {
            u64* part = (u64*)(ws + off_part);
            const unsigned nchunk = (unsigned)((n + chunk - 1) / chunk);
            const bool vec = ((uintptr_t)mask_inout & 7) == 0, vec_out = ((uintptr_t)compact_map_out & 15) == 0;
            k_keep_count<<<nchunk, PR_THREADS, 0, st>>>(mask_inout, n, chunk, vec, part);
            if ((s = check_launch("k_keep_count")) != GS_OK) return s;
            k_keep_write<<<nchunk, PR_THREADS, 0, st>>>(mask_inout, n, chunk, vec, vec_out, part, compact_map_out,
                                                       n_kept_out);
            if ((s = check_launch("k_keep_write")) != GS_OK) return s;
        }
        *k_inout = gs_next_interval(cfg, *k_inout, change_ratio);
        return GS_OK;
    }
    return GS_OK;
}

extern "C" gs_status gs_change_ratio(const gs_config* cfg, const gs_camera* cam, int rec_dtype, const void* splats_a,
                                     const void* splats_b,
                                     int64_t n, void* workspace, size_t* workspace_bytes, float* ratio_out,
                                     gs_stream stream) {
    if (!cfg || !cam || !workspace_bytes) return set_error(GS_ERR_INVALID_ARG, "config, camera or workspace_bytes NULL");
    if (cam->width <= 0 || cam->height <= 0 || cam->sx < 1 || cam->sy < 1)
        return set_error(GS_ERR_INVALID_ARG, "bad camera size or stride");
    if (rec_dtype != GS_F32 && rec_dtype != GS_BF16 && rec_dtype != GS_F16)
        return set_error(GS_ERR_INVALID_ARG, "bad record dtype");
    if (n < 0) return set_error(GS_ERR_INVALID_ARG, "bad Gaussian count");
    const size_t need = 256;
    if (!workspace) { *workspace_bytes = need; return GS_OK; }
    if (*workspace_bytes < need) return set_error(GS_ERR_WORKSPACE, "workspace %zu < %zu", *workspace_bytes, need);
    if (!ratio_out || (n > 0 && (!splats_a || !splats_b))) return set_error(GS_ERR_INVALID_ARG, "NULL pointer");
    cudaStream_t st = (cudaStream_t)stream;
    u64* acc = (u64*)workspace;
    if (cudaMemsetAsync(acc, 0, 3 * sizeof(u64), st) != cudaSuccess) return set_error(GS_ERR_CUDA, "memset");
    const int sms = num_sms();
    const int64_t want = (n + PR_THREADS - 1) / PR_THREADS;
    const unsigned nb = (unsigned)(want < 1 ? 1 : want < 4 * sms ? want : 4 * sms);
    if (rec_dtype == GS_F32)
        k_change<GS_F32><<<nb, PR_THREADS, 0, st>>>(*cam, cfg->alpha_min, splats_a, splats_b, n, acc, ratio_out);
    else if (rec_dtype == GS_BF16)
        k_change<GS_BF16><<<nb, PR_THREADS, 0, st>>>(*cam, cfg->alpha_min, splats_a, splats_b, n, acc, ratio_out);
    else
        k_change<GS_F16><<<nb, PR_THREADS, 0, st>>>(*cam, cfg->alpha_min, splats_a, splats_b, n, acc, ratio_out);
    return check_launch("k_change");
}

extern "C" gs_status gs_compact(const float* src, int64_t n, int32_t width, const uint32_t* compact_map, float* dst,
                                gs_stream stream) {
    if (n < 0 || width < 1) return set_error(GS_ERR_INVALID_ARG, "bad size");
    if (n == 0) return GS_OK;
    if (!src || !compact_map || !dst) return set_error(GS_ERR_INVALID_ARG, "NULL pointer");
    const int sms = num_sms();
    const int rows = compact_rows(width);
    const int64_t want = width <= 4 ? (n + rows - 1) / rows : (n * width + 255) / 256;
    const int64_t cap = (int64_t)(width <= 4 ? 64 : 8) * sms;
    const unsigned nb = (unsigned)(want < cap ? want : cap);
    cudaStream_t st = (cudaStream_t)stream;
    if (width == 1) k_compact<1><<<nb, 256, 0, st>>>(src, n, width, compact_map, dst);
    else if (width == 2) k_compact<2><<<nb, 256, 0, st>>>(src, n, width, compact_map, dst);
    else if (width == 3) k_compact<3><<<nb, 256, 0, st>>>(src, n, width, compact_map, dst);
    else if (width == 4) k_compact<4><<<nb, 256, 0, st>>>(src, n, width, compact_map, dst);
    else k_compact<0><<<nb, 256, 0, st>>>(src, n, width, compact_map, dst);
    return check_launch("k_compact");
}

extern "C" gs_status gs_downsample(int64_t frame_idx, int64_t last_kf_idx, int is_keyframe, int m, int32_t* sx,
                                   int32_t* sy, const float* target_full, int32_t channels, int32_t W, int32_t H,
                                   float* target_out, gs_stream stream) {
    if (!sx || !sy) return set_error(GS_ERR_INVALID_ARG, "sx or sy NULL");
    if (is_keyframe) {
        *sx = 1;
        *sy = 1;
    } else {
        if (m < 2 || (m & (m - 1)) != 0) return set_error(GS_ERR_INVALID_ARG, "m must be a power of two >= 2");
        if (frame_idx <= last_kf_idx) return set_error(GS_ERR_INVALID_ARG, "frame must follow its keyframe");
        // R0/R = max(16 / m^(n-k-1), 4)
        const int64_t e = frame_idx - last_kf_idx - 1;
        int64_t ratio = 16;
        for (int64_t q = 0; q < e && ratio > 4; ++q) ratio /= m;
        if (ratio < 4) ratio = 4;
        if (ratio == 16) { *sx = 4; *sy = 4; }
        else if (ratio == 8) { *sx = 4; *sy = 2; }
        else { *sx = 2; *sy = 2; }
    }
    if (!target_full) return GS_OK;
    if (!target_out || channels < 1 || W < 1 || H < 1) return set_error(GS_ERR_INVALID_ARG, "bad gather arguments");
    const int64_t total = (int64_t)channels * ((W + *sx - 1) / *sx) * ((H + *sy - 1) / *sy);
    const int sms = num_sms();
    const int64_t want = (total + 255) / 256;
    const unsigned nb = (unsigned)(want < 8 * sms ? want : 8 * sms);
    k_gather<<<nb, 256, 0, (cudaStream_t)stream>>>(target_full, channels, W, H, *sx, *sy, target_out);
    return check_launch("k_gather");
}

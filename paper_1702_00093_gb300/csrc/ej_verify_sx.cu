// Verifier for pairs grouped by their longer string (Section 3.3, the last loop
// of Algorithm 3): the same exact test ED(x, y) <= K, with the match masks of x
// shared by a warp.
//
// The candidates arrive grouped by x, the longer string of each pair, and by
// their length difference d = |x| - |y| (sx_band), in warp tasks of up to 32 pairs
// that all share x and two adjacent classes of d, one lane per pair. A path of
// cost <= K of a pair stays on the diagonals i - j in
// [-floor((K - d)/2), floor((K + d)/2)] (the persistent verifier's band); the
// task's band is the union of its pairs' bands, at most K + 1 + (D - 1)/2
// diagonals for differences of a range of D, held in a diagonal window of W 32-bit words
// (ej_diag.cuh). All pairs of a task start together, so at every column their
// windows cover the same rows of x: the warp keeps one ring of W + 1 match words
// per symbol in shared memory. A word is built by the whole warp, every 32
// columns: lane t reads row t, one ballot per bit of the symbol codes gives the
// rows' bit planes, and lane c combines them into symbol c's mask.
//
// One lane per pair rather than two (halves that meet in the middle): nearly all
// of these candidates are rejected after the same number of columns (about
// K / 0.7 for text, 2 K for DNA, in one half or summed over two), and one lane
// per pair halves the tasks, and with them the rings, the loads and the window
// minima per pair.
//
// Early exit. A pair is rejected when no row of its window can lie on an alignment
// of cost <= K (diag_alive). That is looked at first after 9 K / 8 columns, then
// when the growth so far says that the slowest of the pairs about to be rejected
// will be (a multiple of 8 columns). Pairs that are not (similar strings run to the end) would keep the
// warp with most lanes idle: once at most 8 lanes are left and all of them are
// such, they are appended to a list that the persistent verifier takes from the
// start (vo.defer; without one the task runs to its end).
//
// What bounds it: 32-bit integer instructions, 10 W + about 8 per column and
// lane, and 5 per window row and quarter for a minimum.
// The integer pipe is 79% busy (0.59 instructions issued a cycle, K = 40). With the
// pairs handed over: 622M candidates of 200000 protein-like strings (K = 40, W = 2) 274 ->
// 74 ms against two lanes per pair on 64-bit block-aligned words with a minimum every
// 32 columns (77 ms with the plain minimum, first after 11 K / 8 columns); 30M of 120000
// text-like strings (K = 200, W = 7) 97.3 -> 40.3 ms. Any test of the list's room in the
// kernel, even of the whole warp at once, costs protein-like strings 2 to 3%: the list
// has room for SX_DEFER_MAX pairs of every task.
// Narrowing the window as its outer rows drop out was slower (58.6 ms on text):
// the rows that some of 32 pairs still needs leave only in the last third.
#include "ej_diag.cuh"

namespace ej {

namespace {

constexpr int SX_WARPS = 4;       // warps per block
constexpr int SX_PAIRS = 32;      // slots per task

// Symbol i (0 <= i < m) of a packed string.
template <int B>
__device__ __forceinline__ uint32_t sym_at(const uint4 *__restrict__ xc, int64_t i) {
    if (B == 8) return reinterpret_cast<const uint8_t *>(xc)[i];
    return (reinterpret_cast<const uint32_t *>(xc)[i >> 4] >> (2 * (uint32_t)(i & 15))) & 3u;
}

// Row t of a match word whose row 0 is symbol i0 - t of x: its code, or
// NO_SYMBOL outside x.
constexpr uint32_t NO_SYMBOL = 0x100u;
template <int B>
__device__ __forceinline__ uint32_t row_sym(const uint4 *__restrict__ xc, int32_t m, int64_t i) {
    return i >= 0 && i < m ? sym_at<B>(xc, i) : NO_SYMBOL;
}

// The word of the rows' symbols (lane t: row t) for every symbol, into ring
// entries c * RS + slot and, R entries further, their twins (so that a window's
// words sit at consecutive entries from any slot on).
__device__ __forceinline__ void sx_build(uint32_t *ring, int RS, int R, int slot, uint32_t sym, uint32_t alpha, int planes,
                                         int lane) {
    const uint32_t valid = __ballot_sync(FULL, sym != NO_SYMBOL);
    uint32_t bp[8];
#pragma unroll
    for (int k = 0; k < 8; k++)
        if (k < planes) bp[k] = __ballot_sync(FULL, (sym >> k) & 1u);
    for (uint32_t c = lane; c < alpha; c += 32) {
        uint32_t e = valid;
#pragma unroll
        for (int k = 0; k < 8; k++)
            if (k < planes) e &= ((c >> k) & 1u) ? bp[k] : ~bp[k];
        ring[(size_t)c * RS + slot] = e;
        ring[(size_t)c * RS + slot + R] = e;
    }
}

template <int W>
constexpr int sx_blocks() {   // resident blocks per SM the registers are limited to
    return W <= 3 ? 5 : W <= 8 ? 4 : 3;
}

template <int W, int B>
__global__ void __launch_bounds__(SX_WARPS * 32, sx_blocks<W>())
verify_sx_kernel(const uint4 *__restrict__ packed, const uint64_t *__restrict__ pofs,
                 const int32_t *__restrict__ lens, int64_t n_str, uint32_t alpha,
                 const uint64_t *__restrict__ pairs, const uint32_t *__restrict__ tasks,
                 const unsigned long long *__restrict__ ntasks_dev, int64_t ntasks_cap, int32_t K, int32_t RS,
                 int32_t warp_words, VerifyOut vo) {
    uint32_t *__restrict__ err = vo.err;
    unsigned long long *__restrict__ work = vo.work;
    constexpr int R = W + 1;
    extern __shared__ uint32_t sx_smem[];
    __shared__ uint32_t s_tab[256];
    diag_fill_table(s_tab);
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    uint32_t *ring = sx_smem + (size_t)wib * warp_words;
    const int64_t ntasks = (int64_t)*ntasks_dev;
    if (ntasks > ntasks_cap) return;   // tasks are missing: the call is repeated with room for them
    const int64_t nw = (int64_t)gridDim.x * SX_WARPS;
    const int planes = alpha <= 1 ? 1 : 32 - __clz(alpha - 1u);

    unsigned long long loc_cells = 0, loc_cols = 0;
    // a task's count and this lane's pair are loaded during the task before
    int64_t t = (int64_t)blockIdx.x * SX_WARPS + wib;
    int cnt_next = 0;
    uint64_t pr_next = 0;
    if (t < ntasks) {
        cnt_next = (int)tasks[t];
        if (lane < cnt_next) pr_next = pairs[t * SX_PAIRS + lane];
    }
    for (; t < ntasks; t += nw) {   // warp-uniform
        const uint64_t pr = pr_next;
        bool valid = lane < cnt_next;
        if (t + nw < ntasks) {
            cnt_next = (int)tasks[t + nw];
            if (lane < cnt_next) pr_next = pairs[(t + nw) * SX_PAIRS + lane];
        }
        int64_t a = 0, b = 0;
        if (valid) {
            a = (int64_t)(pr >> 32);
            b = (int64_t)(pr & 0xFFFFFFFFull);
            if (a >= n_str || b >= n_str) {
                atomicOr(err, (uint32_t)DERR_PAIR);
                valid = false;
            }
        }
        const int32_t la = valid ? lens[a] : 0, lb = valid ? lens[b] : 0;
        const bool a_long = la > lb;   // of two equally long ones x is the later (a < b)
        const int64_t xi = a_long ? a : b, yi = a_long ? b : a;
        const int32_t m = a_long ? la : lb, n = a_long ? lb : la;
        // every pair of a task has the same x (its first pair's)
        const int64_t xs = __shfl_sync(FULL, valid ? xi : -1, 0);
        if (valid && xi != xs) {
            atomicOr(err, (uint32_t)DERR_GUARD);
            valid = false;
        }
        bool running = valid, pass = false, deferred = false;
        if (valid && m - n > K) running = false;
        else if (valid && n == 0) { running = false; pass = m <= K; }
        int32_t cols_run = 0;
        // the task's band: the diagonals a cost-K alignment of any of its
        // undecided pairs can use (their length differences lie in two classes)
        const unsigned nlo = __reduce_min_sync(FULL, running ? (unsigned)n : 0xFFFFFFFFu);
        const unsigned nhi = __reduce_max_sync(FULL, running ? (unsigned)n : 0u);
        if (nhi > 0) {   // some pair is running
            const int32_t mx = lens[xs];
            const uint4 *xc = packed + pofs[xs];
            const int32_t klo = (K - (mx - (int32_t)nhi)) >> 1, khi = (K + (mx - (int32_t)nlo)) >> 1;
            if (klo + khi + 1 > 32 * W && lane == 0) atomicOr(err, (uint32_t)DERR_GUARD);   // not by construction
            // y, forward from its first chunk, a load ahead of its use: 16 columns
            // (B = 8) or 32 (B = 2) per load
            const char *yp = reinterpret_cast<const char *>(packed + (running ? pofs[yi] : 0));
            const uint32_t ybytes = running ? 16u * (uint32_t)chunks_for(n, B) : 0u;
            constexpr uint32_t YB = B == 8 ? 16 : 8;   // bytes per load
            auto y_load = [&](uint32_t off) {
                uint4 v = make_uint4(0u, 0u, 0u, 0u);
                if (off < ybytes) {
                    if (B == 8) {
                        v = *reinterpret_cast<const uint4 *>(yp + off);
                    } else {
                        const uint2 h = *reinterpret_cast<const uint2 *>(yp + off);
                        v.x = h.x;
                        v.y = h.y;
                    }
                }
                return v;
            };
            uint4 ynext = y_load(0), ycur = ynext;
            uint32_t yoff = YB;
            uint32_t P[W], M[W];
            diag_init<W>(P, M, klo);
            int32_t T = klo;
            // the first W + 1 words of x, and the rows of the next one
            {
                uint32_t sy[W + 1];
#pragma unroll
                for (int w = 0; w <= W; w++) sy[w] = row_sym<B>(xc, mx, 32 * w - klo + lane);
                __syncwarp();   // the ring of the task before is no longer read
#pragma unroll
                for (int w = 0; w <= W; w++) sx_build(ring, RS, R, w, sy[w], alpha, planes, lane);
                __syncwarp();
            }
            uint32_t sym_next = row_sym<B>(xc, mx, (int64_t)32 * (W + 1) - klo + lane);
            int base = 0;
            int32_t j = 0;                                             // columns done
            int32_t next_check = (9 * (K >> 3) + 15) & ~7;              // a multiple of 8, above K
            if (next_check <= K) next_check = (K + 8) & ~7;
            int32_t jend = (int32_t)nlo;                               // the first end of a running pair
            while (true) {
                if ((j & 31) == 0 && j > 0) {
                    // the word that left the window makes room for the one that enters
                    __syncwarp();
                    sx_build(ring, RS, R, base, sym_next, alpha, planes, lane);
                    base = base + 1 == R ? 0 : base + 1;
                    sym_next = row_sym<B>(xc, mx, (int64_t)j + 32 * (W + 1) - klo + lane);
                    __syncwarp();
                }
                // the symbols of 8 columns in two words (B = 8) or in the low half of one
                uint32_t s0, s1 = 0;
                if (B == 8) {
                    if ((j & 15) == 0) {
                        ycur = ynext;
                        ynext = y_load(yoff);
                        yoff += YB;
                        s0 = ycur.x;
                        s1 = ycur.y;
                    } else {
                        s0 = ycur.z;
                        s1 = ycur.w;
                    }
                } else {
                    if ((j & 31) == 0) {
                        ycur = ynext;
                        ynext = y_load(yoff);
                        yoff += YB;
                    }
                    s0 = ((j & 16) ? ycur.y : ycur.x) >> ((j & 8) * 2);
                }
                const uint32_t *wrow = ring + base;
                const uint32_t sh0 = (uint32_t)(j & 31);
                uint32_t tacc = 0;
                if (j + 8 < jend) {
#pragma unroll(W <= 4 ? 2 : 1)
                    for (int h = 0; h < 2; h++) {
                        const uint32_t sw = B == 8 ? (h ? s1 : s0) : s0 >> (8 * h);   // the symbols of 4 columns
#pragma unroll
                        for (int q = 0; q < 4; q++) {
                            const uint32_t c = B == 8 ? __byte_perm(sw, 0u, 0x4440 | q) : (sw >> (2 * q)) & 3u;
                            diag_step<W>(P, M, tacc, wrow + c * (uint32_t)RS, 1, sh0 + 4 * h + q);
                        }
                    }
                    T += 8 - __popc(tacc);
                    j += 8;
                    if (j < next_check) continue;
                } else {
                    // some pair ends within these columns: one at a time
#pragma unroll 1
                    for (int q = 0; q < 8; q++) {
                        const uint32_t c = B == 8 ? ((q & 4 ? s1 : s0) >> (8 * (q & 3))) & 0xFFu : (s0 >> (2 * q)) & 3u;
                        tacc = 0;
                        diag_step<W>(P, M, tacc, wrow + c * (uint32_t)RS, 1, sh0 + q);
                        T += 1 - (int32_t)(tacc >> 31);
                        if (running && j + q + 1 == n) {
                            // D(m, n): the row m is m - n + klo below the window's top
                            int32_t cnt = 0;
                            const int32_t rows = m - n + klo;
#pragma unroll
                            for (int v = 0; v < W; v++) {
                                const int32_t left = rows - 32 * v;
                                const uint32_t msk = left <= 0 ? 0u : left >= 32 ? ~0u : (1u << left) - 1u;
                                cnt += __popc(P[v] & msk) - __popc(M[v] & msk);
                            }
                            pass = T + cnt <= K;
                            running = false;
                            cols_run = n;
                        }
                    }
                    j += 8;
                    if (!__any_sync(FULL, running)) break;
                    jend = (int32_t)__reduce_min_sync(FULL, running ? (unsigned)n : 0x7FFFFFFFu);
                    if (j < next_check) continue;
                }
                // the windows' minima; lanes predicted to be rejected within half as
                // many columns again (a quarter before their minimum would exceed K)
                // keep the task going
                bool alive;
                const int32_t lb = T + diag_alive<W>(P, M, s_tab, T, m - n + klo, K, &alive);
                if (running && !alive) {
                    running = false;
                    cols_run = j;
                }
                const unsigned left = __ballot_sync(FULL, running);
                if (left == 0u) break;
                const float rem = 0.75f * (float)(K + 1 - lb) * (float)j / (float)(lb > 1 ? lb : 1);
                const bool soon = running && rem <= 0.5f * (float)j;
                const unsigned far = __reduce_max_sync(FULL, soon ? (unsigned)rem + 1u : 0u);
                if (far > 0u) {
                    next_check = j + (int32_t)((far + 7u) & ~7u);
                } else {
                    const int32_t most = (int32_t)__reduce_max_sync(FULL, running ? (unsigned)(n - j) : 0u);
                    if (vo.defer && __popc(left) <= SX_DEFER_MAX && most > j / 2) {
                        // similar pairs: to the persistent verifier
                        unsigned long long at = 0;
                        if (lane == 0) at = atomicAdd(vo.defer_count, (unsigned long long)__popc(left));
                        at = __shfl_sync(FULL, at, 0);
                        if (running) {
                            vo.defer[at + __popc(left & ((1u << lane) - 1u))] = pr;
                            deferred = true;
                            running = false;
                            cols_run = j;
                        }
                        break;
                    }
                    next_check = j + 64;
                }
                jend = (int32_t)__reduce_min_sync(FULL, running ? (unsigned)n : 0x7FFFFFFFu);
            }
        }
        if (valid && !deferred) {
            emit_result(vo, t * SX_PAIRS + lane, pairs, pass);
            loc_cells += band_cells(m, n, K);   // a deferred pair's are counted by its second verifier
        }
        if (valid) {
            const int32_t d = m - n;   // the pair's own band: ((K - d) >> 1) + ((K + d) >> 1) + 1 diagonals
            loc_cols += (unsigned long long)cols_run * (unsigned long long)((((K - d) >> 1) + ((K + d) >> 1) + 64) >> 6);
        }
    }
    // work counters: one atomic per warp (per-pair atomics on two addresses
    // serialise in the memory system)
    if (work) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            loc_cells += __shfl_xor_sync(FULL, loc_cells, o);
            loc_cols += __shfl_xor_sync(FULL, loc_cols, o);
        }
        if (lane == 0) {
            if (loc_cells) atomicAdd(&work[0], loc_cells);
            if (loc_cols) atomicAdd(&work[1], loc_cols);
        }
    }
}

// Ring row stride: both copies of W + 1 words, odd (lanes reading different
// symbols spread over the banks).
int sx_row(int W) { return 2 * (W + 1) + 1; }

template <int W, int B>
cudaError_t launch_sx_t(const uint4 *packed, const uint64_t *pofs, const int32_t *lens, int64_t n, uint32_t alpha,
                        const uint64_t *pairs, const uint32_t *tasks, const unsigned long long *ntasks_dev,
                        int64_t ntasks_cap, int32_t K, VerifyOut vo, cudaStream_t s) {
    const size_t smem = sx_smem_bytes(W, alpha);
    if (smem > 220 * 1024) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(verify_sx_kernel<W, B>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, verify_sx_kernel<W, B>, SX_WARPS * 32, smem);
    if (per_sm < 1) per_sm = 1;
    int64_t blocks = (int64_t)sms * per_sm;
    const int64_t need = (ntasks_cap + SX_WARPS - 1) / SX_WARPS;
    if (blocks > need) blocks = need > 0 ? need : 1;
    verify_sx_kernel<W, B><<<(unsigned)blocks, SX_WARPS * 32, smem, s>>>(
        packed, pofs, lens, n, alpha, pairs, tasks, ntasks_dev, ntasks_cap, K, sx_row(W), (int32_t)(alpha * sx_row(W)),
        vo);
    note_launches(1);
    return cudaGetLastError();
}

}  // namespace

SxBand sx_band(int32_t K) {
    int W = (K + 32) / 32;             // ceil((K + 1) / 32)
    int slack = 32 * W - (K + 1);      // diagonals the window has beyond a single pair's band
    if (K > 2 * slack + 1 && (slack + 1 < 4 || K / (slack + 1) + 1 > 16)) {
        // length differences narrower than 8 split a string's pairs too finely, and
        // more than 16 classes cost their searches: one word more
        W += 1;
        slack += 32;
    }
    if (K <= 2 * slack + 1) return SxBand{W, (uint32_t)K + 1u, 1u};   // every difference fits one task
    return SxBand{W, (uint32_t)slack + 1u, (uint32_t)K / ((uint32_t)slack + 1u) + 1u};
}

size_t sx_smem_bytes(int W, uint32_t alpha) { return (size_t)alpha * sx_row(W) * sizeof(uint32_t) * SX_WARPS; }

cudaError_t launch_verify_sx(int W, const uint4 *packed, const uint64_t *pofs, int B, const int32_t *lens, int64_t n,
                             uint32_t alpha, const uint64_t *pairs, const uint32_t *tasks,
                             const unsigned long long *ntasks_dev, int64_t ntasks_cap, int32_t K, VerifyOut vo,
                             cudaStream_t s) {
    if (ntasks_cap == 0) return cudaGetLastError();
#define EJ_SX(WW)                                                                                          \
    if (W == WW) {                                                                                        \
        if (B == 2) return launch_sx_t<WW, 2>(packed, pofs, lens, n, alpha, pairs, tasks, ntasks_dev, ntasks_cap, K, vo, s); \
        return launch_sx_t<WW, 8>(packed, pofs, lens, n, alpha, pairs, tasks, ntasks_dev, ntasks_cap, K, vo, s);   \
    }
    EJ_SX(1) EJ_SX(2) EJ_SX(3) EJ_SX(4) EJ_SX(5) EJ_SX(6) EJ_SX(7) EJ_SX(8) EJ_SX(9) EJ_SX(10) EJ_SX(11) EJ_SX(12)
#undef EJ_SX
    return cudaErrorInvalidValue;
}

}  // namespace ej

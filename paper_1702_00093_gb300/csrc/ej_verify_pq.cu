// Persistent verifier: the same exact test ED(x, y) <= K as the banded
// bit-parallel verifiers (Section 3.3, the last loop of Algorithm 3), with the
// pairs pulled from a device work queue so that a lane pair whose pair is done
// takes the next one instead of idling until the slowest pair of its warp ends.
//
// Per pair, two lanes: the forward half computes D(., n1) for n1 = n/2 over a
// diagonal window (ej_diag.cuh), the backward half runs the same
// recurrence on the reversed strings for the remaining n - n1 columns, and
// ED(x, y) = min_i D(i, n1) + ED(x[i:], y[n1:]) joins them (the argument and the
// boundary conditions are the ones of the block-aligned two-lane verifier).
//
// Band. With x the longer string (m rows), y the shorter (n columns) and
// d = m - n, a path of cost c through cell (i, j) has c >= |i - j| + |d - (i - j)|
// (the distances to the diagonals of both corners), so a path of cost <= K
// stays on the diagonals i - j in [-K_lo, K_hi], K_lo = floor((K - d) / 2),
// K_hi = floor((K + d) / 2): at most K + 1 diagonals, where Ukkonen's band has
// 2K + 1 (the same argument as his cutoff). Both halves use it (reversing both
// strings keeps d). The window is diagonal (ej_diag.cuh): W = ceil((K + 1) / 32)
// 32-bit words hold exactly those diagonals.
//
// Scheduling. A warp advances its 16 pair slots in chunks of 32 columns, one
// match-mask word of the window entering per chunk. Both halves of a pair are
// padded in front with a common prefix (which changes no distance) to the same
// multiple of 32 columns, N1 = 32 ceil((n - floor(n/2)) / 32): every slot starts
// and ends at a chunk boundary, both lanes of a slot together, and the column
// loop has no test (a lane without a pair advances values that nothing reads; its
// reads stay inside its own ring and the packed strings). The number of working
// warps is capped (by default one per SM sub-partition), so that a batch larger
// than the slots keeps every slot busy until the queue runs dry.
//
// Early exit. After every other chunk of a pair each half computes the minimum value
// m_h of its window (including the top cell). A path of cost <= K crosses both halves'
// current columns inside their bands, where the values are exact, so
// m_fwd + m_bwd > K proves ED > K; both lanes of the pair stop.
//
// What bounds it: 32-bit integer instructions, 10 W + about 8 per column. Many pairs
// fill their pipe: the 5.7M candidates of 20000 reads of 5000 bases at K = 250, z = 7
// take 20.2 ms at four warps per sub-partition (the choice for so many) or three, 21.5
// at two and 28.4 at one (that join's default is the shared-string verifier, 17.1 ms);
// the block-aligned window with a test per column, which this form replaced, took 28.2 ms.
// Few pairs are set by the columns of the longest on one warp per sub-partition: about
// 13000 at K = 250 take 0.38 ms (0.50 before), 5200 at K = 150 0.25 ms (0.49 before:
// 8 words of 64 bits where there are 5 of 32).
#include <climits>

#include "ej_diag.cuh"

namespace ej {

namespace {

constexpr int64_t kMaxIters = 1ll << 24;   // default bound on loop passes per warp (VerifyOut::max_passes)

// The two words under 64/B symbols of a packed string starting at symbol o
// (any int64; words outside the string read as 0) and the bit offset of symbol
// o in the first: loads only, combined by sym_join when the symbols are needed
// (so that the load's latency passes while the previous word is consumed).
struct SymRaw {
    uint64_t a, b;
    uint32_t sh;
};
template <int B>
__device__ __forceinline__ SymRaw sym_fetch(const uint64_t *__restrict__ y64, int64_t nwords, int64_t o) {
    const int64_t bit = o * B;
    const int64_t w0 = bit >= 0 ? (bit >> 6) : -((-bit + 63) >> 6);
    SymRaw r;
    r.sh = (uint32_t)(bit - 64 * w0);
    r.a = (w0 >= 0 && w0 < nwords) ? y64[w0] : 0ull;
    r.b = (w0 + 1 >= 0 && w0 + 1 < nwords) ? y64[w0 + 1] : 0ull;
    return r;
}
__device__ __forceinline__ uint64_t sym_join(const SymRaw &r) {
    return r.sh ? ((r.a >> r.sh) | (r.b << (64u - r.sh))) : r.a;
}


__device__ __forceinline__ unsigned sm_id() {
    unsigned r;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(r));
    return r;
}

// Reverses the order of the 64/B symbols of a word.
template <int B>
__device__ __forceinline__ uint64_t sym_reverse(uint64_t u) {
    if (B == 8) {
        const uint32_t lo = (uint32_t)u, hi = (uint32_t)(u >> 32);
        return ((uint64_t)__byte_perm(lo, 0u, 0x0123) << 32) | (uint64_t)__byte_perm(hi, 0u, 0x0123);
    }
    const uint64_t r = __brevll(u);   // B == 2: reverse bits, then swap the two bits of each symbol
    return ((r >> 1) & 0x5555555555555555ull) | ((r & 0x5555555555555555ull) << 1);
}

// Match-mask word of a pair's padded x (or reversed x) from symbol q on (bit t:
// symbol q + t; symbols -pad .. -1 are the padding, code 0; none outside
// [-pad, m)) for every symbol c < alpha, into ring entries c * R2 + slot and,
// R entries further, its twin.
template <int B, int R>
__device__ __forceinline__ void pq_build(uint32_t *ring, int T_, int slot, const uint64_t *__restrict__ x64, int32_t m,
                                         int64_t q, int32_t pad, bool rev, uint32_t alpha) {
    constexpr int R2 = 2 * R;
    const int t_lo = (int)max((int64_t)0, -(q + pad)), t_hi = (int)min((int64_t)32, m - q);
    uint32_t valid = 0u;
    if (t_hi > t_lo) valid = (t_hi >= 32 ? ~0u : (1u << t_hi) - 1u) & ~((1u << t_lo) - 1u);
    const int64_t xwords = 2 * chunks_for(m, B);
    if (B == 2) {
        const uint64_t v = sym_join(sym_fetch<2>(x64, xwords, rev ? m - 32 - q : q));
        const uint32_t w0 = (uint32_t)v, w1 = (uint32_t)(v >> 32);
        uint32_t lo = compress_even(w0) | (compress_even(w1) << 16);
        uint32_t hi = compress_even(w0 >> 1) | (compress_even(w1 >> 1) << 16);
        if (rev) {
            lo = __brev(lo);
            hi = __brev(hi);
        }
        for (uint32_t c = 0; c < alpha; c++) {
            const uint32_t e = ((c & 1u) ? lo : ~lo) & ((c & 2u) ? hi : ~hi) & valid;
            ring[(size_t)(c * R2 + slot) * T_] = e;
            ring[(size_t)(c * R2 + slot + R) * T_] = e;
        }
    } else {
        for (uint32_t c = 0; c < alpha; c++) ring[(size_t)(c * R2 + slot) * T_] = 0u;
        if (valid) {
            // every symbol sets its bit with a shared-memory OR that returns
            // nothing, so consecutive symbols (which may hit the same word) do
            // not wait on one another
#pragma unroll
            for (int g = 0; g < 4; g++) {
                uint64_t v = sym_join(sym_fetch<8>(x64, xwords, rev ? m - 8 - q - 8 * g : q + 8 * g));
                if (rev) v = sym_reverse<8>(v);
#pragma unroll
                for (int t = 8 * g; t < 8 * g + 8; t++) {
                    const uint32_t c = (uint32_t)v & 0xFFu;
                    v >>= 8;
                    if (t >= t_lo && t < t_hi) atomicOr(ring + (size_t)(c * R2 + slot) * T_, 1u << t);
                }
            }
        }
        for (uint32_t c = 0; c < alpha; c++)
            ring[(size_t)(c * R2 + slot + R) * T_] = ring[(size_t)(c * R2 + slot) * T_];
    }
}

template <int W, int B, int TPB>
__global__ void __launch_bounds__(TPB, 1)
verify_pq_kernel(const uint4 *__restrict__ packed, const uint64_t *__restrict__ pofs,
                 const int32_t *__restrict__ lens, int64_t n_str, uint32_t alpha,
                 const uint64_t *__restrict__ pairs, int64_t np, int32_t K, int32_t nsm, int32_t spw_force,
                 int32_t wps, VerifyOut vo) {
    uint32_t *__restrict__ err = vo.err;
    const VerifySeg *__restrict__ segs = vo.segs;   // merged launch: the joins' candidates in turn
    const int nseg = segs ? vo.nseg : 0;
    const bool uni = segs && vo.umask;              // ... or their union, each pair once
    __shared__ long long s_cum[MAX_VERIFY_SEGS + 1];
    if (segs) {
        if (threadIdx.x == 0) {
            long long acc = 0;
            for (int g = 0; g < nseg; g++) {
                s_cum[g] = acc;
                const long long c = (long long)*segs[g].np_dev;
                acc += c < (long long)segs[g].cap ? c : (long long)segs[g].cap;
            }
            if (uni) {
                const unsigned long long c = *vo.unp_dev;
                acc = (long long)(c < vo.ucap ? c : vo.ucap);
            }
            s_cum[nseg] = acc;
        }
    } else {
        if (vo.np_dev) {
            const int64_t dn = (int64_t)*vo.np_dev;
            np = dn < np ? dn : np;
        }
        if (vo.pairs_off_dev) pairs += *vo.pairs_off_dev;
    }
    // error bits of one pair (its join's word in a merged launch), or of the warp
    auto pair_err = [&](int g, uint32_t bits) { atomicOr(segs ? segs[g].err : err, bits); };
    auto warp_err = [&](uint32_t bits) {
        if (!segs) atomicOr(err, bits);
        else
            for (int g = 0; g < nseg; g++) atomicOr(segs[g].err, bits);
    };
    // union pair q (listed by the joins of mask mk) with edit distance ed (or
    // INT_MAX when above the band's K): to every listing join whose K it meets
    auto emit_union = [&](int64_t q, uint32_t mk, int32_t ed) {
        for (int g = 0; g < nseg; g++) {
            if (!((mk >> g) & 1u) || ed > segs[g].K) continue;
            const unsigned long long idx = atomicAdd(segs[g].app_count, 1ull);
            if (idx < segs[g].app_cap) segs[g].app[idx] = vo.upairs[q];
        }
    };
    // a finished pair's result: to its join's outputs in a merged launch
    auto emit = [&](int g, int64_t q, bool pass) {
        if (!segs) {
            emit_result(vo, q, pairs, pass);
        } else if (pass) {
            const VerifySeg &sg_ = segs[g];
            const unsigned long long idx = atomicAdd(sg_.app_count, 1ull);
            if (idx < sg_.app_cap) sg_.app[idx] = sg_.pairs[q];
        }
    };
    constexpr int R = W + 1;                 // words of the window at any shift
    constexpr int R2 = 2 * R;                // ring slots per symbol: every word is kept twice,
                                             // at slot k mod R and k mod R + R, so that the
                                             // window's words sit at consecutive slots
    constexpr int SPW = 64 / B;              // symbols per 64-bit word
    extern __shared__ uint32_t pq_smem[];
    __shared__ uint32_t s_tab[256];
    diag_fill_table(s_tab);
    __syncthreads();
    if (segs) np = s_cum[nseg];
    constexpr int T_ = TPB;                   // slot stride of the per-thread ring
    uint32_t *ring = pq_smem + threadIdx.x;   // (c*R2 + slot)*T_, reused as a dump area
    const int lane = threadIdx.x & 31;
    const bool rev = lane & 1;
    const int slot = lane >> 1;

    // Slots per warp and working warps. The working blocks are chosen per SM
    // (the first ones to take a ticket on their SM), so that they are spread
    // evenly over the SMs whatever order the blocks were placed in. A block of
    // four warps has one on each sub-partition and takes one ticket: tickets per
    // warp let the first warps of two blocks that start together land on the
    // same sub-partitions (0.61 instead of 0.38 ms for the headline batch's
    // launch). One-warp blocks: at most 4*wps per SM, fewer when the pairs are few.
    const int64_t spw = spw_force > 0 ? (spw_force > 16 ? 16 : spw_force) : 16;
    const int64_t warps_needed = (np + spw - 1) / spw;
    int64_t per_sm = (warps_needed + nsm - 1) / (nsm > 0 ? nsm : 1);
    if (wps <= 0) {
        // automatic: one working warp per sub-partition while the pairs are few
        // (more warps would only start them all at once, and the launch ends
        // with its slowest pairs); 2 or 4 when every slot of one warp per
        // sub-partition would take at least 8 or 32 pairs (the second and third
        // warps then hide the step's fixed latencies)
        const int64_t per_slot = np / ((int64_t)(nsm > 0 ? nsm : 1) * 4 * spw);
        wps = per_slot >= 32 ? 4 : per_slot >= 8 ? 2 : 1;
    }
    if (per_sm > 4ll * wps) per_sm = 4ll * wps;
    constexpr int BW = TPB / 32;
    __shared__ unsigned s_ticket;
    if (threadIdx.x == 0) s_ticket = atomicAdd(&vo.sm_tickets[sm_id() & (SM_TICKETS - 1)], 1u);
    __syncthreads();
    bool exhausted = (slot >= spw) || ((int64_t)s_ticket >= (per_sm + BW - 1) / BW);
    if (__all_sync(FULL, exhausted)) return;
    // merged launch: the warp's work counters per join, in shared memory (added
    // to the joins' global counters once, when the warp ends)
    __shared__ unsigned long long s_wk[TPB / 32][MAX_VERIFY_SEGS][2];
    unsigned long long *wk = &s_wk[threadIdx.x >> 5][0][0];
    if (lane < 2 * MAX_VERIFY_SEGS) wk[lane] = 0ull;
    __syncwarp();

    unsigned long long loc_cells = 0, loc_cols = 0;
    bool have = false, rejected = false;
    int64_t p = 0;
    const uint64_t *x64 = reinterpret_cast<const uint64_t *>(packed), *y64 = x64;
    int64_t ywords = 0;
    int32_t m = 0, n = 0, klo = 0, T = 0;
    int32_t ncols = 0;       // padded columns of either half (a multiple of 32)
    int32_t pad = 0;         // padding columns of this lane's half
    int32_t j0 = 0;          // columns done
    int32_t wpair = 1;       // words of the pair's band, ceil((K_lo + K_hi + 1) / 64) (work counter)
    // the raw word of padded y's (or reversed y's) symbols from column sidx + 1 on
    auto sym_word = [&](int32_t sidx) -> SymRaw {
        const int64_t q = (int64_t)sidx - pad;
        return sym_fetch<B>(y64, ywords, rev ? (int64_t)n - SPW - q : q);
    };
    SymRaw snext{0ull, 0ull, 0u};   // the next word of the stream, already requested
    int32_t kp = K;          // the pair's threshold (<= K, the band)
    int sg = 0;              // the pair's join (merged launch; of the union: the largest K's)
    uint32_t umk = 0;        // union pair: the mask of the joins that list it
    int64_t iters = 0;       // chunks of this warp (bounded by max_iters)
    // the warp's running pairs have done an odd number of chunks: pairs start together
    // only where it is even, so that every pair meets the joint bound after its own
    // second, fourth, ... chunk, whichever pairs ran beside it
    bool odd = false;
    // a pass of the documented bound is 64 columns, two chunks
    const int64_t max_iters = 2 * (vo.max_passes > 0 ? min(vo.max_passes, (int64_t)1 << 61) : kMaxIters);
    int base = 0;
    uint32_t P[W], M[W];
#pragma unroll
    for (int v = 0; v < W; v++) { P[v] = 0; M[v] = 0; }

    while (true) {
        if (++iters > max_iters) {
            // every lane counts the same passes, so the whole warp leaves here
            // (no block barrier follows); the call reports EJ_ERR_TIMEOUT
            if (lane == 0) warp_err((uint32_t)DERR_TIMEOUT);
            break;
        }
        // refill free slots (both lanes of a slot agree on `have` and `exhausted`),
        // several at a time: a refill takes the whole warp through the loads and the
        // W + 1 match words of its pairs however few they are, and pairs that start
        // together mostly end together (956000 text-like pairs, W = 4: one slot at a
        // time 3.94 ms, four 2.82, eight 2.72; 5.7M DNA pairs, W = 8: 21.6, four 20.5)
        // With fewer slots, half of them.
        constexpr int REFILL = B == 8 ? 8 : 4;
        const int refill_at = min(REFILL, max(1, (int)spw / 2));
        const unsigned idle = __ballot_sync(FULL, !have && !exhausted && !rev);
        const bool none = !__any_sync(FULL, have);
        if (none) odd = false;
        const bool refill = idle && !odd && (none || __popc(idle) >= refill_at);
        while (refill) {
            const bool need = !have && !exhausted;
            const unsigned nb = __ballot_sync(FULL, need && !rev);
            if (nb == 0u) break;
            const int leader = __ffs(nb) - 1;
            unsigned long long qb = 0;
            if (lane == leader) qb = atomicAdd(vo.queue, (unsigned long long)__popc(nb));
            qb = __shfl_sync(FULL, qb, leader);
            if (need) {
                const unsigned fl = (unsigned)(lane & ~1);
                const int64_t idx = (int64_t)qb + __popc(nb & ((1u << fl) - 1u));
                if (idx >= np) {
                    exhausted = true;
                } else {
                    p = idx;
                    const uint64_t *pp = pairs;
                    if (uni) {
                        pp = vo.upairs;
                        umk = vo.umask[idx];
                        sg = -1;
                        for (int g = 0; g < nseg; g++)
                            if (((umk >> g) & 1u) && (sg < 0 || segs[g].K > segs[sg].K)) sg = g;
                        if (sg < 0) sg = 0;   // an empty mask cannot occur; its pair reaches no join
                    } else if (segs) {
                        sg = 0;
                        while (sg + 1 < nseg && idx >= s_cum[sg + 1]) sg++;
                        p = idx - s_cum[sg];
                        pp = segs[sg].pairs;
                    }
                    const uint64_t pr = pp[p];
                    const int64_t a = (int64_t)(pr >> 32), b = (int64_t)(pr & 0xFFFFFFFFull);
                    const bool two = vo.packed_b != nullptr;   // b indexes the second set
                    if (a >= n_str || b >= (two ? vo.n_b : n_str)) {
                        if (!rev) pair_err(sg, (uint32_t)DERR_PAIR);
                    } else {
                        const int32_t la = lens[a], lb = two ? vo.lens_b[b] : lens[b];
                        const uint4 *pa = packed + pofs[a];
                        const uint4 *pb = two ? vo.packed_b + vo.pofs_b[b] : packed + pofs[b];
                        const bool a_long = la >= lb;
                        m = a_long ? la : lb;
                        n = a_long ? lb : la;
                        kp = segs ? segs[sg].K : (vo.thr ? vo.thr[a] : K);
                        if (!rev) {
                            if (uni) {
                                for (int g = 0; g < nseg; g++)
                                    if ((umk >> g) & 1u) atomicAdd(&wk[2 * g], band_cells(m, n, segs[g].K));
                            } else if (segs) {
                                atomicAdd(&wk[2 * sg], band_cells(m, n, kp));
                            } else {
                                loc_cells += band_cells(m, n, kp);
                            }
                        }
                        if (m - n > kp || n == 0) {
                            if (!rev) {
                                if (uni) emit_union(p, umk, n == 0 ? m : INT_MAX);
                                else emit(sg, p, n == 0 && m <= kp);
                            }
                        } else {
                            const int32_t n1 = n / 2;
                            const int32_t nh = rev ? n - n1 : n1;
                            ncols = (n - n1 + 31) & ~31;
                            pad = ncols - nh;
                            x64 = reinterpret_cast<const uint64_t *>(a_long ? pa : pb);
                            y64 = reinterpret_cast<const uint64_t *>(a_long ? pb : pa);
                            ywords = 2 * chunks_for(n, B);
                            // the pair's band (see the head of this file); m - n <= kp here
                            klo = (kp - (m - n)) >> 1;
                            const int32_t khi = (kp + (m - n)) >> 1;
                            wpair = (klo + khi + 64) >> 6;
                            for (int wi = 0; wi <= W; wi++)
                                pq_build<B, R>(ring, T_, wi, x64, m, (int64_t)(32 * wi) - klo - pad, pad, rev, alpha);
                            diag_init<W>(P, M, klo);
                            T = klo;
                            base = 0;
                            j0 = 0;
                            snext = sym_word(0);
                            rejected = false;
                            have = true;
                        }
                    }
                }
            }
        }
        if (!__any_sync(FULL, have)) break;

        // one chunk: columns j0 + 1 .. j0 + 32 of every slot
        if (have && j0 > 0) {
            // the word that left the window makes room for the one that enters
            pq_build<B, R>(ring, T_, base, x64, m, (int64_t)j0 + 32 * W - klo - pad, pad, rev, alpha);
            base = base + 1 == R ? 0 : base + 1;
        }
        const uint32_t *wrow = ring + base * T_;   // symbol 0's words of the window
        uint32_t tacc = 0;
#pragma unroll 1
        for (int g = 0; g < 32; g += SPW) {
            const uint64_t sv = sym_join(snext);
            uint64_t sreg = rev ? sym_reverse<B>(sv) : sv;
            snext = sym_word(j0 + g + SPW);
            // four symbols per step; a 2-bit code is masked in place and its row's
            // offset is one multiplication (CST is a multiple of 64)
            constexpr uint32_t CST = R2 * T_ * sizeof(uint32_t);
            const char *wbase = reinterpret_cast<const char *>(wrow);
#pragma unroll(W <= 4 ? 2 : 1)
            for (int t = 0; t < SPW; t += 4) {
                const uint32_t sw = (uint32_t)sreg;
                sreg >>= 4 * B;
#pragma unroll
                for (int q = 0; q < 4; q++) {   // codes are < alpha (0 outside the string)
                    const uint32_t off = B == 2 ? (sw & (3u << (2 * q))) * (CST >> (2 * q))
                                                : __byte_perm(sw, 0u, 0x4440 | q) * CST;
                    diag_step<W>(P, M, tacc, reinterpret_cast<const uint32_t *>(wbase + off), T_, (uint32_t)(g + t + q));
                }
            }
        }
        T += 32 - __popc(tacc);
        j0 += 32;
        if (odd) {   // the joint bound (every chunk: 2.92 against 2.72 ms on text, W = 4)
            const int32_t lb = T + diag_min<W>(P, M, s_tab);
            const int32_t lb_other = __shfl_xor_sync(FULL, lb, 1);
            if (have && j0 < ncols && lb + lb_other > kp) rejected = true;
        }
        odd = !odd;

        // finished pairs: all columns run, or rejected (both lanes agree)
        const bool pair_done = have && (rejected || j0 >= ncols);
        if (__any_sync(FULL, pair_done)) {
            if (pair_done) {
                const int32_t real = j0 - pad;
                const unsigned long long cols = real > 0 ? (unsigned long long)real : 0ull;
                if (segs) atomicAdd(&wk[2 * sg + 1], cols * (unsigned long long)wpair);
                else loc_cols += cols * (unsigned long long)wpair;
                if (!rejected) diag_dump<W>(ring, T_, P, M, T);
            }
            __syncwarp();
            int32_t ed = INT_MAX;                           // the distance when <= kp
            if (pair_done && !rejected) {
                const uint32_t *f = pq_smem + (threadIdx.x & ~1u);   // forward half's dump, then the backward one's
                ed = diag_meet<W>(f, f + 1, T_, m, n / 2, n - n / 2, klo, rev ? 1 : 0);
            }
            ed = min(ed, __shfl_xor_sync(FULL, ed, 1));
            if (pair_done && !rev) {
                const bool pass = ed <= kp;
                if (!pass) ed = INT_MAX;
                if (uni) emit_union(p, umk, ed);
                else emit(sg, p, pass);
            }
            __syncwarp();
            if (pair_done) have = false;
        }
    }

    if (segs) {
        __syncwarp();
        if (lane < 2 * nseg && wk[lane]) atomicAdd(&segs[lane >> 1].work[lane & 1], wk[lane]);
    }
    if (vo.work) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            loc_cells += __shfl_xor_sync(FULL, loc_cells, o);
            loc_cols += __shfl_xor_sync(FULL, loc_cols, o);
        }
        if (lane == 0) {
            if (loc_cells) atomicAdd(&vo.work[0], loc_cells);
            if (loc_cols) atomicAdd(&vo.work[1], loc_cols);
        }
    }
}

template <int W, int B, int TPB>
cudaError_t launch_pq_tt(const uint4 *packed, const uint64_t *pofs, const int32_t *lens, int64_t n, uint32_t alpha,
                         const uint64_t *pairs, int64_t np, int32_t K, int spw_force, int wps, VerifyOut vo,
                         cudaStream_t s) {
    constexpr int threads = TPB;
    const size_t smem = pq_smem_bytes(W, alpha, threads);
    cudaError_t e = cudaFuncSetAttribute(verify_pq_kernel<W, B, TPB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, verify_pq_kernel<W, B, TPB>, threads, smem);
    if (per_sm < 1) per_sm = 1;
    const int64_t blocks = (int64_t)sms * per_sm;
    verify_pq_kernel<W, B, TPB><<<(unsigned)blocks, threads, smem, s>>>(packed, pofs, lens, n, alpha, pairs, np, K,
                                                                       sms, spw_force, wps, vo);
    note_launches(1);
    return cudaGetLastError();
}

}  // namespace

size_t pq_smem_bytes(int W, uint32_t alpha, int threads) {
    return (size_t)alpha * 2 * ((size_t)W + 1) * sizeof(uint32_t) * (size_t)threads;
}

int pq_threads_for(int W, uint32_t alpha) {
    if (W > PQ_MAX_WORDS) return 0;
    if (pq_smem_bytes(W, alpha, 128) <= 160 * 1024) return 128;
    // blocks of one warp only for alphabets of more than four symbols (the rings
    // of up to four fit 128 threads at every W)
    return pq_smem_bytes(W, alpha, 32) <= 220 * 1024 ? 32 : 0;
}

cudaError_t launch_verify_pq(int W, int threads, int spw_force, int wps, const uint4 *packed, const uint64_t *pofs, int B,
                             const int32_t *lens, int64_t n, uint32_t alpha, const uint64_t *pairs, int64_t np,
                             int32_t K, VerifyOut vo, cudaStream_t s) {
    if (np == 0) return cudaGetLastError();
    if (!vo.queue || !vo.sm_tickets || (threads != 128 && threads != 32)) return cudaErrorInvalidValue;
#define EJ_PQ(WW)                                                                                                  \
    if (W == WW) {                                                                                                 \
        if (B == 2 && threads == 128)                                                                              \
            return launch_pq_tt<WW, 2, 128>(packed, pofs, lens, n, alpha, pairs, np, K, spw_force, wps, vo, s);    \
        if (B == 8 && threads == 128)                                                                              \
            return launch_pq_tt<WW, 8, 128>(packed, pofs, lens, n, alpha, pairs, np, K, spw_force, wps, vo, s);    \
        if (B == 8) return launch_pq_tt<WW, 8, 32>(packed, pofs, lens, n, alpha, pairs, np, K, spw_force, wps, vo, s); \
    }
    EJ_PQ(1) EJ_PQ(2) EJ_PQ(3) EJ_PQ(4) EJ_PQ(5) EJ_PQ(6) EJ_PQ(7) EJ_PQ(8) EJ_PQ(9) EJ_PQ(10) EJ_PQ(11) EJ_PQ(12)
    EJ_PQ(14) EJ_PQ(16) EJ_PQ(18) EJ_PQ(20) EJ_PQ(22) EJ_PQ(24)
#undef EJ_PQ
    return cudaErrorInvalidValue;
}

}  // namespace ej

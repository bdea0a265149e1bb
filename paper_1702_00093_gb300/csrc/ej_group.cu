// Candidates grouped for the shared-string verifier (Alg. 3's filtering and
// deduplication): for every string x, the strings y that precede it in (length,
// id) order, share a signature with it in some table and differ in length by at
// most K, each once, in warp tasks of up to 32 pairs that share x and two adjacent
// classes of the length difference (partners come in increasing difference; a task
// that is not full takes pairs of the next class, so that few leave part empty).
//
// Every table's records are sorted by (signature, length, id), so the partners of
// x in a table are the records of one window just before x's own. A warp takes
// one x: each lane finds x's windows in one table (a galloping search), the
// windows of 32 tables are read as one list, and a partner is kept in the first
// table only in which it meets x. That test replaces a sort of all raw pairs: the
// signatures of a string in all its tables lie side by side as 16-bit
// fingerprints, so "did x and y meet before table t" is a comparison of the first t
// fingerprints of two rows, eight per 16-byte load, and only equal fingerprints
// compare the signatures themselves. The kept pairs collect in shared memory and
// leave as whole tasks; nothing is sorted or scattered, and a raw pair that is a
// duplicate never reaches memory.
//
// What bounds it: the L2 reads of the fingerprint rows (2 T bytes per string, at
// most 2 T bytes per raw pair and half of that on average for a new one).
// From the signatures to the tasks, 0.80G raw pairs of 200000 protein-like strings
// (T = 49, K = 40, 622M distinct): 24 ms (the tables' sorting 1.2), where hashed record
// lists (36 ms), five radix passes over the raw pairs (63 ms) and their compaction
// (15 ms) took 114 ms; 5003 such strings at K = 60: 0.25 ms against 3.6 ms for lists in
// shared memory, one block per table walking buckets of a thousand records.
#include "ej_internal.cuh"

namespace ej {

namespace {

constexpr int GE_WARPS = 8;    // warps per block of the emitting kernel
constexpr int GE_BLOCKS = 8;   // blocks per SM
constexpr int GE_KEEP = 160;   // tables whose windows are kept from class to class

__device__ __forceinline__ uint32_t fingerprint(uint64_t k) { return (uint32_t)(key_hash(k) >> 48); }

// Per record of every sorted table: its string's length beside its id, and for
// every string its place in the table. counters[1]: the largest run of equal
// signatures (taken at each run's last record).
__global__ void group_prep_kernel(const uint64_t *__restrict__ rk, const uint32_t *__restrict__ rid,
                                  const int32_t *__restrict__ lens, int64_t n, uint64_t *__restrict__ rec,
                                  uint32_t *__restrict__ pos, unsigned long long *__restrict__ counters) {
    const int64_t t = blockIdx.y;
    rk += t * n;
    rid += t * n;
    rec += t * n;
    pos += t * n;
    unsigned long long mb = 0;
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t id = rid[p];
        rec[p] = ((uint64_t)(uint32_t)lens[id] << 32) | id;
        pos[id] = (uint32_t)p;
        const uint64_t key = rk[p];
        if (p + 1 < n && rk[p + 1] == key) continue;
        int64_t lo = 0, hi = p;   // the first record of the run
        while (lo < hi) {
            const int64_t mid = (lo + hi) >> 1;
            if (rk[mid] < key) lo = mid + 1;
            else hi = mid;
        }
        mb = max(mb, (unsigned long long)(p - lo + 1));
    }
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long v = __shfl_xor_sync(FULL, mb, o);
        mb = v > mb ? v : mb;
    }
    if ((threadIdx.x & 31) == 0 && mb) atomicMax(&counters[1], mb);
}

// Row x of fp: the fingerprints of x's signatures in tables 0 .. T-1, eight per
// 16 bytes (zero padded).
__global__ void fingerprint_kernel(const uint64_t *__restrict__ keys, int64_t n, int32_t T, int32_t FW,
                                   uint4 *__restrict__ fp) {
    const int g = blockIdx.y;
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n; x += (int64_t)gridDim.x * blockDim.x) {
        uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
        for (int k = 0; k < 8; k++) {
            const int t = 8 * g + k;
            if (t < T) w[k >> 1] |= fingerprint(keys[(int64_t)t * n + x]) << (16 * (k & 1));
        }
        fp[x * FW + g] = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// Records q of the run of record p (the same signature, q < p) with at least
// `lim` as length are a suffix [first, p) of the run: its first record.
__device__ __forceinline__ uint32_t window_first(const uint64_t *__restrict__ rk, const uint64_t *__restrict__ rec,
                                                 uint32_t p, uint64_t key, int64_t lim) {
    const uint64_t vlim = lim > 0 ? (uint64_t)lim << 32 : 0ull;
    auto in = [&](uint32_t q) { return rk[q] == key && rec[q] >= vlim; };
    if (p == 0 || !in(p - 1)) return p;
    uint32_t good = p - 1, step = 1;   // in(good); gallop down
    while (good >= step && in(good - step)) {
        good -= step;
        step <<= 1;
    }
    // the boundary lies in (good - step, good]
    uint32_t lo = good >= step ? good - step + 1 : 0u;
    while (lo < good) {
        const uint32_t mid = (lo + good) >> 1;
        if (in(mid)) good = mid;
        else lo = mid + 1;
    }
    return good;
}

// The first record in [lo, end), ascending by length, of at least `lim` as length.
__device__ __forceinline__ uint32_t lower_len(const uint64_t *__restrict__ rec, uint32_t lo, uint32_t end, int64_t lim) {
    const uint64_t vlim = lim > 0 ? (uint64_t)lim << 32 : 0ull;
    while (lo < end) {
        const uint32_t mid = (lo + end) >> 1;
        if (rec[mid] >= vlim) end = mid;
        else lo = mid + 1;
    }
    return lo;
}

// x and y share a signature in some table before t: rows fx, fy of fingerprints,
// equal ones confirmed on the signatures.
__device__ __forceinline__ bool met_before(const uint4 *__restrict__ fx, const uint4 *__restrict__ fy, int32_t t,
                                           const uint64_t *__restrict__ keys, int64_t n, uint32_t x, uint32_t y) {
    for (int32_t t0 = 0; t0 < t; t0 += 8) {
        const uint4 a = __ldg(fx + (t0 >> 3)), b = __ldg(fy + (t0 >> 3));
        const uint32_t v[4] = {a.x ^ b.x, a.y ^ b.y, a.z ^ b.z, a.w ^ b.w};
        uint32_t z = 0;   // a zero half anywhere (also among the tables from t on, sorted out below)
#pragma unroll
        for (int i = 0; i < 4; i++) z |= (v[i] - 0x00010001u) & ~v[i] & 0x80008000u;
        if (z == 0u) continue;
#pragma unroll
        for (int k = 0; k < 8; k++) {
            const int32_t u = t0 + k;
            if (u < t && ((v[k >> 1] >> (16 * (k & 1))) & 0xFFFFu) == 0u && keys[(int64_t)u * n + x] == keys[(int64_t)u * n + y])
                return true;
        }
    }
    return false;
}

__global__ void __launch_bounds__(GE_WARPS * 32)
group_emit_kernel(const uint64_t *__restrict__ rk, const uint64_t *__restrict__ rec, const uint32_t *__restrict__ pos,
                  const uint64_t *__restrict__ keys, const uint4 *__restrict__ fp, int32_t FW,
                  const int32_t *__restrict__ lens, int64_t n, int32_t T, int32_t K, int32_t width, int32_t nclass,
                  int64_t tcap, int32_t chunk, uint64_t *__restrict__ pairs, uint32_t *__restrict__ tasks,
                  unsigned long long *__restrict__ counters) {
    __shared__ uint64_t s_stage[GE_WARPS][64];
    const int lane = threadIdx.x & 31;
    uint64_t *stage = s_stage[threadIdx.x >> 5];
    // the windows of the first GE_KEEP tables from class to class (own lane's entries)
    __shared__ uint32_t s_keep[GE_WARPS][2][GE_KEEP];
    uint32_t *keep_lo = s_keep[threadIdx.x >> 5][0], *keep_end = s_keep[threadIdx.x >> 5][1];
    const int64_t nw = (int64_t)gridDim.x * GE_WARPS;
    unsigned long long raw = 0, kept = 0;
    int64_t tnext = 0, tend = 0;   // the warp's task numbers left of its last reservation
    // pairs stage[0 .. cnt) leave as one task
    auto flush = [&](int cnt) {
        if (tnext == tend) {
            unsigned long long at = 0;
            if (lane == 0) at = atomicAdd(&counters[7], (unsigned long long)chunk);
            tnext = (int64_t)__shfl_sync(FULL, at, 0);
            tend = tnext + chunk;
        }
        if (tnext < tcap) {
            if (lane < cnt) pairs[tnext * 32 + lane] = stage[lane];
            if (lane == 0) tasks[tnext] = (uint32_t)cnt;
        }
        tnext++;
        kept += (unsigned)cnt;
        __syncwarp();
    };
    for (int64_t x = (int64_t)blockIdx.x * GE_WARPS + (threadIdx.x >> 5); x < n; x += nw) {   // warp-uniform
        const int64_t lx = lens[x];
        const uint4 *fx = fp + x * FW;
        int staged = 0;
        int32_t oldest = 0;   // the class of the first staged pair
        for (int32_t c = 0; c < nclass; c++) {
            // partners of lengths lx - dhi .. lx - dlo
            const int64_t dlo = (int64_t)c * width, dhi = min((int64_t)K, dlo + width - 1);
            if (dlo > lx) break;
            if (staged && c > oldest + 1) {   // two classes at most
                flush(staged);
                staged = 0;
            }
            for (int32_t t0 = 0; t0 < T; t0 += 32) {
                uint32_t first = 0, cnt = 0;
                const int32_t t = t0 + lane;
                if (t < T) {
                    const int64_t tb = (int64_t)t * n;
                    uint32_t lo = 0, end = 0;   // x's window in the table, without the classes done
                    if (c == 0 || t >= GE_KEEP) {
                        const uint32_t p = pos[tb + x];
                        const uint64_t key = rk[tb + p];
                        lo = end = p;
                        if (p > 0 && rk[tb + p - 1] == key) {
                            lo = window_first(rk + tb, rec + tb, p, key, lx - K);
                            if (c > 0) end = lower_len(rec + tb, lo, p, lx - dlo + 1);
                        }
                    } else {
                        lo = keep_lo[t];
                        end = keep_end[t];
                    }
                    first = c + 1 < nclass && lo < end ? lower_len(rec + tb, lo, end, lx - dhi) : lo;
                    cnt = end - first;
                    if (t < GE_KEEP && nclass > 1) {
                        keep_lo[t] = lo;
                        keep_end[t] = first;
                    }
                }
                if (!__any_sync(FULL, cnt > 0)) continue;
                uint32_t incl = cnt;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t v = __shfl_up_sync(FULL, incl, o);
                    if (lane >= o) incl += v;
                }
                const uint32_t total = __shfl_sync(FULL, incl, 31);
                raw += total;
                for (uint32_t base = 0; base < total; base += 32) {
                    // item -> (table, record): the first lane whose windows end beyond it
                    const uint32_t item = base + lane;
                    int l = 0;
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) {
                        const uint32_t v = __shfl_sync(FULL, incl, l + o - 1);
                        if (v <= item) l += o;
                    }
                    l = l < 31 ? l : 31;
                    const uint32_t ex = __shfl_sync(FULL, incl - cnt, l), f = __shfl_sync(FULL, first, l);
                    bool keep = false;
                    uint32_t y = 0;
                    if (item < total) {
                        const int32_t ti = t0 + l;
                        y = (uint32_t)rec[(int64_t)ti * n + f + (item - ex)];
                        keep = !met_before(fx, fp + (int64_t)y * FW, ti, keys, n, (uint32_t)x, y);
                    }
                    const unsigned mask = __ballot_sync(FULL, keep);
                    if (keep) {
                        const uint32_t xi = (uint32_t)x;
                        stage[staged + __popc(mask & ((1u << lane) - 1u))] =
                            xi < y ? ((uint64_t)xi << 32) | y : ((uint64_t)y << 32) | xi;
                    }
                    __syncwarp();
                    if (staged == 0) oldest = c;
                    staged += __popc(mask);
                    if (staged >= 32) {
                        flush(32);
                        staged -= 32;
                        const uint64_t rest = stage[32 + lane];
                        __syncwarp();
                        if (lane < staged) stage[lane] = rest;
                        __syncwarp();
                        oldest = c;   // what is left came with the last 32 items
                    }
                }
            }
        }
        if (staged) flush(staged);
    }
    // reserved and not used
    if (tnext + lane < tend && tnext + lane < tcap) tasks[tnext + lane] = 0u;
    if (lane == 0) {
        if (raw) atomicAdd(&counters[0], raw);
        if (kept) atomicAdd(&counters[2], kept);
    }
}

int group_blocks(int64_t n) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t need = (n + GE_WARPS - 1) / GE_WARPS, most = (int64_t)(sms > 0 ? sms : 1) * GE_BLOCKS;
    return (int)(need < most ? (need > 0 ? need : 1) : most);
}

// Task numbers a warp reserves at once (at most 32): fewer additions on the one
// counter, but tasks that a warp leaves unused are visited by the verifier. Whole joins
// of protein-like strings, K = 40, with 1 / 4 / 16: n = 5003 0.489 / 0.499 / 0.555 ms,
// 20000 1.93 / 1.93 / 2.15, 40000 5.54 / 5.43 / 5.64, 65536 12.9 / 12.4 / 12.6, 200000
// 107.5 / 102.9 / 103.1; text-like n = 120000, K = 200 with 4 / 8 / 16: 46.3 / 47.1 / 48.7.
int group_chunk(int64_t n) { return n >= 32768 ? 4 : 1; }

}  // namespace

int64_t group_task_cap(uint64_t cap, int64_t n, uint32_t nclass) {
    // whole tasks, the partial ones (the first classes of a string's partial tasks lie
    // at least two apart, and each holds a pair), and what the warps reserve and do not
    // use
    const uint64_t partial = (uint64_t)n * ((nclass + 1) / 2);
    return (int64_t)(cap / 32 + (partial < cap ? partial : cap)) + (int64_t)group_blocks(n) * GE_WARPS * group_chunk(n);
}

size_t fingerprint_bytes(int64_t n, int64_t T) { return (size_t)n * ((size_t)(T + 7) / 8) * sizeof(uint4); }

cudaError_t launch_group_prep(const uint64_t *rk, const uint32_t *rid, const uint64_t *keys, const int32_t *lens,
                              int64_t n, int64_t T, uint64_t *rec, uint32_t *pos, uint4 *fp,
                              unsigned long long *counters, cudaStream_t s) {
    if (n == 0 || T == 0) return cudaSuccess;
    const int64_t g = (n + 255) / 256;
    const int32_t FW = (int32_t)((T + 7) / 8);
    group_prep_kernel<<<dim3((unsigned)(g > 1024 ? 1024 : g), (unsigned)T), 256, 0, s>>>(rk, rid, lens, n, rec, pos,
                                                                                      counters);
    fingerprint_kernel<<<dim3((unsigned)(g > 4096 ? 4096 : g), (unsigned)FW), 256, 0, s>>>(keys, n, (int32_t)T, FW, fp);
    note_launches(2);
    return cudaGetLastError();
}

cudaError_t launch_group_emit(const uint64_t *rk, const uint64_t *rec, const uint32_t *pos, const uint64_t *keys,
                              const uint4 *fp, const int32_t *lens, int64_t n, int64_t T, int32_t K, uint32_t width,
                              uint32_t nclass, int64_t tcap, uint64_t *pairs, uint32_t *tasks,
                              unsigned long long *counters, cudaStream_t s) {
    if (width < 1 || nclass < 1) return cudaErrorInvalidValue;
    if (n == 0 || T == 0) return cudaSuccess;
    group_emit_kernel<<<group_blocks(n), GE_WARPS * 32, 0, s>>>(rk, rec, pos, keys, fp, (int32_t)((T + 7) / 8), lens, n,
                                                               (int32_t)T, K, (int32_t)width, (int32_t)nclass, tcap,
                                                               group_chunk(n), pairs, tasks, counters);
    note_launches(1);
    return cudaGetLastError();
}

}  // namespace ej

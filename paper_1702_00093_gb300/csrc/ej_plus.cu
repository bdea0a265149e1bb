// Device kernels of EmbedJoin+ (Section 5, Algorithms 4 and 5).
//
// Alg. 4 embeds, for every string s_i, the substrings (suffixes)
// s_{i,k} = s_i[(k-1)*delta ..] for k = 1 .. S (S = ceil(K/delta), at least 1).
// Here every suffix becomes a string of its own (record q = i*S + k-1), packed from
// its place in s_i, so that the ordinary fused walk signs it, and every record
// carries the length of its whole string for the length filter of Alg. 5.
// The hashed buckets then emit each pair of records that share a bucket in a
// table once per table: a record pair (q_a, q_b) is exactly Alg. 5's match
// (x, y, k_x, k_y). After a sort of the record pairs, a run of equal pairs is
// the count of that tuple over the tables; a pair of different strings with a
// count of at least T becomes a candidate (pairs of two substrings of one
// string share buckets too; they are counted apart and dropped).
#include "ej_internal.cuh"

namespace ej {

namespace {

// Record q = i*S + (k-1): its length sub_len[q] = max(0, |s_i| - (k-1)*delta), its
// chunks of B-bit codes (counts[n*S] = 0), its first byte's place in the byte array
// and whole_len[q] = |s_i|. The records are packed from there: their bytes are never
// copied (a copy of three suffixes of 20000 x 5000 bytes took 0.29 ms, validating
// and packing it again 0.2 ms more).
__global__ void suffix_records_kernel(const int32_t *__restrict__ lens, const int64_t *__restrict__ offsets, int64_t n,
                                      int32_t S, int32_t delta, int B, int32_t *__restrict__ sub_len,
                                      uint32_t *__restrict__ counts, int64_t *__restrict__ start,
                                      int32_t *__restrict__ whole_len) {
    const int64_t nq = n * (int64_t)S;
    if (blockIdx.x == 0 && threadIdx.x == 0) counts[nq] = 0u;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < nq; q += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = q / S;
        const int64_t skip = (q - i * S) * (int64_t)delta;
        const int32_t len = lens[i];
        const int64_t sub = skip < len ? len - skip : 0;
        sub_len[q] = (int32_t)sub;
        counts[q] = (uint32_t)chunks_for(sub, B);
        start[q] = offsets[i] + (len - sub);
        whole_len[q] = len;
    }
}

// Runs of equal record pairs in the sorted raw matches: a run of length >= T
// whose records belong to different strings appends the string pair
// (q_a / S) << 32 | (q_b / S) (each pair of records is one tuple; a string
// pair may come from several tuples, duplicates are removed afterwards).
__global__ void plus_runs_kernel(const uint64_t *__restrict__ sorted, int64_t nraw, int32_t S, int32_t T,
                                 uint64_t *__restrict__ out, unsigned long long cap,
                                 unsigned long long *__restrict__ count, unsigned long long *__restrict__ same) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nraw; e += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t v = sorted[e];
        if (e > 0 && sorted[e - 1] == v) continue;   // not the first of its run
        int64_t run = 1;
        while (e + run < nraw && sorted[e + run] == v) run++;   // at most one per table
        const uint64_t a = (v >> 32) / (uint64_t)S, b = (v & 0xFFFFFFFFull) / (uint64_t)S;
        if (a == b) {   // two substrings of one string: not a match of Alg. 5
            atomicAdd(same, (unsigned long long)run);
            continue;
        }
        if (run < T) continue;
        const unsigned long long idx = atomicAdd(count, 1ull);
        if (idx < cap) out[idx] = a < b ? (a << 32 | b) : (b << 32 | a);
    }
}

int grid_for(int64_t items, int threads) {
    int64_t b = (items + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > 65535LL * 16) b = 65535LL * 16;
    return (int)b;
}

}  // namespace

cudaError_t launch_suffix_records(const int32_t *lens, const int64_t *offsets, int64_t n, int32_t S, int32_t delta, int B,
                                  int32_t *sub_len, uint32_t *counts, int64_t *start, int32_t *whole_len, cudaStream_t s) {
    const int64_t nq = n * (int64_t)S;
    if (nq == 0) return cudaGetLastError();
    const int64_t g = (nq + 255) / 256;
    suffix_records_kernel<<<(unsigned)(g > 4096 ? 4096 : g), 256, 0, s>>>(lens, offsets, n, S, delta, B, sub_len, counts,
                                                                         start, whole_len);
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_plus_runs(const uint64_t *sorted, int64_t nraw, int32_t S, int32_t T, uint64_t *out,
                             uint64_t cap, unsigned long long *count, unsigned long long *same, cudaStream_t s) {
    if (nraw == 0) return cudaSuccess;
    plus_runs_kernel<<<grid_for(nraw, 256), 256, 0, s>>>(sorted, nraw, S, T, out, (unsigned long long)cap, count,
                                                          same);
    note_launches(1);
    return cudaGetLastError();
}

}  // namespace ej

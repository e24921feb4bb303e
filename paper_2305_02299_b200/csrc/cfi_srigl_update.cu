// cfi_srigl_update: one SRigL mask update of one layer on the device (Sec. 3.1, steps 1-7 "for each layer").
//
// Dense layout, as a training loop holds it: w[out][in] (zero where masked), mask[out][in] (0/1), grad[out][in].
// The update needs two selections over the whole layer -- the K smallest magnitudes among the active weights and the
// K largest gradient magnitudes among the inactive positions of live neurons -- and one selection per neuron (regrow
// to the new fan-in k', or trim down to it).  All of them are "the m smallest of a set of (32-bit key, position)
// pairs, ties to the smaller position", with key = the bits of |w| (a non-negative float orders like its bits) or
// the complement of the bits of |grad| (so that a larger gradient is a smaller key).  Key and position together are one
// 62-bit number, the composite, and no two elements share one, so ties need no ranking of their own.
//
// The two layer-wide selections are radix selections that stop sweeping the layer early.  One sweep counts the first 12
// bits of the keys, which leaves about 1 % of the elements open; a second one lists those, and the rest is decided on
// the lists.  Per neuron one 11-bit digit leaves a few dozen open, which are ranked against one another.  A layer with
// so many equal keys that the open elements do not fit the lists takes further digits first, at last of the position.
//
// 4096 x 4096 at 80 %, K = 30 % of the weights, four kernels: 34 + 41 + 16 + 60 us, 0.19 ms with the host's wait
// (before: four sweeps of 8-bit digits, flags for every entry and a four-digit selection per neuron, 12 kernels: 0.39 ms);
// 3072 x 768 at 90 %: 17 + 19 + 13 + 19 us, 0.10 ms (0.17 ms).  Moved per entry: 9 bytes in each of the two sweeps and the
// per-neuron step, and what changes: 30 against 50.
//
// Readings where Sec. 3.1 leaves a choice (the same as the CPU oracle used by the tests takes): already ablated
// neurons stay out; a weight is salient if it is active and not among the K smallest, or inactive and among the K
// largest gradients; a neuron is ablated if its salient count is below max(1, gamma_sal * k);
// k' = min(in, floor(k * live_before / live_after)); step 7 may regrow any position of the neuron that is not active
// at that moment (a weight pruned in step 6 included; grown weights start at 0); a neuron left with more than k'
// weights after step 6 loses its smallest down to k'.
#include "cfi.h"

#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <type_traits>

namespace {

constexpr int kThreads = 256;
constexpr int kDigit = 12, kBins = 1 << kDigit;  // layer-wide digits
constexpr int kKeyBits = 31, kPosBits = 31, kAllBits = kKeyBits + kPosBits;

// One layer-wide selection: the `want` smallest of its elements, as far as it is narrowed down.
struct Select {
    unsigned long long prefix;   // elements with (composite >> shift) < prefix are taken, > prefix are not, == are open
    unsigned long long want;     // how many of the open ones are still to take
    unsigned long long cut;      // after resolve_kernel: composite <= cut is taken
    unsigned int count;          // open elements
    unsigned int listed, listed_ties;  // entries of the two lists
    int shift;
    int on;                      // 0: nothing to select (K = 0 after clipping)
};

struct StateHead {               // what the host reads back
    Select sel[2];
    unsigned long long active_total;
    int live, k, blocks_done;
    int listable;                // both selections' open elements fit their lists
    int done;                    // resolve_kernel has run
    int k_new, live_after;
};
struct State : StateHead {       // zeroed before the first sweep
    alignas(16) unsigned int hist[2][kBins];
};

// 31-bit keys: the bits of |v| for a weight; for a gradient their complement, so that a larger one is a smaller key.
__device__ __forceinline__ unsigned int weight_key(float v) { return __float_as_uint(v) & 0x7FFFFFFFu; }
__device__ __forceinline__ unsigned int grad_key(float v) { return ~__float_as_uint(v) & 0x7FFFFFFFu; }
__device__ __forceinline__ unsigned long long composite(unsigned int key, unsigned int pos) {
    return ((unsigned long long)key << kPosBits) | pos;
}
// composite >> shift, with 32-bit arithmetic while the shift leaves key bits only.
__device__ __forceinline__ unsigned long long composite_top(unsigned int key, unsigned int pos, int shift) {
    if (shift >= kPosBits) return key >> (shift - kPosBits);
    return composite(key, pos) >> shift;
}

// VEC consecutive columns of a row: mask bytes (one per byte of m), weights, gradients.
template <int VEC> struct Cols;
template <> struct Cols<4> {
    unsigned int m;
    float4 w4, g4;
    __device__ __forceinline__ void load_mask(const uint8_t* mask, size_t at, bool in) { m = in ? *reinterpret_cast<const unsigned int*>(mask + at) : 0u; }
    __device__ __forceinline__ void load_values(const float* w, const float* grad, size_t at, bool in) {
        w4 = g4 = make_float4(0.f, 0.f, 0.f, 0.f);
        if (in) {
            w4 = *reinterpret_cast<const float4*>(w + at);
            g4 = *reinterpret_cast<const float4*>(grad + at);
        }
    }
    __device__ __forceinline__ bool on(int e) const { return (m >> (8 * e)) & 0xFFu; }
    __device__ __forceinline__ int count() const { return __popc(__vcmpne4(m, 0u)) >> 3; }
    __device__ __forceinline__ float w(int e) const { return e == 0 ? w4.x : e == 1 ? w4.y : e == 2 ? w4.z : w4.w; }
    __device__ __forceinline__ float g(int e) const { return e == 0 ? g4.x : e == 1 ? g4.y : e == 2 ? g4.z : g4.w; }
};
template <> struct Cols<1> {
    unsigned int m;
    float w1, g1;
    __device__ __forceinline__ void load_mask(const uint8_t* mask, size_t at, bool in) { m = in ? mask[at] : 0u; }
    __device__ __forceinline__ void load_values(const float* w, const float* grad, size_t at, bool in) {
        w1 = in ? w[at] : 0.f;
        g1 = in ? grad[at] : 0.f;
    }
    __device__ __forceinline__ bool on(int) const { return m != 0u; }
    __device__ __forceinline__ int count() const { return m != 0u; }
    __device__ __forceinline__ float w(int) const { return w1; }
    __device__ __forceinline__ float g(int) const { return g1; }
};

// Programmatic dependent launch: a kernel of the chain may start while the one before it ends, and waits for it before it
// reads what that one writes.  (Every block waits, so a kernel that has ended has also seen the end of all before it.)
// An update of 3072 x 768 99.4 -> 95.9 us, of 4096 x 4096 216 -> 212.
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Sum over the block of one int per thread; slot alternates between calls so that one barrier per call is enough.
template <int T>
__device__ __forceinline__ int block_sum(int v, int (&part)[2][T / 32], int slot) {
    v = __reduce_add_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0) part[slot][threadIdx.x >> 5] = v;
    __syncthreads();
    int total = 0;
#pragma unroll
    for (int i = 0; i < T / 32; ++i) total += part[slot][i];
    return total;
}

// The bin of a histogram that holds the `want`-th element (1-based; the caller guarantees that there are so many), how
// many elements the bins before it hold and how many it holds itself.  The whole block, T threads, the kPer consecutive bins v of each.
struct Pick { unsigned int bin, below, count; };
template <int T, int kPer>
__device__ Pick block_pick(unsigned long long want, const unsigned int (&v)[kPer], unsigned int* part, Pick& out) {
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    unsigned int mine = 0;
#pragma unroll
    for (int e = 0; e < kPer; ++e) mine += v[e];
    unsigned int incl = mine;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const unsigned int up = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += up;
    }
    if (lane == 31) part[wid] = incl;
    __syncthreads();
    unsigned int seen = incl - mine;
#pragma unroll
    for (int i = 0; i < T / 32; ++i) seen += i < wid ? part[i] : 0u;
    if (seen < want && want <= (unsigned long long)seen + mine) {  // exactly one thread
        bool found = false;
#pragma unroll
        for (int e = 0; e < kPer; ++e) {
            if (!found && want <= (unsigned long long)seen + v[e]) {
                out = Pick{(unsigned int)(kPer * t + e), seen, v[e]};
                found = true;
            }
            if (!found) seen += v[e];
        }
    }
    __syncthreads();
    return out;
}

// Called by the block of a sweep whose counts arrive last: both selections take their next digit from the histograms,
// which are cleared for the next sweep.
__device__ void narrow(State* st, bool first, long long K, int in_f, unsigned int cap) {
    __shared__ unsigned int part[kThreads / 32];
    __shared__ Pick pick;
    __shared__ Select q[2];
    constexpr int kPer = kBins / kThreads;
    const int t = threadIdx.x;
    uint4 v[2][kPer / 4];  // both histograms and the totals are on their way together: one trip to L2
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int i = 0; i < kPer / 4; ++i) v[s][i] = __ldcg(reinterpret_cast<const uint4*>(st->hist[s]) + t * (kPer / 4) + i);
    if (t == 0) {
        if (first) {
            const unsigned long long act = __ldcg(&st->active_total);
            const unsigned long long inact = (unsigned long long)__ldcg(&st->live) * in_f - act;
            unsigned long long kk = K < 0 ? 0ull : (unsigned long long)K;
            kk = kk > act ? act : kk;
            kk = kk > inact ? inact : kk;
            for (int s = 0; s < 2; ++s) {
                Select z{};
                z.want = kk, z.on = kk != 0, z.shift = kAllBits;
                z.count = (unsigned int)(s ? inact : act);  // at most 2^31
                q[s] = z;
            }
        } else {
            for (int s = 0; s < 2; ++s) {
                q[s] = st->sel[s];
                q[s].listed = __ldcg(&st->sel[s].listed);
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        const int digit = q[s].shift < kDigit ? q[s].shift : kDigit;
        if (q[s].on && digit > 0) {
            unsigned int bins[kPer];
#pragma unroll
            for (int i = 0; i < kPer / 4; ++i) bins[4 * i] = v[s][i].x, bins[4 * i + 1] = v[s][i].y, bins[4 * i + 2] = v[s][i].z, bins[4 * i + 3] = v[s][i].w;
            const Pick p = block_pick<kThreads>(q[s].want, bins, part, pick);
            if (t == 0) {
                q[s].prefix = (q[s].prefix << digit) | p.bin;
                q[s].shift -= digit;
                q[s].want -= p.below;
                q[s].count = p.count;
            }
        }
#pragma unroll
        for (int i = 0; i < kPer / 4; ++i) reinterpret_cast<uint4*>(st->hist[s])[t * (kPer / 4) + i] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
    }
    if (t < 2) st->sel[t] = q[t];
    if (t == 0) st->listable = (!q[0].on || q[0].count <= cap) && (!q[1].on || q[1].count <= cap);
}

// True in every thread of the block of this launch that gets here last; everything the other blocks wrote is visible.
__device__ bool last_block(int* done) {
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        last = atomicAdd(done, 1) == (int)gridDim.x - 1;
        if (last) *done = 0, __threadfence();
    }
    __syncthreads();
    return last;
}

// A sweep over the layer that counts the next digit of both selections' open elements; a block takes whole rows.  The
// first sweep also counts the rows' weights (FIRST; whether a position of the gradient pool counts depends on whether
// its row has any).  Later ones run only for layers with so many equal keys that a digit's open elements exceed the lists.
//
// Bound by memory: 9 bytes per entry, 4.4 TB/s on 4096 x 4096.  A thread has mask, weights and gradients of four chunks in
// flight, of one row or of two or four short ones (3072 x 768: 21 us with one row at a time, 17 with four).  12-bit digits: a first digit of 8 exponent and 4 mantissa bits leaves about 1 % of the elements open, few
// enough to list them in the next sweep instead of sweeping again for every digit.
template <int VEC, int ROWS, bool FIRST>
__global__ void __launch_bounds__(kThreads, 4) sweep_kernel(const float* w, const uint8_t* mask, const float* grad, int* row_count, int out_f,
                                                         int in_f, long long K, unsigned int cap, State* st) {
    extern __shared__ unsigned int h[];  // [2][kBins]
    __shared__ int part[2][ROWS][kThreads / 32];
    constexpr int kAhead = (VEC == 4 ? 4 : 8) / ROWS;  // chunks of each row
    const int t = threadIdx.x;
    let_next_start();
    for (int b = t; b < 2 * kBins; b += kThreads) h[b] = 0;
    int shift[2] = {kAllBits, kAllBits}, digit[2] = {kDigit, kDigit};
    unsigned long long prefix[2] = {0, 0};
    bool on[2] = {true, true};
    if (!FIRST) {
        for (int s = 0; s < 2; ++s) {
            prefix[s] = st->sel[s].prefix, shift[s] = st->sel[s].shift, on[s] = st->sel[s].on != 0;
            digit[s] = shift[s] < kDigit ? shift[s] : kDigit;
        }
    }
    __syncthreads();
    unsigned long long total = 0;
    int live = 0, k = 0, slot = 0;
    auto count = [&](const Cols<VEC>& c, bool in, int col, size_t base) {
#pragma unroll
        for (int e = 0; e < VEC; ++e) {
            if (!in) continue;
            const int s = c.on(e) ? 0 : 1;
            const unsigned int key = s ? grad_key(c.g(e)) : weight_key(c.w(e));
            if (FIRST) {
                atomicAdd(&h[s * kBins + (key >> (kKeyBits - kDigit))], 1u);
            } else if (on[s]) {
                const unsigned int pos = (unsigned int)(base + col + e);
                if (composite_top(key, pos, shift[s]) == prefix[s])
                    atomicAdd(&h[s * kBins + (int)(composite_top(key, pos, shift[s] - digit[s]) & ((1u << digit[s]) - 1u))], 1u);
            }
        }
    };
    for (long long r0 = blockIdx.x; r0 < out_f; r0 += (long long)ROWS * gridDim.x) {
        Cols<VEC> c[ROWS][kAhead];
#pragma unroll
        for (int j = 0; j < ROWS; ++j) {
            const long long r = r0 + (long long)j * gridDim.x;
#pragma unroll
            for (int u = 0; u < kAhead; ++u) {
                const int col = (u * kThreads + t) * VEC;
                c[j][u].load_mask(mask, (size_t)r * in_f + col, r < out_f && col < in_f);
                c[j][u].load_values(w, grad, (size_t)r * in_f + col, r < out_f && col < in_f);
            }
        }
        if (FIRST) {
#pragma unroll
            for (int j = 0; j < ROWS; ++j) {
                int mine = 0;
#pragma unroll
                for (int u = 0; u < kAhead; ++u) mine += c[j][u].count();
                for (int col = (kAhead * kThreads + t) * VEC; ROWS == 1 && col < in_f; col += kThreads * VEC) {
                    Cols<VEC> m;
                    m.load_mask(mask, (size_t)r0 * in_f + col, true);
                    mine += m.count();
                }
                mine = __reduce_add_sync(0xffffffffu, mine);
                if ((t & 31) == 0) part[slot][j][t >> 5] = mine;
            }
            __syncthreads();  // one per step: the slots alternate
        }
#pragma unroll
        for (int j = 0; j < ROWS; ++j) {
            const long long r = r0 + (long long)j * gridDim.x;
            if (r >= out_f) continue;
            int n = 0;
            if (FIRST) {
#pragma unroll
                for (int i = 0; i < kThreads / 32; ++i) n += part[slot][j][i];
                if (t == 0) row_count[r] = n, total += n, live += n > 0, k = max(k, n);
            } else {
                n = row_count[r];
            }
            if (n == 0) continue;  // a neuron without weights is in neither pool
            const size_t base = (size_t)r * in_f;
#pragma unroll
            for (int u = 0; u < kAhead; ++u) count(c[j][u], (u * kThreads + t) * VEC < in_f, (u * kThreads + t) * VEC, base);
            for (int c0 = kAhead * kThreads * VEC; ROWS == 1 && c0 < in_f; c0 += kAhead * kThreads * VEC) {
#pragma unroll
                for (int u = 0; u < kAhead; ++u) {
                    const int col = c0 + (u * kThreads + t) * VEC;
                    c[j][u].load_mask(mask, base + col, col < in_f);
                    c[j][u].load_values(w, grad, base + col, col < in_f);
                }
#pragma unroll
                for (int u = 0; u < kAhead; ++u) count(c[j][u], c0 + (u * kThreads + t) * VEC < in_f, c0 + (u * kThreads + t) * VEC, base);
            }
        }
        slot ^= 1;
    }
    __syncthreads();
    for (int b = t; b < 2 * kBins; b += kThreads)
        if (h[b]) atomicAdd(&st->hist[b / kBins][b % kBins], h[b]);
    if (FIRST && t == 0 && live) {
        atomicAdd(&st->active_total, total);
        atomicAdd(&st->live, live);
        atomicMax(&st->k, k);
    }
    if (last_block(&st->blocks_done)) narrow(st, FIRST, K, in_f, cap);
}

// The last sweep: lists the open elements of both selections (key, position), counts their next digit, and counts per
// row the weights that are salient whatever becomes of the open ones.  Listed elements are gathered in shared memory
// and leave it together, so that the list's length is one global atomic per block and not one per element.
template <int VEC, int ROWS>
__global__ void __launch_bounds__(kThreads, 4) collect_kernel(const float* w, const uint8_t* mask, const float* grad, const int* row_count, int out_f,
                                                           int in_f, unsigned int cap, uint2* list, int* salient, State* st) {
    constexpr int kAhead = (VEC == 4 ? 4 : 8) / ROWS;  // chunks of each row
    constexpr unsigned int kBuf = 1024;
    __shared__ uint2 buf[2][kBuf];
    __shared__ unsigned int n_buf[2], at_buf[2];
    __shared__ int part[2][ROWS][kThreads / 32];
    let_next_start();
    wait_for_previous();
    if (!st->listable) return;
    const int t = threadIdx.x;
    if (t < 2) n_buf[t] = 0;
    // Both selections take the same number of elements, so both are on or off and have consumed the same digits.
    const unsigned long long prefix0 = st->sel[0].prefix, prefix1 = st->sel[1].prefix;
    const bool on = st->sel[0].on != 0;
    const int shift = st->sel[0].shift, digit = shift < kDigit ? shift : kDigit;
    // The cuts as the leading digits of a magnitude (a gradient's key is the complement of its bits).
    const int key_shift = shift - kPosBits;
    const unsigned int key_tops = key_shift > 0 ? 0x7FFFFFFFu >> key_shift : 0x7FFFFFFFu;
    const unsigned int top_w = (unsigned int)prefix0, top_g = key_tops - (unsigned int)prefix1;
    auto push = [&](bool is_w, unsigned int key, unsigned int pos) {
        const int s = is_w ? 0 : 1;
        atomicAdd(&st->hist[s][composite_top(key, pos, shift - digit) & ((1u << digit) - 1u)], 1u);
        const unsigned int at = atomicAdd(&n_buf[s], 1u);
        if (at < kBuf) {
            buf[s][at] = make_uint2(key, pos);
        } else {  // a row with more open elements than the buffer holds
            const unsigned int g = atomicAdd(&st->sel[s].listed, 1u);
            if (g < cap) list[(size_t)s * cap + g] = make_uint2(key, pos);
        }
    };
    __syncthreads();
    int slot = 0;
    auto flush = [&]() {  // whole block
        __syncthreads();
        if (t < 2) {
            const unsigned int n = n_buf[t] < kBuf ? n_buf[t] : kBuf;
            at_buf[t] = n ? atomicAdd(&st->sel[t].listed, n) : 0u;
        }
        __syncthreads();
#pragma unroll
        for (int s = 0; s < 2; ++s)
            for (unsigned int i = t; i < (n_buf[s] < kBuf ? n_buf[s] : kBuf); i += kThreads)
                if (at_buf[s] + i < cap) list[(size_t)s * cap + at_buf[s] + i] = buf[s][i];
        __syncthreads();
        if (t < 2) n_buf[t] = 0;
        __syncthreads();
    };
    for (long long r0 = blockIdx.x; r0 < out_f; r0 += (long long)ROWS * gridDim.x) {
        int weights[ROWS], mine[ROWS];
#pragma unroll
        for (int j = 0; j < ROWS; ++j) {
            const long long r = r0 + (long long)j * gridDim.x;
            weights[j] = r < out_f ? row_count[r] : 0, mine[j] = 0;
        }
        for (int c0 = 0; c0 < in_f; c0 += kAhead * kThreads * VEC) {
            Cols<VEC> c[ROWS][kAhead];
#pragma unroll
            for (int j = 0; j < ROWS; ++j)
#pragma unroll
                for (int u = 0; u < kAhead; ++u) {
                    const long long r = r0 + (long long)j * gridDim.x;
                    const int col = c0 + (u * kThreads + t) * VEC;
                    c[j][u].load_mask(mask, (size_t)r * in_f + col, r < out_f && col < in_f);
                    c[j][u].load_values(w, grad, (size_t)r * in_f + col, r < out_f && col < in_f);
                }
#pragma unroll
            for (int j = 0; j < ROWS; ++j)
#pragma unroll
            for (int u = 0; u < kAhead; ++u) {
                const int col = c0 + (u * kThreads + t) * VEC;
                // no weights: in neither pool; selections off: nothing is pruned and nothing grown
                if (col >= in_f || weights[j] == 0 || !on) continue;
                const size_t base = (size_t)(r0 + (long long)j * gridDim.x) * in_f;
                if (key_shift >= 0) {
                    // |v| against the selection's cut, both in the digits found so far.  In magnitudes a weight above its
                    // cut stays and a gradient above its cut is taken: salient either way, so the two need no branches.
                    bool open[VEC], any = false;
#pragma unroll
                    for (int e = 0; e < VEC; ++e) {
                        const bool is_w = c[j][u].on(e);
                        const unsigned int top = weight_key(is_w ? c[j][u].w(e) : c[j][u].g(e)) >> key_shift, at = is_w ? top_w : top_g;
                        mine[j] += top > at;
                        open[e] = top == at;
                        any |= open[e];
                    }
                    if (any) {
#pragma unroll
                        for (int e = 0; e < VEC; ++e)
                            if (open[e]) push(c[j][u].on(e), c[j][u].on(e) ? weight_key(c[j][u].w(e)) : grad_key(c[j][u].g(e)), (unsigned int)(base + col + e));
                    }
                } else {  // position digits: very many equal keys
                    for (int e = 0; e < VEC; ++e) {
                        const bool is_w = c[j][u].on(e);
                        const unsigned int key = is_w ? weight_key(c[j][u].w(e)) : grad_key(c[j][u].g(e)), pos = (unsigned int)(base + col + e);
                        const unsigned long long top = composite_top(key, pos, shift), at = is_w ? prefix0 : prefix1;
                        mine[j] += is_w ? top > at : top < at;
                        if (top == at) push(is_w, key, pos);
                    }
                }
            }
        }
#pragma unroll
        for (int j = 0; j < ROWS; ++j) {
            const int n = __reduce_add_sync(0xffffffffu, mine[j]);
            if ((t & 31) == 0) part[slot][j][t >> 5] = n;
        }
        __syncthreads();  // also completes these rows' entries
        const long long mine_r = r0 + (long long)t * gridDim.x;
        if (t < ROWS && mine_r < out_f) {
            int n = 0;
#pragma unroll
            for (int i = 0; i < kThreads / 32; ++i) n += part[slot][t][i];
            salient[mine_r] = on ? n : row_count[mine_r];
        }
        slot ^= 1;
        const bool full = n_buf[0] > kBuf / 2 || n_buf[1] > kBuf / 2;
        if (__syncthreads_or(full)) flush();
    }
    flush();
    if (last_block(&st->blocks_done)) narrow(st, false, 0, in_f, cap);
}

// For lists in which one digit leaves too many elements open (very many equal keys): one more digit of both selections,
// counted over the lists.
__global__ void list_sweep_kernel(const uint2* list, unsigned int cap, int in_f, State* st) {
    const unsigned int first = blockIdx.x * kThreads + threadIdx.x, step = gridDim.x * kThreads;
    for (int s = 0; s < 2; ++s) {
        const Select q = st->sel[s];
        if (!q.on) continue;
        const int digit = q.shift < kDigit ? q.shift : kDigit;
        for (unsigned int i = first; i < q.listed; i += step) {
            const uint2 e = list[(size_t)s * cap + i];
            if (composite_top(e.x, e.y, q.shift) == q.prefix)
                atomicAdd(&st->hist[s][composite_top(e.x, e.y, q.shift - digit) & ((1u << digit) - 1u)], 1u);
        }
    }
    if (last_block(&st->blocks_done)) narrow(st, false, 0, in_f, cap);
}

// The `want`-th smallest composite (1-based) of `count` elements that the block's threads enumerate:
// visit(f) calls f(key, pos) for each element, every element in exactly one thread.  Digits of 11 bits narrow the
// elements down until there is at most one per thread; these are ranked against one another.
constexpr unsigned int kRowBins = 2048;
template <int T>
struct SelectSmem {
    alignas(16) unsigned int hist[kRowBins];
    unsigned long long open[T];
    unsigned long long result;
    unsigned int part[T / 32], n;
    Pick pick;
};
//
// Where the caller knows the smallest key (base, else 0), the first histogram is of 64 bins a binade from there on instead of
// the 11 leading bits, which are 8 a binade: most gradients of a row lie within two binades of one another, so with those a
// warp's counts met in a few bins and were added one after the other (4096 x 4096: finalize_kernel 73 -> 60 us).  A bin that holds too many all the same (its elements equal, or 32 binades and more away) leaves it to the leading bits.
constexpr int kFineShift = 23 - 6;
template <int T, typename Visit>
__device__ unsigned long long block_select(unsigned int want, unsigned int count, Visit visit, SelectSmem<T>& sm, unsigned int base = 0) {
    const int t = threadIdx.x;
    constexpr int kPer = kRowBins / T;
    auto clear = [&]() {
#pragma unroll
        for (int i = 0; i < kPer / 4; ++i) reinterpret_cast<uint4*>(sm.hist)[i * T + t] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
    };
    auto find = [&]() {
        __syncthreads();
        unsigned int bins[kPer];
#pragma unroll
        for (int i = 0; i < kPer / 4; ++i) {
            const uint4 q = reinterpret_cast<const uint4*>(sm.hist)[t * (kPer / 4) + i];
            bins[4 * i] = q.x, bins[4 * i + 1] = q.y, bins[4 * i + 2] = q.z, bins[4 * i + 3] = q.w;
        }
        return block_pick<T>(want, bins, sm.part, sm.pick);
    };
    unsigned long long prefix = 0;
    int shift = kAllBits;
    bool fine = false;
    unsigned int fine_bin = 0;
    if (base != 0 && count > T) {
        clear();
        visit([&](unsigned int key, unsigned int) { atomicAdd(&sm.hist[min((key - base) >> kFineShift, kRowBins - 1u)], 1u); });
        const Pick p = find();
        if (p.count <= T) fine = true, fine_bin = p.bin, want -= p.below, count = p.count;
        __syncthreads();
    }
    while (!fine && count > T && shift > 0) {
        const int digit = shift < 11 ? shift : 11;
        clear();
        if (shift == kAllBits) {
            visit([&](unsigned int key, unsigned int) { atomicAdd(&sm.hist[key >> (kKeyBits - 11)], 1u); });
        } else {
            visit([&](unsigned int key, unsigned int pos) {
                if (composite_top(key, pos, shift) == prefix)
                    atomicAdd(&sm.hist[composite_top(key, pos, shift - digit) & ((1u << digit) - 1u)], 1u);
            });
        }
        const Pick p = find();
        want -= p.below, count = p.count;
        prefix = (prefix << digit) | p.bin;
        shift -= digit;
    }
    if (t == 0) sm.n = 0;
    __syncthreads();
    auto list = [&](unsigned int key, unsigned int pos) {
        const unsigned int at = atomicAdd(&sm.n, 1u);
        if (at < T) sm.open[at] = composite(key, pos);
    };
    if (fine) {  // the usual end
        visit([&](unsigned int key, unsigned int pos) {
            if (min((key - base) >> kFineShift, kRowBins - 1u) == fine_bin) list(key, pos);
        });
    } else if (shift >= kPosBits) {  // a key digit left few enough
        const int key_shift = shift - kPosBits;
        const unsigned int top = (unsigned int)prefix;
        visit([&](unsigned int key, unsigned int pos) {
            if (key >> key_shift == top) list(key, pos);
        });
    } else {
        visit([&](unsigned int key, unsigned int pos) {
            if (composite(key, pos) >> shift == prefix) list(key, pos);
        });
    }
    __syncthreads();
    if ((unsigned int)t < count) {
        const unsigned long long mine = sm.open[t];
        unsigned int rank = 0;
#pragma unroll 8
        for (unsigned int i = 0; i < count; ++i) rank += sm.open[i] < mine;
        if (rank == want - 1) sm.result = mine;
    }
    __syncthreads();
    const unsigned long long result = sm.result;
    __syncthreads();
    return result;
}

// Decides the listed elements: those below the cut's digits are taken, those above are not, and the last block finds the
// cut among the few that are left.  Salient counts are completed on the way, then steps 4 and 5 (who is ablated, the new
// fan-in) follow from them.
__global__ void __launch_bounds__(kThreads) resolve_kernel(const uint2* list, unsigned int cap, uint2* ties, unsigned int ties_cap, const int* row_count,
                                                           int* salient, uint8_t* survives, int out_f, int in_f, float gamma_sal, State* st) {
    __shared__ SelectSmem<kThreads> sm;
    __shared__ int part[2][kThreads / 32];
    let_next_start();
    wait_for_previous();
    if (!st->listable) return;
    for (int s = 0; s < 2; ++s)
        if (st->sel[s].on && st->sel[s].count > ties_cap) return;  // another digit first (list_sweep_kernel)
    const int t = threadIdx.x;
    const unsigned int first = blockIdx.x * kThreads + t, step = gridDim.x * kThreads;
    for (int s = 0; s < 2; ++s) {
        if (!st->sel[s].on) continue;
        const unsigned long long prefix = st->sel[s].prefix;
        const int shift = st->sel[s].shift;
        const unsigned int n = st->sel[s].listed;
        for (unsigned int i = first; i < n; i += step) {
            const uint2 e = list[(size_t)s * cap + i];
            const unsigned long long top = composite_top(e.x, e.y, shift);
            if (top == prefix) {
                const unsigned int at = atomicAdd(&st->sel[s].listed_ties, 1u);
                if (at < ties_cap) ties[(size_t)s * ties_cap + at] = e;
            } else if ((s == 0) == (top > prefix)) {
                atomicAdd(&salient[e.y / (unsigned int)in_f], 1);  // a weight that stays, a gradient that is taken
            }
        }
    }
    if (!last_block(&st->blocks_done)) return;
    for (int s = 0; s < 2; ++s) {
        const Select& q = st->sel[s];
        if (!q.on) continue;
        const unsigned int n = __ldcg(&q.listed_ties);
        const uint2* mine = ties + (size_t)s * ties_cap;
        const uint2 own = t < (int)n ? __ldcg(&mine[t]) : make_uint2(0u, 0u);
        const unsigned long long cut = block_select<kThreads>((unsigned int)q.want, n, [&](auto f) {
            if (t < (int)n) f(own.x, own.y);
            for (unsigned int i = t + kThreads; i < n; i += kThreads) {
                const uint2 e = __ldcg(&mine[i]);
                f(e.x, e.y);
            }
        }, sm);
        for (unsigned int i = t; i < n; i += kThreads) {
            const uint2 e = __ldcg(&mine[i]);
            if ((s == 0) == (composite(e.x, e.y) > cut)) atomicAdd(&salient[e.y / (unsigned int)in_f], 1);
        }
        if (t == 0) st->sel[s].cut = cut;
        __syncthreads();
    }
    __threadfence();
    __syncthreads();
    // Steps 4 and 5.
    const double threshold = fmax(1.0, (double)gamma_sal * (double)st->k);
    int mine = 0;
    for (int r0 = t; r0 < out_f; r0 += 8 * kThreads) {  // eight rows' loads in flight: one block walks all rows
        int rc[8], sa[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int r = r0 + u * kThreads;
            rc[u] = r < out_f ? row_count[r] : 0, sa[u] = r < out_f ? __ldcg(&salient[r]) : 0;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int r = r0 + u * kThreads;
            if (r < out_f) {
                const bool live = rc[u] > 0 && !((double)sa[u] < threshold);
                survives[r] = live ? 1 : 0;
                mine += live ? 1 : 0;
            }
        }
    }
    const int after = block_sum<kThreads>(mine, part, 0);
    if (t == 0) {
        long long kn = after > 0 ? ((long long)st->k * st->live) / after : 0;
        if (kn > in_f) kn = in_f;
        st->k_new = (int)kn, st->live_after = after, st->done = 1;
    }
}

// Steps 6 and 7 for one neuron per block: prune, then trim or regrow to k'.  A thread keeps the keys of its columns (rows of
// up to COLS columns) in registers, so that the row is read once; longer rows (COLS = 0) are read again for every visit.
//
// 9 bytes read per entry, and of the outputs only what changes is written (a masked-off weight is 0 already, a kept one
// keeps its value); bound by instruction issue as much as by memory, hence the one key per column: columns that cannot be
// chosen carry kNoKey, above every key, and every later step is a compare (4096 x 4096: 105 us with 62-bit compares per
// column, 73 with these, 60 with the finer first histogram of block_select).  The selection takes two visits of the row as a
// rule: one histogram, then the few elements left in its bin are ranked against one another.
constexpr unsigned int kNoKey = 0xFFFFFFFFu;
template <int VEC, int COLS, int T>
__global__ void __launch_bounds__(T, (COLS > 2048 ? 1024 : 1536) / T) finalize_kernel(float* w, uint8_t* mask, const float* grad, const uint8_t* survives,
                                                                              int in_f, const State* st) {
    __shared__ SelectSmem<T> sm;
    __shared__ int part[2][T / 32];
    constexpr bool kCached = COLS > 0;
    constexpr int kChunks = kCached ? COLS / (T * VEC) : 1;
    const int r = blockIdx.x, t = threadIdx.x;
    const size_t base = (size_t)r * in_f;
    float* wr = w + base;
    uint8_t* mr = mask + base;
    const float* gr = grad + base;
    Cols<VEC> c[kChunks];
    if (kCached) {  // on the way while the flags below are read
#pragma unroll
        for (int u = 0; u < kChunks; ++u) {
            const int col = (u * T + t) * VEC;
            c[u].load_mask(mr, col, col < in_f);
            c[u].load_values(wr, gr, col, col < in_f);
        }
    }
    wait_for_previous();  // the rows themselves are written by no kernel before this one
    if (!st->done) return;
    if (!survives[r]) {  // ablated now or before: nothing left
        for (int c = t * VEC; c < in_f; c += T * VEC) {
            if (VEC == 4) *reinterpret_cast<float4*>(wr + c) = make_float4(0.f, 0.f, 0.f, 0.f), *reinterpret_cast<unsigned int*>(mr + c) = 0u;
            else wr[c] = 0.0f, mr[c] = 0;
        }
        return;
    }
    const int k_new = st->k_new;
    const bool on0 = st->sel[0].on != 0;
    const unsigned int cut_key = (unsigned int)(st->sel[0].cut >> kPosBits);
    // Position of the last pruned weight of magnitude cut_key, as a column of this row.
    const long long cut_col = (long long)(st->sel[0].cut & 0x7FFFFFFFull) - (long long)base;
    // Kept after step 6: in the mask and not among the K smallest of the layer.
    auto is_kept = [&](const Cols<VEC>& c, int e, int col) {
        const unsigned int u = weight_key(c.w(e));
        const bool dropped = u < cut_key || (u == cut_key && (long long)(col + e) <= cut_col);
        return c.on(e) && !(on0 && dropped);
    };
    __shared__ unsigned int least[T / 32];
    unsigned int key[kChunks][VEC], kept_bits[kChunks], lowest = kNoKey;
    int mine = 0;
    if (kCached) {
#pragma unroll
        for (int u = 0; u < kChunks; ++u) {
            const int col = (u * T + t) * VEC;
            kept_bits[u] = 0;
#pragma unroll
            for (int e = 0; e < VEC; ++e) {
                const bool kept = is_kept(c[u], e, col);
                if (!kept && __float_as_uint(c[u].w(e)) != 0u) wr[col + e] = 0.0f;  // pruned, or free (a weight grown later starts at 0)
                kept_bits[u] |= kept ? 1u << e : 0u;
                key[u][e] = kept || col >= in_f ? kNoKey : grad_key(c[u].g(e));
                lowest = min(lowest, key[u][e]);
            }
            mine += __popc(kept_bits[u]);
        }
        lowest = __reduce_min_sync(0xffffffffu, lowest);
        if ((t & 31) == 0) least[t >> 5] = lowest;
    } else {
        for (int col = t * VEC; col < in_f; col += T * VEC) {
            Cols<VEC> v;
            v.load_mask(mr, col, true);
            v.load_values(wr, gr, col, true);
#pragma unroll
            for (int e = 0; e < VEC; ++e) mine += is_kept(v, e, col) ? 1 : 0;
        }
    }
    const int kept = block_sum<T>(mine, part, 0);
    if (kCached) {
#pragma unroll
        for (int i = 0; i < T / 32; ++i) lowest = min(lowest, least[i]);
    }
    const bool trim = kept > k_new;
    const int m = trim ? kept - k_new : k_new - kept;
    if (kCached && trim) {  // the other keys: magnitudes of the kept weights
#pragma unroll
        for (int u = 0; u < kChunks; ++u)
#pragma unroll
            for (int e = 0; e < VEC; ++e) key[u][e] = (kept_bits[u] >> e) & 1u ? weight_key(wr[(u * T + t) * VEC + e]) : kNoKey;
    }
    // Trim: the kept weights with the smallest magnitudes go; otherwise the free positions with the largest gradient
    // magnitudes come.  Ties go to the smaller column.
    unsigned long long cut = 0;
    if (m > 0) {
        cut = block_select<T>((unsigned int)m, (unsigned int)(trim ? kept : in_f - kept), [&](auto f) {
            if (kCached) {
#pragma unroll
                for (int u = 0; u < kChunks; ++u)
#pragma unroll
                    for (int e = 0; e < VEC; ++e)
                        if (key[u][e] != kNoKey) f(key[u][e], (unsigned int)((u * T + t) * VEC + e));
            } else {
                for (int col = t * VEC; col < in_f; col += T * VEC) {
                    Cols<VEC> v;
                    v.load_mask(mr, col, true);
                    v.load_values(wr, gr, col, true);
#pragma unroll
                    for (int e = 0; e < VEC; ++e)
                        if (is_kept(v, e, col) == trim) f(trim ? weight_key(v.w(e)) : grad_key(v.g(e)), (unsigned int)(col + e));
                }
            }
        }, sm, kCached && !trim ? lowest : 0u);
    }
    const unsigned int row_key = (unsigned int)(cut >> kPosBits), row_col = (unsigned int)(cut & 0x7FFFFFFFull);
    auto chosen = [&](unsigned int k, int col) { return m > 0 && (k < row_key || (k == row_key && (unsigned int)col <= row_col)); };
    if (kCached) {
#pragma unroll
        for (int u = 0; u < kChunks; ++u) {
            const int col = (u * T + t) * VEC;
            if (col >= in_f) continue;
            unsigned int out = 0;
#pragma unroll
            for (int e = 0; e < VEC; ++e) {
                const bool flip = chosen(key[u][e], col + e);  // a kept one goes, a free one comes
                if (trim && flip) wr[col + e] = 0.0f;
                out |= (((kept_bits[u] >> e) & 1u) != 0u) != flip ? 1u << (8 * e) : 0u;
            }
            if (VEC == 4) *reinterpret_cast<unsigned int*>(mr + col) = out;
            else mr[col] = (uint8_t)out;
        }
    } else {
        for (int col = t * VEC; col < in_f; col += T * VEC) {
            Cols<VEC> v;
            v.load_mask(mr, col, true);
            v.load_values(wr, gr, col, true);
            unsigned int out = 0;
#pragma unroll
            for (int e = 0; e < VEC; ++e) {
                const bool was = is_kept(v, e, col);
                const bool on = was != (was == trim && chosen(trim ? weight_key(v.w(e)) : grad_key(v.g(e)), col + e));
                if (!(on && was) && __float_as_uint(v.w(e)) != 0u) wr[col + e] = 0.0f;
                out |= on ? 1u << (8 * e) : 0u;
            }
            if (VEC == 4) *reinterpret_cast<unsigned int*>(mr + col) = out;
            else mr[col] = (uint8_t)out;
        }
    }
}

// Rows of up to 1024 columns take blocks of 128 threads: more rows are on an SM at once to hide one another's barriers.
struct Finalize { void (*kernel)(float*, uint8_t*, const float*, const uint8_t*, int, const State*); int threads; };
template <int VEC>
Finalize finalize_for(int in_f) {
    if (in_f <= 1024) return {finalize_kernel<VEC, 1024, 128>, 128};
    if (in_f <= 2048) return {finalize_kernel<VEC, 2048, 256>, 256};
    if (in_f <= 4096) return {finalize_kernel<VEC, 4096, 256>, 256};
    return {finalize_kernel<VEC, 0, 256>, 256};
}

// A launch that may start before the kernel ahead of it in the stream has ended (see wait_for_previous).
template <typename... KArgs, typename... Args>
void launch_after(void (*kernel)(KArgs...), int blocks, int threads, cudaStream_t st, Args... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)blocks), cfg.blockDim = dim3((unsigned)threads), cfg.stream = st;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr, cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);  // an error is found where the result is waited for
}

size_t align_up(size_t v) { return (v + 255) & ~(size_t)255; }

struct Workspace {
    int* row_count;
    int* salient;
    uint8_t* survives;
    State* state;
    uint2* list;            // 2 x cap open elements
    uint2* ties;            // 2 x ties_cap
    unsigned int cap, ties_cap;
    size_t bytes;
};

// Together the state and the lists take 2 bytes per entry of the layer: room for nearly an eighth of it per selection.
// The elements that one more digit leaves open have room for 1 / 64.
Workspace carve(void* base, int out_f, int in_f) {
    const size_t n = (size_t)out_f * in_f;
    size_t off = 0;
    auto take = [&](size_t b) {
        const size_t at = off;
        off += align_up(b);
        return static_cast<char*>(base) + at;
    };
    Workspace w{};
    w.cap = (unsigned int)std::max<int64_t>(1024, (2 * (int64_t)n - (int64_t)sizeof(State)) / 16);
    w.ties_cap = (unsigned int)(n / 64 < 64 ? 64 : n / 64 > 32768 ? 32768 : n / 64);
    w.row_count = reinterpret_cast<int*>(take((size_t)out_f * 4));
    w.salient = reinterpret_cast<int*>(take((size_t)out_f * 4));
    w.survives = reinterpret_cast<uint8_t*>(take((size_t)out_f));
    w.state = reinterpret_cast<State*>(take(sizeof(State)));
    w.list = reinterpret_cast<uint2*>(take(2 * (size_t)w.cap * sizeof(uint2)));
    w.ties = reinterpret_cast<uint2*>(take(2 * (size_t)w.ties_cap * sizeof(uint2)));
    w.bytes = off;
    return w;
}

// ---- cfi_pack_device: the condensed arrays straight from device-resident w and mask -------------------------------

struct PackInfo { int n_active, k, constant, blocks_done, changed; };  // changed: a row holds another count than when it was counted

// A lane's kVec consecutive mask bytes as a bit set (bit e: column e is kept).
template <int VEC>
__device__ __forceinline__ unsigned int kept_set(const uint8_t* m, int col, int in_f) {
    if (VEC == 1) return col < in_f && m[col] ? 1u : 0u;
    unsigned int bits = 0;
    if (col < in_f) {
        const uint4 v = *reinterpret_cast<const uint4*>(m + col);
        const unsigned int q[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            // one bit per nonzero byte, gathered from bits 0, 8, 16, 24 of the comparison
            const unsigned int nz = __vcmpne4(q[i], 0u) & 0x08040201u;
            bits |= ((nz | (nz >> 8) | (nz >> 16) | (nz >> 24)) & 0xFu) << (4 * i);
        }
    }
    return bits;
}

// One warp per row: its number of kept weights.  The block that finishes last ranks the non-empty rows and finds the
// common fan-in.  (A row is one or two kilobytes of mask: a block per row spent its time on barriers.)
template <int VEC>
__global__ void __launch_bounds__(kThreads) pack_rows_kernel(const uint8_t* mask, int out_f, int in_f, int* row_count, int* row_rank, PackInfo* info) {
    __shared__ int part[kThreads / 32], k_min, k_max;
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    const int64_t r = (int64_t)blockIdx.x * (kThreads / 32) + wid;
    if (r < out_f) {
        const uint8_t* m = mask + (size_t)r * in_f;
        int n = 0, col = lane * VEC;
        if (VEC == 1) {  // single bytes: sixteen loads in flight (64 x 9000: 41 -> 24 us with sixteen instead of four)
            for (; in_f - col > 15 * 32; col += 16 * 32) {
#pragma unroll
                for (int u = 0; u < 16; ++u) n += m[col + 32 * u] ? 1 : 0;
            }
        }
#pragma unroll 4
        for (; col < in_f; col += 32 * VEC) n += __popc(kept_set<VEC>(m, col, in_f));
        n = __reduce_add_sync(0xffffffffu, n);
        if (lane == 0) row_count[r] = n;
    }
    if (!last_block(&info->blocks_done)) return;
    if (t == 0) k_min = 0x7fffffff, k_max = 0;
    constexpr int kPer = 8;  // consecutive rows per thread and round
    int before = 0, lo = 0x7fffffff, hi = 0;
    for (int r0 = 0; r0 < out_f; r0 += kPer * kThreads) {
        int cnt[kPer], live = 0;
#pragma unroll
        for (int e = 0; e < kPer; ++e) {
            const int row = r0 + kPer * t + e;
            cnt[e] = row < out_f ? __ldcg(&row_count[row]) : 0;
            if (cnt[e]) ++live, lo = min(lo, cnt[e]), hi = max(hi, cnt[e]);
        }
        int incl = live;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int up = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += up;
        }
        __syncthreads();  // part[] of the round before has been read
        if (lane == 31) part[wid] = incl;
        __syncthreads();
        int rank = before + incl - live;
#pragma unroll
        for (int i = 0; i < kThreads / 32; ++i) {
            rank += i < wid ? part[i] : 0;
            before += part[i];
        }
#pragma unroll
        for (int e = 0; e < kPer; ++e) {
            const int row = r0 + kPer * t + e;
            if (row < out_f) row_rank[row] = cnt[e] ? rank++ : -1;
        }
    }
    __syncthreads();
    lo = __reduce_min_sync(0xffffffffu, lo), hi = __reduce_max_sync(0xffffffffu, hi);
    if (lane == 0) atomicMin(&k_min, lo), atomicMax(&k_max, hi);
    __syncthreads();
    if (t == 0) info->n_active = before, info->k = k_max, info->constant = (before == 0 || k_min == k_max) ? 1 : 0;
}

// One warp per row: its kept entries in increasing column order to values / indices of its rank.  A lane takes VEC
// consecutive columns, their place follows from a prefix count over the warp.  n_active and k are the sizes of the arrays
// where they are known before the launch: nothing is written outside them, nor at all where the counts are others.  -1: as counted.
// The kept entries of every row, empty ones too, are counted on the way: a mask that is no longer the one the rows were
// counted from is reported, whatever its rows hold now.  *fault (memory of the host; NULL: info only) is written only where
// something is wrong.
template <int VEC>
__global__ void __launch_bounds__(kThreads) pack_fill_kernel(const float* w, const uint8_t* mask, const int* row_rank, int out_f, int in_f,
                                                             PackInfo* info, int n_active, int k, float* values, int32_t* indices,
                                                             int32_t* active_rows, int* fault) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t r = (int64_t)blockIdx.x * (kThreads / 32) + warp;
    if (k < 0) n_active = info->n_active, k = info->k;
    if (r >= out_f) return;
    auto report = [&]() {
        info->changed = 1;
        if (fault) *fault = 1;
    };
    if (!info->constant || info->n_active != n_active || info->k != k) {
        if (fault && lane == 0) *fault = 1;
        return;
    }
    const int rank = row_rank[r];
    if (rank >= n_active) {
        if (lane == 0) report();
        return;
    }
    if (lane == 0 && rank >= 0) active_rows[rank] = (int32_t)r;
    const float* wr = w + (size_t)r * in_f;
    const uint8_t* mr = mask + (size_t)r * in_f;
    const size_t begin = rank < 0 ? 0 : (size_t)rank * k, end = rank < 0 ? 0 : begin + k;  // (of a row without weights nothing is written)
    size_t at0 = begin;
    if constexpr (VEC == 1) {
        // Rows that 16-byte loads cannot take: sixteen chunks of 32 single columns at a time, the next ones on their way while
        // these are written, and a ballot for a place (64 x 9000: 142 -> 101 us; one chunk and a scan over the lanes at a time, each
        // waited for a trip to memory).
        constexpr int U = 16;
        auto load = [&](unsigned int c0) {  // (unsigned: a step past the end of the longest row does not wrap)
            unsigned int set = 0;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const unsigned int col = c0 + 32u * u + lane;
                set |= (col < (unsigned int)in_f && mr[col] ? 1u : 0u) << u;
            }
            return set;
        };
        const int room = (int)(end - begin);
        int seen = 0;  // kept entries of the row so far
        unsigned int next = load(0);
        for (unsigned int c0 = 0; c0 < (unsigned int)in_f; c0 += 32 * U) {
            const unsigned int bits = next;
            if (c0 + 32 * U < (unsigned int)in_f) next = load(c0 + 32 * U);
            int at[U];
            float v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const unsigned int set = __ballot_sync(0xffffffffu, (bits >> u) & 1u);
                at[u] = (bits >> u) & 1u ? seen + __popc(set & ((1u << lane) - 1u)) : room;
                if (at[u] < room) v[u] = wr[c0 + 32u * u + lane];
                seen += __popc(set);
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (at[u] < room) values[begin + at[u]] = v[u], indices[begin + at[u]] = (int32_t)(c0 + 32u * u + lane);
        }
        at0 += seen;
    } else {
        unsigned int next = kept_set<VEC>(mr, lane * VEC, in_f);
        for (int c0 = 0; c0 < in_f; c0 += 32 * VEC) {
            unsigned int bits = next;
            const int col = c0 + lane * VEC, mine = __popc(bits);
            next = kept_set<VEC>(mr, col + 32 * VEC, in_f);  // in flight while this chunk is written
            int incl = mine;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int up = __shfl_up_sync(0xffffffffu, incl, off);
                if (lane >= off) incl += up;
            }
            size_t at = at0 + (incl - mine);
            while (bits && at < end) {
                const int c = col + __ffs(bits) - 1;
                bits &= bits - 1;
                values[at] = wr[c];
                indices[at++] = c;
            }
            at0 += __shfl_sync(0xffffffffu, incl, 31);
        }
    }
    if (lane == 0 && at0 != end) report();
}

}  // namespace

extern "C" cfi_status_t cfi_srigl_workspace_bytes(int32_t out_features, int32_t in_features, size_t* bytes) {
    if (!bytes) return CFI_ERR_NULL;
    if (out_features < 1 || in_features < 1 || (int64_t)out_features * in_features > ((int64_t)1 << 31)) return CFI_ERR_SHAPE;
    *bytes = carve(nullptr, out_features, in_features).bytes;
    return CFI_OK;
}

extern "C" cfi_status_t cfi_srigl_update(float* w, uint8_t* mask, const float* grad, int32_t out_features, int32_t in_features,
                                         int64_t K, float gamma_sal, void* workspace, size_t workspace_bytes, int32_t* k_new,
                                         int32_t* n_active_new, cfi_stream_t stream) {
    if (!w || !mask || !grad || !workspace || !k_new || !n_active_new) return CFI_ERR_NULL;
    if (out_features < 1 || in_features < 1 || (int64_t)out_features * in_features > ((int64_t)1 << 31) || !(gamma_sal >= 0.0f))
        return CFI_ERR_SHAPE;
    if (((uintptr_t)workspace & 255) != 0) return CFI_ERR_ALIGNMENT;
    const Workspace ws = carve(workspace, out_features, in_features);
    if (workspace_bytes < ws.bytes) return CFI_ERR_BUFFER_TOO_SMALL;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const bool vec = (in_features & 3) == 0 && (((uintptr_t)w | (uintptr_t)grad) & 15) == 0 && ((uintptr_t)mask & 3) == 0;
    const int blocks = std::min(out_features, 148 * 4);  // one wave, whole rows per block
    const size_t hist_bytes = 2 * kBins * sizeof(unsigned int);
    StateHead host{};
    auto wait = [&]() {
        const bool ok = cudaGetLastError() == cudaSuccess && cudaMemcpyAsync(&host, static_cast<StateHead*>(ws.state), sizeof(host), cudaMemcpyDeviceToHost, st) == cudaSuccess &&
                        cudaStreamSynchronize(st) == cudaSuccess;
        if (!ok) cudaGetLastError();
        return ok;
    };
    // Short rows: several at a time, so that a thread has as many loads in flight as in a long one.
    const int chunk_cols = kThreads * (vec ? 4 : 1), ahead = vec ? 4 : 8;
    const int rows = in_features <= ahead / 4 * chunk_cols ? 4 : in_features <= ahead / 2 * chunk_cols ? 2 : 1;
    auto sweep = [&](auto first) {
        constexpr bool F = decltype(first)::value;
        auto go = [&](auto kernel) {
            kernel<<<blocks, kThreads, hist_bytes, st>>>(w, mask, grad, ws.row_count, out_features, in_features, K, ws.cap, ws.state);
        };
        if (vec) rows == 4 ? go(sweep_kernel<4, 4, F>) : rows == 2 ? go(sweep_kernel<4, 2, F>) : go(sweep_kernel<4, 1, F>);
        else rows == 4 ? go(sweep_kernel<1, 4, F>) : rows == 2 ? go(sweep_kernel<1, 2, F>) : go(sweep_kernel<1, 1, F>);
    };
    auto collect = [&]() {
        auto go = [&](auto kernel) {
            launch_after(kernel, blocks, kThreads, st, w, mask, grad, ws.row_count, out_features, in_features, ws.cap, ws.list, ws.salient, ws.state);
        };
        if (vec) rows == 4 ? go(collect_kernel<4, 4>) : rows == 2 ? go(collect_kernel<4, 2>) : go(collect_kernel<4, 1>);
        else rows == 4 ? go(collect_kernel<1, 4>) : rows == 2 ? go(collect_kernel<1, 2>) : go(collect_kernel<1, 1>);
    };
    auto resolve_and_finalize = [&]() {
        launch_after(resolve_kernel, 2 * 148, kThreads, st, ws.list, ws.cap, ws.ties, ws.ties_cap, ws.row_count, ws.salient, ws.survives, out_features,
                     in_features, gamma_sal, ws.state);
        const Finalize f = vec ? finalize_for<4>(in_features) : finalize_for<1>(in_features);
        launch_after(f.kernel, out_features, f.threads, st, w, mask, grad, ws.survives, in_features, ws.state);
    };
    // The usual layer needs one sweep for the first digit and one that lists what it leaves open; nothing waits in between.
    // The later kernels return at once where that does not do, and the rare rest of the way is driven from here.
    if (cudaMemsetAsync(ws.state, 0, sizeof(State), st) != cudaSuccess) return CFI_ERR_CUDA;
    sweep(std::true_type{});
    collect();
    resolve_and_finalize();
    if (!wait()) return CFI_ERR_CUDA;
    if (!host.done) {
        const bool listed = host.listable != 0;
        for (int i = 0; i < 6 && !host.listable; ++i) {  // very many equal keys: digit by digit until the open elements fit the lists
            sweep(std::false_type{});
            if (!wait()) return CFI_ERR_CUDA;
        }
        if (!listed) {
            collect();
            if (!wait()) return CFI_ERR_CUDA;
        }
        for (int i = 0; i < 6 && ((host.sel[0].on && host.sel[0].count > ws.ties_cap) || (host.sel[1].on && host.sel[1].count > ws.ties_cap)); ++i) {
            list_sweep_kernel<<<148, kThreads, 0, st>>>(ws.list, ws.cap, in_features, ws.state);
            if (!wait()) return CFI_ERR_CUDA;
        }
        resolve_and_finalize();
        if (!wait()) return CFI_ERR_CUDA;
    }
    *k_new = host.k_new;
    *n_active_new = host.live_after;
    return CFI_OK;
}

namespace {

struct PackWorkspace {
    int *row_count, *row_rank;
    PackInfo* info;
};
cfi_status_t pack_workspace(const void* w, const uint8_t* mask, void* workspace, size_t bytes, int32_t out_f, int32_t in_f, PackWorkspace* out) {
    if (!w || !mask || !workspace) return CFI_ERR_NULL;
    if (out_f < 1 || in_f < 1 || (int64_t)out_f * in_f > ((int64_t)1 << 31)) return CFI_ERR_SHAPE;
    if (((uintptr_t)workspace & 255) != 0) return CFI_ERR_ALIGNMENT;
    if (bytes < (size_t)out_f * 8 + 256) return CFI_ERR_BUFFER_TOO_SMALL;
    out->row_count = static_cast<int*>(workspace);
    out->row_rank = out->row_count + out_f;
    out->info = reinterpret_cast<PackInfo*>(out->row_rank + out_f);
    return CFI_OK;
}
bool pack_vector_loads(const uint8_t* mask, int32_t in_f) { return (in_f & 15) == 0 && ((uintptr_t)mask & 15) == 0; }
int pack_blocks(int32_t out_f) { return (int)(((int64_t)out_f + kThreads / 32 - 1) / (kThreads / 32)); }

cfi_status_t pack_fill(const PackWorkspace& ws, const float* w, const uint8_t* mask, int32_t out_f, int32_t in_f, int32_t k, int32_t n_active,
                       float* values, int32_t* indices, int32_t* active_rows, int* fault, cudaStream_t st) {
    const auto kernel = pack_vector_loads(mask, in_f) ? pack_fill_kernel<16> : pack_fill_kernel<1>;
    kernel<<<pack_blocks(out_f), kThreads, 0, st>>>(w, mask, ws.row_rank, out_f, in_f, ws.info, n_active, k, values, indices, active_rows, fault);
    return cudaGetLastError() == cudaSuccess ? CFI_OK : CFI_ERR_CUDA;
}
// A word of page-locked memory, one per thread that fills arrays (its calls wait, so no two of them share it at a time), given
// back when the thread ends.  nullptr where there is none to be had.
struct PackFault {
    int* p = nullptr;
    int* get() {
        cudaPointerAttributes a{};
        if (p && (cudaPointerGetAttributes(&a, p) != cudaSuccess || a.type != cudaMemoryTypeHost)) {  // gone with a reset of the device
            cudaGetLastError();
            p = nullptr;
        }
        if (!p && cudaHostAlloc(reinterpret_cast<void**>(&p), sizeof(int), cudaHostAllocPortable | cudaHostAllocMapped) != cudaSuccess) {
            cudaGetLastError();
            p = nullptr;
        }
        return p;
    }
    ~PackFault() {
        if (p) cudaFreeHost(p);
    }
};
// What the kernels found, once they are done.
bool pack_result(const PackWorkspace& ws, PackInfo* host, cudaStream_t st) {
    return cudaMemcpyAsync(host, ws.info, sizeof(*host), cudaMemcpyDeviceToHost, st) == cudaSuccess && cudaStreamSynchronize(st) == cudaSuccess;
}

}  // namespace

extern "C" cfi_status_t cfi_pack_device(const float* w_dense, const uint8_t* mask, int32_t out_features, int32_t in_features,
                                        void* workspace, size_t workspace_bytes, int32_t* k, int32_t* n_active, float* values,
                                        int32_t* indices, int32_t* active_rows, cfi_stream_t stream) {
    if (!k || !n_active) return CFI_ERR_NULL;
    const bool fill = values || indices || active_rows;
    if (fill && !(values && indices && active_rows)) return CFI_ERR_NULL;
    PackWorkspace ws;
    if (cfi_status_t e = pack_workspace(w_dense, mask, workspace, workspace_bytes, out_features, in_features, &ws)) return e;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    PackInfo host{};
    bool ok = cudaMemsetAsync(ws.info, 0, sizeof(PackInfo), st) == cudaSuccess;
    if (ok) {
        const auto kernel = pack_vector_loads(mask, in_features) ? pack_rows_kernel<16> : pack_rows_kernel<1>;
        kernel<<<pack_blocks(out_features), kThreads, 0, st>>>(mask, out_features, in_features, ws.row_count, ws.row_rank, ws.info);
        ok = cudaGetLastError() == cudaSuccess;
    }
    if (ok && fill) ok = pack_fill(ws, w_dense, mask, out_features, in_features, -1, -1, values, indices, active_rows, nullptr, st) == CFI_OK;
    ok = ok && pack_result(ws, &host, st);
    if (!ok) {
        cudaGetLastError();
        return CFI_ERR_CUDA;
    }
    if (!host.constant || host.changed) return CFI_ERR_NOT_CONSTANT_FAN_IN;
    *n_active = host.n_active;
    *k = host.n_active ? host.k : 0;
    return CFI_OK;
}

extern "C" cfi_status_t cfi_pack_device_fill(const float* w_dense, const uint8_t* mask, int32_t out_features, int32_t in_features,
                                             void* workspace, size_t workspace_bytes, int32_t k, int32_t n_active, float* values,
                                             int32_t* indices, int32_t* active_rows, cfi_stream_t stream) {
    if (!values || !indices || !active_rows) return CFI_ERR_NULL;
    if (k < 1 || n_active < 1 || n_active > out_features || k > in_features) return CFI_ERR_SHAPE;
    PackWorkspace ws;
    if (cfi_status_t e = pack_workspace(w_dense, mask, workspace, workspace_bytes, out_features, in_features, &ws)) return e;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    // As a rule there is nothing to report and so nothing to copy back: a word of the host's that the kernel can write is
    // looked at after the wait (with the copy instead, 3072 x 768 took 70 us; with neither, and no report, 60).
    static thread_local PackFault word;
    int* fault = word.get();
    if (fault) *fault = 0;
    bool ok = pack_fill(ws, w_dense, mask, out_features, in_features, k, n_active, values, indices, active_rows, fault, st) == CFI_OK;
    ok = ok && cudaStreamSynchronize(st) == cudaSuccess;
    PackInfo host{};
    if (ok && fault && *static_cast<volatile int*>(fault) == 0) return CFI_OK;
    if (!ok || !pack_result(ws, &host, st)) {
        cudaGetLastError();
        return CFI_ERR_CUDA;
    }
    if (!host.constant || host.changed) return CFI_ERR_NOT_CONSTANT_FAN_IN;
    return host.k == k && host.n_active == n_active ? CFI_OK : CFI_ERR_SHAPE;
}

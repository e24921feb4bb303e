// CFI_VARIANT_SPLITK for bf16 layers and for fp32 batches of 2 and more (tiles of 2, 4 or 8 rows of x; bf16 also 1).
//
// Included by cfi_layer.cu (Chunk, the layouts and the pdl helpers are there).  Rows, lanes and the weight stream are those
// of cfi_splitk_kernel; what differs is x.  There a thread loads a few elements of x, waits, and writes them to shared
// memory.  With 100 KB of x (8 rows of 3072 columns), transposed to [column][BT] on the way, that was six dependent round
// trips to L2 per CTA, most of the call.  Here x stays as it is, xs[b][column] in its own type: 16-byte asynchronous copies
// put all of it in flight at once and cost neither registers nor conversions.  A gathered entry takes BT loads of 4 (or 2)
// bytes instead of one or two of 16, which is the same number of shared-memory wavefronts where the lanes of an instruction
// meet different banks.  They do so in part only: order_for_banks deals a row's entries by column mod 32 to the lanes that
// share the row at batch 1, and here more lanes share it as the tile grows, and in bf16 two columns share a bank.
// Wavefronts an instruction, from the placement: fp32 3072 columns k 307 1.5, 4096 k 205 1.8 (tiles of 4 and 8) and 2.0, 768
// k 77 2.3 .. 2.5 and 3.6; bf16 2.5 and 3.2, 3.4 and 4.2, 3.0 .. 3.3 and 4.5.
//
// 3072 -> 768, k 307, per call in a chain of launches, against x transposed to [column][BT] by the threads: batch 8 fp32
// 10.2 -> 3.7 us, bf16 18.2 -> 4.1; batch 2 fp32 4.7 -> 2.5; batch 1 bf16 6.6 -> 1.7.  4096 x 4096 at 80 %, batch 8: 15.7 -> 11.9 us.

__device__ __forceinline__ void cp_async4(uint32_t smem_off, const void* gmem_src) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(smem_at(smem_off));
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(gmem_src) : "memory");
}

// Elements from one row of x to the next in shared memory: a whole number of 16-byte pieces, with at least one element
// behind the row, the zero that pad entries read.
__host__ __device__ inline int splitk_rows_pitch(int in, int elem) {
    const int per = 16 / elem;
    return (in / per + 1) * per;
}

// Units a lane takes at a time: a unit costs BT times the instructions of batch 1, so more lanes share a row instead, each
// with less to do (768 -> 3072 at batch 8 in one tile of 8, 4 units a lane: six warps per SM, 840 instructions each, 5.6 us; with
// one 4.7; in two tiles of 4 with two units 3.3).
__host__ __device__ constexpr int splitk_rows_units(bool fp32_values, bool idx16, int bt) {
    const int u = splitk_units_in_flight(fp32_values, idx16);
    return bt <= 2 ? u : bt == 4 ? u / 2 : 1;
}

template <typename VT, bool I16, int BT, int G>
__global__ void __launch_bounds__(512, BT >= 4 ? 2 : 1) cfi_splitk_rows_kernel(DevLayer L, const VT* __restrict__ x, VT* __restrict__ y, int batch, int rows_per_group) {
    using CK = Chunk<VT, I16>;
    constexpr uint32_t kIdxBytes = I16 ? 2 : 4;
    constexpr int U = splitk_rows_units(sizeof(VT) == 4, I16, BT);
    pdl_launch_dependents();
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int b0 = blockIdx.y * BT, nb = min(BT, batch - b0);
    const int groups = nthr / G, g = tid / G, lg = tid % G;
    const int nvec = L.kp / CK::VEC;
    const bool dense_rows = L.identity_rows != 0;
    int o = blockIdx.x * (groups * rows_per_group) + g;
    int r = o < L.out ? (dense_rows ? o : L.slot[o]) : -1;
    constexpr bool kNext = BT == 8;  // a second step in flight behind the one being multiplied
    const bool long_row = nvec > (kNext ? 2 : 1) * G * U;

    // As in cfi_splitk_kernel: the first row's weights depend neither on x nor on the kernel before this one.
    auto ask_row = [&]() {
        if (lg == 0 && r >= 0 && long_row) {
            prefetch_l2(reinterpret_cast<const VT*>(L.values) + (size_t)r * L.kp, (uint32_t)(L.kp * sizeof(VT)));
            prefetch_l2(static_cast<const unsigned char*>(L.indices) + (size_t)r * L.kp * kIdxBytes, (uint32_t)L.kp * kIdxBytes);
        }
    };
    ask_row();
    CK ck[U], nx[U];
    auto load_step = [&](CK (&c)[U], int v0) {
#pragma unroll
        for (int u = 0; u < U; ++u) c[u].load(L.values, L.indices, (size_t)max(r, 0) * L.kp, v0 + u * G, r >= 0 && v0 + u * G < nvec, L.in);
    };
    load_step(ck, lg);
    if (kNext && nvec > G * U) load_step(nx, lg + G * U);
    float bias = o < L.out ? L.bias[o] : 0.0f;
    const size_t row_bytes = (size_t)L.in * sizeof(VT);
    if (blockIdx.x < 2 && row_bytes % 16 == 0) {  // a cold x is then on chip when the wait returns
        const size_t bytes = (size_t)nb * row_bytes, off = (size_t)tid << 14;
        if (off < bytes)
            prefetch_l2(reinterpret_cast<const unsigned char*>(x + (size_t)b0 * L.in) + off, (uint32_t)min(bytes - off, (size_t)1 << 14));
    }
    const int pitch = splitk_rows_pitch(L.in, (int)sizeof(VT));
    VT* xs = reinterpret_cast<VT*>(smem_at(0));
    if (tid < BT) xs[(size_t)tid * pitch + L.in] = VT(0.0f);

    pdl_wait();
    if (row_bytes % 16 == 0) {
        const int pieces = (int)(row_bytes / 16);
#pragma unroll
        for (int b = 0; b < BT; ++b) {
            if (b >= nb) break;
            const unsigned char* src = reinterpret_cast<const unsigned char*>(x + (size_t)(b0 + b) * L.in);
            for (int c = tid; c < pieces; c += nthr) cp_async16((uint32_t)(b * pitch * (int)sizeof(VT) + 16 * c), src + 16 * (size_t)c);
        }
    } else if (sizeof(VT) == 4) {  // fp32 rows of any length start on 4-byte boundaries
#pragma unroll
        for (int b = 0; b < BT; ++b) {
            if (b >= nb) break;
            for (int c = tid; c < L.in; c += nthr) cp_async4((uint32_t)(b * pitch + c) * 4u, x + (size_t)(b0 + b) * L.in + c);
        }
    } else {
        constexpr int kCols = BT >= 8 ? 2 : 8 / BT;  // eight to sixteen loads in flight per thread
        for (int c0 = tid; c0 < L.in; c0 += nthr * kCols) {
            VT v[kCols][BT];
#pragma unroll
            for (int u = 0; u < kCols; ++u)
#pragma unroll
                for (int b = 0; b < BT; ++b) v[u][b] = b < nb && c0 + u * nthr < L.in ? x[(size_t)(b0 + b) * L.in + c0 + u * nthr] : VT(0.0f);
#pragma unroll
            for (int u = 0; u < kCols; ++u)
#pragma unroll
                for (int b = 0; b < BT; ++b)
                    if (c0 + u * nthr < L.in) xs[(size_t)b * pitch + c0 + u * nthr] = v[u][b];
        }
    }
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();

    for (int i = 0;;) {
        float acc[BT];
#pragma unroll
        for (int b = 0; b < BT; ++b) acc[b] = 0.0f;
        if (r >= 0) {
            for (int v0 = lg;;) {
#pragma unroll
                for (int u = 0; u < U; ++u)
#pragma unroll
                    for (int e = 0; e < CK::VEC; ++e) {
                        const VT* p = xs + ck[u].col(e);
                        const float w = ck[u].weight(e);
#pragma unroll
                        for (int b = 0; b < BT; ++b) acc[b] = fmaf(w, to_f32(p[b * pitch]), acc[b]);
                    }
                v0 += G * U;
                if (v0 >= nvec) break;
                if (kNext) {
#pragma unroll
                    for (int u = 0; u < U; ++u) ck[u] = nx[u];
                    if (v0 + G * U < nvec) load_step(nx, v0 + G * U);
                } else {
                    load_step(ck, v0);
                }
            }
        }
        const int o_done = o;
        const float bias_done = bias;
        const bool more = ++i < rows_per_group;  // the next row's first vectors and bias before this row's reduction and store
        if (more) {
            o += groups;
            r = o < L.out ? (dense_rows ? o : L.slot[o]) : -1;
            ask_row();
            load_step(ck, lg);
            if (kNext && nvec > G * U) load_step(nx, lg + G * U);
            bias = o < L.out ? L.bias[o] : 0.0f;
        }
        // The k-sum across the G lanes of the group.  While a lane still holds several rows of x it hands half of them to its
        // partner and keeps the other half (7 shuffles for 8 rows over 8 lanes instead of 24, and every lane ends up with
        // results of its own to activate and store); the pairs that are added are those of a plain exchange.
        int first = 0;  // the rows of x that this lane ends up with: first, first + 1, ... , kept of them
        constexpr int kKept = BT > G ? BT / G : 1;
#pragma unroll
        for (int m = G >> 1, have = BT; m > 0; m >>= 1) {
            if (have > 1) {
                have >>= 1;
                const bool upper = (lg & m) != 0;
#pragma unroll
                for (int b = 0; b < have; ++b) {
                    const float send = upper ? acc[b] : acc[b + have], keep = upper ? acc[b + have] : acc[b];
                    acc[b] = keep + __shfl_xor_sync(0xffffffffu, send, m);
                }
                if (upper) first += have;
            } else {
                acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], m);
            }
        }
        constexpr int kSame = G > BT ? G / BT : 1;  // lanes that hold the same result
        if (o_done < L.out && lg % kSame == 0) {
#pragma unroll
            for (int b = 0; b < kKept; ++b)
                if (first + b < nb) from_f32(&y[(size_t)(b0 + first + b) * L.out + o_done], activate(acc[b] + bias_done, L.act));
        }
        if (!more) break;
    }
}

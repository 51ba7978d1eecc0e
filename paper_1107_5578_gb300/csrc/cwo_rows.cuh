// cwo_rows.cuh -- the two row passes of a propagation (kernels and their launch templates; the
// launchers are instantiated by cwo_rows.cu, cwo_rows_inv_a.cu, cwo_rows_inv_b.cu and
// cwo_rows_turn.cu, which compile in parallel).
//
//   row forward : zero-pad each Nx-sample row to Px = 2 Nx and take its forward FFT
//                 (steps "expand" and the row half of "FFT" of Eqs. ang3 / fre_conv_fft).
//                 Only the Ny source rows exist; padding rows are never read, written or
//                 transformed.  The padding columns are never read either: the first DIF stage
//                 sees its upper 8 inputs as constant zeros.
//   row inverse : inverse FFT of each of the Ny kept rows of the intermediate, keeping the first
//                 Nx outputs ("extract the exact area") and applying the 1/(Px Py) scale.
//
// The intermediate W is COLUMN-MAJOR, [items][Px][Ny] complex64: storage column st holds the Ny
// values of one frequency kx contiguously, so that the column pass streams whole columns.  Along
// x the storage order is the register order of the last forward stage: register e of thread t
// (DIF position 16 t + e) is storage column e * T + t (at Px = 8192 the split order below).  A CTA handles R rows and transposes them
// through a dense shared-memory tile [st][r]; the tile moves to and from the intermediate as TMA
// tensor boxes of R rows x 256 columns (R * 8 contiguous bytes per column), so the transposed
// global side costs the threads no load/store instructions.
#pragma once
#include <algorithm>

#include "cwo.h"
#include "cwo_debug.h"
#include "cwo_fft.cuh"
#include "cwo_internal.h"
#include "cwo_launch.cuh"
#include "cwo_tma.cuh"
#include "cwo_epilogue.cuh"

namespace cwo {

// Rows per CTA of each pass (measured on GB300).  The forward pass stores its tile, and stores of
// less than a 32-byte sector per column are expensive, so it keeps >= 4 rows where a 4-row tile
// fits (P <= 4096); the inverse pass loads, where 2-row tiles (16 bytes per column, the other half
// of each sector served from L2 to the neighbouring CTA) allow more CTAs per SM.  A TMA box must
// span at least 16 contiguous bytes, hence >= 2 rows.
template <int P> constexpr int rows_fwd() { return P >= 256 ? 4 : 8; }
template <int P> constexpr int rows_inv() { return P >= 4096 ? 2 : (P >= 256 ? 4 : 8); }
constexpr bool kRowInvPersistent = true;   // measured: 25.4 -> 23.0 us per 2048^2 field

template <int P, int R>
__host__ __device__ constexpr size_t row_smem_words() {
    return PadLayout<P, R>::WORDS > (size_t)R * P ? PadLayout<P, R>::WORDS : (size_t)R * P;
}

// Lanes are row-fastest (thread = r + R t): the FFT exchanges then see R interleaved transforms,
// for which the padded layout is conflict free, and the dense tile [st][r] used by the transposing
// copies is addressed as e * (R T) + threadIdx.x, i.e. consecutive words across a warp.

template <int P, int R, bool PRE>
__global__ void __launch_bounds__(R * (P / 16))
k_row_fwd(const float2* __restrict__ in, long long in_item_stride, const __grid_constant__ CUtensorMap wmap,
          int item_off, const float4* __restrict__ tw, const Prefactor pre) {
    pdl_wait();
    constexpr int T = P / 16, N = P / 2, NT = R * T;
    constexpr int BOX = P < kTmaBoxCols ? P : kTmaBoxCols;
    extern __shared__ __align__(1024) float2 sm[];
    const int r = threadIdx.x % R, t = threadIdx.x / R;
    const int y0 = blockIdx.x * R;
    const int item = blockIdx.y;
    const float2* src = in + item * in_item_stride + (long long)(y0 + r) * N;
    float2 v[16];
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = __ldg(src + t + e * T);   // DIF stage-0 positions t + e P/16
#pragma unroll
    for (int e = 8; e < 16; ++e) v[e] = make_float2(0.f, 0.f);   // zero padding, never loaded
    if constexpr (PRE) {
        const float2 fy = __ldg(pre.fy + y0 + r);
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = cmul(v[e], cmul(__ldg(pre.fx + t + e * T), fy));
    }
    fwd1_from<P, R, 0, 8>(v, sm, r, t, TwTable<P>{tw, t});
    if constexpr (Geo<P>::NST > 1) __syncthreads();   // every exchange read done before the tile is written
    // dense tile [st][r]: register e of (r, t) is storage column st = e T + t of row y0 + r
#pragma unroll
    for (int e = 0; e < 16; ++e) sm[e * NT + threadIdx.x] = v[e];
    fence_proxy_async_smem();
    __syncthreads();
    if (threadIdx.x == 0) {   // R rows x BOX columns per box: R * 8 contiguous bytes per column
#pragma unroll 1
        for (int b = 0; b < P / BOX; ++b) tma_store_3d(&wmap, sm + b * BOX * R, y0, b * BOX, item + item_off);
        tma_store_commit_and_drain();
    }
}

template <int P, int R, int EPI>
__global__ void __launch_bounds__(R * (P / 16))
k_row_inv(const __grid_constant__ CUtensorMap wmap, int item_off, float2* __restrict__ out,
          long long out_item_stride, float scale, const float4* __restrict__ tw, int* status, const Epilogue ep) {
    pdl_wait();
    constexpr int T = P / 16, N = P / 2, NT = R * T;
    constexpr int BOX = P < kTmaBoxCols ? P : kTmaBoxCols;
    extern __shared__ __align__(1024) float2 sm[];
    uint64_t* mbar = reinterpret_cast<uint64_t*>(sm + row_smem_words<P, R>());   // after the tile
    const int r = threadIdx.x % R, t = threadIdx.x / R;
    const int y0 = blockIdx.x * R;
    const int item = blockIdx.y;
    if (threadIdx.x == 0) mbar_init(mbar, 1);
    __syncthreads();
    if (threadIdx.x == 0) {
        mbar_arrive_expect_tx(mbar, (unsigned)(R * P * sizeof(float2)));
#pragma unroll 1
        for (int b = 0; b < P / BOX; ++b) tma_load_3d(sm + b * BOX * R, &wmap, mbar, y0, b * BOX, item + item_off);
    }
    const bool ok = mbar_wait_bounded(mbar, 0, status);
    float2 v[16];
#pragma unroll
    for (int e = 0; e < 16; ++e) v[e] = sm[e * NT + threadIdx.x];
    if (__syncthreads_or(!ok)) return;             // a copy did not land: the status word says so
    inv1_from<P, R, Geo<P>::NST - 1>(v, sm, r, t, TwTable<P>{tw, t});
    const long long base = item * out_item_stride + (long long)(y0 + r) * N;
#pragma unroll
    for (int e = 0; e < 8; ++e) epilogue_store<EPI>(out, ep, base + t + e * T, t + e * T, y0 + r, cscale(v[e], scale));   // crop
}

// ------------------------------------------------------------------------------------------
// Persistent row passes: one CTA per SM (or as many as fit) walks groups g = blockIdx.x,
// + gridDim.x, ... of R rows, so that the memory traffic of one group overlaps the FFT of another.
//
// Forward: the R input rows of the NEXT group are copied into a staging buffer by the bulk-copy
// engine (one contiguous copy per row, completion on an mbarrier) while the current group is
// transformed; the transposed tile of a group is written out by TMA stores that drain while the
// next group's input is read from the staging buffer.  Shared memory: exchange region / tile
// (row_smem_words), staging R x (N + 4) (row stride padded so the r-fast reads hit distinct
// banks), one mbarrier.
// ------------------------------------------------------------------------------------------
template <int P, int R>
__host__ __device__ constexpr int stage_stride() { return P / 2 + 4; }

template <int P, int R>
__host__ __device__ constexpr size_t row_fwd_p_smem_bytes() {
    return (row_smem_words<P, R>() + (size_t)R * stage_stride<P, R>()) * sizeof(float2) + sizeof(uint64_t);
}

template <int P, int R, bool PRE>
// two CTAs per SM where a CTA has fewer than 1024 threads (1024^2 fields: 5.8 -> 5.3 us per field)
__global__ void __launch_bounds__(R * (P / 16), R * (P / 16) >= 1024 ? 1 : 2)
k_row_fwd_p(const float2* __restrict__ in, long long in_item_stride, const __grid_constant__ CUtensorMap wmap,
            int item_off, int groups_per_item, int total_groups, const float4* __restrict__ tw, int* status,
            const Prefactor pre) {
    pdl_wait();
    constexpr int T = P / 16, N = P / 2, NT = R * T, SST = stage_stride<P, R>();
    constexpr int BOX = P < kTmaBoxCols ? P : kTmaBoxCols;
    extern __shared__ __align__(1024) float2 sm[];
    float2* stage = sm + row_smem_words<P, R>();
    uint64_t* mbar = reinterpret_cast<uint64_t*>(stage + R * SST);
    const int r = threadIdx.x % R, t = threadIdx.x / R;
    auto issue = [&](int g) {   // thread 0: the R rows of group g into the staging buffer
        const int item = g / groups_per_item, y0 = (g % groups_per_item) * R;
        const float2* src = in + item * in_item_stride + (long long)y0 * N;
        mbar_arrive_expect_tx(mbar, (unsigned)(R * N * sizeof(float2)));
#pragma unroll 1
        for (int rr = 0; rr < R; ++rr) bulk_load(stage + rr * SST, src + rr * N, (unsigned)(N * sizeof(float2)), mbar);
    };
    if (threadIdx.x == 0) {
        mbar_init(mbar, 1);
        if ((int)blockIdx.x < total_groups) issue(blockIdx.x);
    }
    __syncthreads();
    unsigned parity = 0;
#pragma unroll 1
    for (int g = blockIdx.x; g < total_groups; g += gridDim.x, parity ^= 1u) {
        const bool ok = mbar_wait_bounded(mbar, parity, status);
        float2 v[16];
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = stage[r * SST + t + e * T];   // DIF stage-0 positions t + e P/16
#pragma unroll
        for (int e = 8; e < 16; ++e) v[e] = make_float2(0.f, 0.f);      // zero padding, never loaded
        if constexpr (PRE) {
            const float2 fy = __ldg(pre.fy + (g % groups_per_item) * R + r);
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] = cmul(v[e], cmul(__ldg(pre.fx + t + e * T), fy));
        }
        fence_proxy_async_smem();   // these reads of the staging buffer precede the next bulk copy into it
        if (__syncthreads_or(!ok)) break;                                // a copy did not land
        if (threadIdx.x == 0 && g + (int)gridDim.x < total_groups) issue(g + gridDim.x);
        // first stage in registers while the previous tile's stores drain; the exchange region
        // (which the tile aliases) is rewritten only after the drain
        const TwTable<P> twt{tw, t};
        stage_butterflies<P, 0, false, 8>(v);
        if constexpr (Geo<P>::NST > 1) twt.template apply<0, false>(v);
        if (threadIdx.x == 0) tma_store_wait_read();
        __syncthreads();
        if constexpr (Geo<P>::NST > 1) {
            xch1<P, R, 0, 1>(sm, r, t, v);
            fwd1_from<P, R, 1, 8>(v, sm, r, t, twt);
            __syncthreads();   // every exchange read done before the tile (which aliases the region) is written
        }
#pragma unroll
        for (int e = 0; e < 16; ++e) sm[e * NT + threadIdx.x] = v[e];
        fence_proxy_async_smem();
        __syncthreads();
        if (threadIdx.x == 0) {
            const int item = g / groups_per_item, y0 = (g % groups_per_item) * R;
#pragma unroll 1
            for (int b = 0; b < P / BOX; ++b) tma_store_3d(&wmap, sm + b * BOX * R, y0, b * BOX, item + item_off);
            tma_store_commit();
        }
    }
    if (threadIdx.x == 0) tma_store_wait_read();
}

// ------------------------------------------------------------------------------------------
// Split row passes (P = 8192 = 2 Q).  A row holds Q samples zero-padded to 2 Q, so its transform is
// exactly the Q-point transforms of x_n (the even frequencies) and of x_n W_P^n (the odd ones), and
// the cropped inverse is the Q-point inverse of the even half plus W_P^-n times that of the odd half.
// The storage order along x is the split one: column h Q + e T + t holds frequency 2 k + h, k the
// Q-point frequency of register e of thread t.  Against the 8192-point transform (radix 16, 16, 16,
// 2) a row takes two exchanges of Q points per half instead of three of 2 Q, the tables of the
// Q-point transform (34 against 70 KB), and each half is a tile of its own, so that one half's copy
// runs beside the other's transform.  tw points to the Q-point twiddles, followed by W_P^n for n < Q.
// Measured, two 4096^2 fields: forward 244 us against 313 for a pair of CTAs sharing four-row tiles
// through distributed shared memory, inverse 238 against 318 for one tile buffer per CTA; the copies
// alone (no transforms) took 254 and 228 in those forms, so both now run at the rate at which TMA
// moves 32- and 16-byte column pieces.
// ------------------------------------------------------------------------------------------
template <int P>
__device__ __forceinline__ const float2* split_phase_of(const float4* tw) {
    return reinterpret_cast<const float2*>(tw + Geo<P / 2>::TW_WORDS);
}

// Forward: a CTA of 1024 threads walks groups of R = 4 rows, half by half (whole 32-byte sectors of
// each stored column, without a partner CTA).  The samples of the next half are loaded into registers
// as soon as the current tile is written, so that the loads overlap its TMA store; the store drains
// behind the first stage.  The second half reads the same rows again, from L2.
template <int P, int R, bool PRE>
__global__ void __launch_bounds__(R * (P / 32), 1)
k_row_fwd_s(const float2* __restrict__ in, long long in_item_stride, const __grid_constant__ CUtensorMap wmap,
            int item_off, int groups_per_item, int total_groups, const float4* __restrict__ tw, const Prefactor pre) {
    pdl_wait();
    constexpr int Q = P / 2, T = Q / 16, NT = R * T, BOX = kTmaBoxCols;
    extern __shared__ __align__(1024) float2 sm[];
    const int r = threadIdx.x % R, t = threadIdx.x / R;
    const float2* w = split_phase_of<P>(tw) + t;
    const TwTable<Q> twt{tw, t};
    float2 v[16];
    auto load = [&](int g) {
        const int item = g / groups_per_item, y = (g % groups_per_item) * R + r;
        const float2* src = in + item * in_item_stride + (long long)y * Q + t;
#pragma unroll
        for (int e = 0; e < 16; ++e) v[e] = __ldg(src + e * T);
    };
    int g = blockIdx.x, h = 0;
    if (g < total_groups) load(g);
#pragma unroll 1
    while (g < total_groups) {
        const int item = g / groups_per_item, y0 = (g % groups_per_item) * R;
        if constexpr (PRE) {
            const float2 fy = __ldg(pre.fy + y0 + r);
#pragma unroll
            for (int e = 0; e < 16; ++e) v[e] = cmul(v[e], cmul(__ldg(pre.fx + t + e * T), fy));
        }
        if (h) {
#pragma unroll
            for (int e = 0; e < 16; ++e) v[e] = cmul(v[e], __ldg(w + e * T));
        }
        stage_butterflies<Q, 0, false, 16>(v);
        twt.template apply<0, false>(v);
        if (threadIdx.x == 0) tma_store_wait_read();   // the previous tile, which the exchange region aliases
        __syncthreads();
        xch1<Q, R, 0, 1>(sm, r, t, v);
        fwd1_from<Q, R, 1, 16>(v, sm, r, t, twt);
        __syncthreads();   // every exchange read done before the tile is written
#pragma unroll
        for (int e = 0; e < 16; ++e) sm[e * NT + threadIdx.x] = v[e];
        const int half = h;
        h ^= 1;
        if (h == 0) g += gridDim.x;
        if (g < total_groups) load(g);
        fence_proxy_async_smem();
        __syncthreads();
        if (threadIdx.x == 0) {
#pragma unroll 1
            for (int b = 0; b < Q / BOX; ++b) tma_store_3d(&wmap, sm + b * BOX * R, y0, half * Q + b * BOX, item + item_off);
            tma_store_commit();
        }
    }
    if (threadIdx.x == 0) tma_store_wait_read();
}

// Inverse: two tile buffers, one per half, each aliasing its exchange region.  A half's tile of the
// next group is requested as soon as the half's last exchange has been read back, so it loads while
// the other half is transformed; the even half's values wait in registers for the odd ones.
template <int P, int R>
__host__ __device__ constexpr size_t row_inv_s_smem_bytes() {
    return 2 * row_smem_words<P / 2, R>() * sizeof(float2) + 2 * sizeof(uint64_t);
}

template <int P, int R, int EPI>
__global__ void __launch_bounds__(R * (P / 32), 1)
k_row_inv_s(const __grid_constant__ CUtensorMap wmap, int item_off, float2* __restrict__ out,
            long long out_item_stride, int groups_per_item, int total_groups, float scale,
            const float4* __restrict__ tw, int* status, const Epilogue ep) {
    pdl_wait();
    constexpr int Q = P / 2, T = Q / 16, NT = R * T, BOX = kTmaBoxCols;
    constexpr size_t BUF = row_smem_words<Q, R>();
    static_assert(BUF * sizeof(float2) % 128 == 0, "TMA destination");
    extern __shared__ __align__(1024) float2 sm[];
    uint64_t* mbar = reinterpret_cast<uint64_t*>(sm + 2 * BUF);
    const int r = threadIdx.x % R, t = threadIdx.x / R;
    auto issue = [&](int g, int h) {   // thread 0: half h of the R-row tile of group g
        const int item = g / groups_per_item, y0 = (g % groups_per_item) * R;
        mbar_arrive_expect_tx(mbar + h, (unsigned)(R * Q * sizeof(float2)));
#pragma unroll 1
        for (int b = 0; b < Q / BOX; ++b)
            tma_load_3d(sm + h * BUF + b * BOX * R, &wmap, mbar + h, y0, h * Q + b * BOX, item + item_off);
    };
    if (threadIdx.x == 0) {
        mbar_init(mbar, 1);
        mbar_init(mbar + 1, 1);
        if ((int)blockIdx.x < total_groups) {
            issue(blockIdx.x, 0);
            issue(blockIdx.x, 1);
        }
    }
    __syncthreads();
    const TwTable<Q> twt{tw, t};
    const float2* w = split_phase_of<P>(tw) + t;
    unsigned parity = 0;
    int h = 0;
    float2 even[16];
#pragma unroll 1
    for (int g = blockIdx.x; g < total_groups;) {
        const bool ok = mbar_wait_bounded(mbar + h, parity, status);
        float2* buf = sm + h * BUF;
        float2 v[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) v[e] = buf[e * NT + threadIdx.x];
        if (__syncthreads_or(!ok)) {   // a copy did not land: the status word says so
            // the copies of the other half still in flight land (or give up) before the block leaves
            if (h == 0 || g + (int)gridDim.x < total_groups) mbar_wait_bounded(mbar + (h ^ 1), h == 0 ? parity : parity ^ 1u, status);
            break;
        }
        inv1_to_stage0<Q, R, Geo<Q>::NST - 1, true>(v, buf, r, t, twt);
        fence_proxy_async_smem();      // the exchange reads precede the next tile load
        __syncthreads();
        if (threadIdx.x == 0 && g + (int)gridDim.x < total_groups) issue(g + gridDim.x, h);
        twt.template apply<0, true>(v);
        stage_butterflies<Q, 0, true, 16, true>(v);
        if (h == 0) {
#pragma unroll
            for (int e = 0; e < 16; ++e) even[e] = v[e];
        } else {
            const int item = g / groups_per_item, y0 = (g % groups_per_item) * R;
            const long long base = item * out_item_stride + (long long)(y0 + r) * Q;
#pragma unroll
            for (int e = 0; e < 16; ++e)
                epilogue_store<EPI>(out, ep, base + t + e * T, t + e * T, y0 + r,
                                    cscale(cadd(even[e], cmulc(v[e], __ldg(w + e * T))), scale));
            g += gridDim.x;
            parity ^= 1u;
        }
        h ^= 1;
    }
}

// Inverse, persistent: R rows per group, one tile buffer.  The tile of the NEXT group is
// requested as soon as the last exchange of the current group has been read back, so its load
// overlaps the last stage, the crop and the stores of the current group.
template <int P, int R> constexpr int row_inv_p_min_blocks() { return R * (P / 16) >= 1024 ? 1 : 1024 / (R * (P / 16)); }

template <int P, int R, int EPI>
__global__ void __launch_bounds__(R * (P / 16), row_inv_p_min_blocks<P, R>())
k_row_inv_p(const __grid_constant__ CUtensorMap wmap, int item_off, float2* __restrict__ out,
            long long out_item_stride, int groups_per_item, int total_groups, float scale,
            const float4* __restrict__ tw, int* status, const Epilogue ep) {
    pdl_wait();
    constexpr int T = P / 16, N = P / 2, NT = R * T;
    constexpr int BOX = P < kTmaBoxCols ? P : kTmaBoxCols;
    static_assert(Geo<P>::NST >= 2, "at least two stages");
    extern __shared__ __align__(1024) float2 sm[];
    uint64_t* mbar = reinterpret_cast<uint64_t*>(sm + row_smem_words<P, R>());   // after the tile
    const int r = threadIdx.x % R, t = threadIdx.x / R;
    auto issue = [&](int g) {   // thread 0: the R-row tile of group g
        const int item = g / groups_per_item, y0 = (g % groups_per_item) * R;
        mbar_arrive_expect_tx(mbar, (unsigned)(R * P * sizeof(float2)));
#pragma unroll 1
        for (int b = 0; b < P / BOX; ++b) tma_load_3d(sm + b * BOX * R, &wmap, mbar, y0, b * BOX, item + item_off);
    };
    if (threadIdx.x == 0) {
        mbar_init(mbar, 1);
        if ((int)blockIdx.x < total_groups) issue(blockIdx.x);
    }
    __syncthreads();
    const TwTable<P> twt{tw, t};
    unsigned parity = 0;
#pragma unroll 1
    for (int g = blockIdx.x; g < total_groups; g += gridDim.x, parity ^= 1u) {
        const bool ok = mbar_wait_bounded(mbar, parity, status);
        float2 v[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) v[e] = sm[e * NT + threadIdx.x];
        if (__syncthreads_or(!ok)) break;          // a copy did not land: the status word says so
        inv1_to_stage0<P, R, Geo<P>::NST - 1, P == 4096>(v, sm, r, t, twt);
        fence_proxy_async_smem();                  // the exchange reads precede the next tile load
        __syncthreads();
        if (threadIdx.x == 0 && g + (int)gridDim.x < total_groups) issue(g + gridDim.x);
        twt.template apply<0, true>(v);
        stage_butterflies<P, 0, true, 16, P == 4096>(v);
        const int item = g / groups_per_item, y0 = (g % groups_per_item) * R;
        const long long base = item * out_item_stride + (long long)(y0 + r) * N;
#pragma unroll
        for (int e = 0; e < 8; ++e) epilogue_store<EPI>(out, ep, base + t + e * T, t + e * T, y0 + r, cscale(v[e], scale));   // crop
    }
}

// Turn (P <= 2048): the inverse row pass of one propagation and the forward row pass of the next
// in one kernel, for loops that constrain the field between propagations (the GS iteration of
// Section "GS algorithm").  A CTA loads its R rows of the intermediate by TMA, takes their
// inverse FFTs, crops to the Nx kept samples, scales, applies the constraint (EPI_PHASE or
// EPI_AMPLITUDE), zero-pads and takes the forward FFTs, and stores the R rows back into the same
// place of the intermediate by TMA (in place: no other CTA touches these rows).  The inverse
// ends with register e of thread t at position t + e T, which is where the forward's first
// stage takes its inputs, so the crop, constraint and padding act on the registers and no
// exchange is added; each row's arithmetic is that of k_row_inv_p followed by k_row_fwd_p, so
// the loop computes bit for bit what the separate passes compute through the stored field (not at
// P = 4096, where k_row_inv_p merges its roots).
template <int P, int R, int EPI>
__global__ void __launch_bounds__(R * (P / 16))
k_row_turn(const __grid_constant__ CUtensorMap wmap, int groups_per_item, long long field_item_stride,
           float scale, const float4* __restrict__ tw, int* status, const Epilogue ep) {
    pdl_wait();
    constexpr int T = P / 16, N = P / 2, NT = R * T;
    constexpr int BOX = P < kTmaBoxCols ? P : kTmaBoxCols;
    static_assert(Geo<P>::NST >= 2, "at least two stages");
    extern __shared__ __align__(1024) float2 sm[];
    uint64_t* mbar = reinterpret_cast<uint64_t*>(sm + row_smem_words<P, R>());   // after the tile
    const int r = threadIdx.x % R, t = threadIdx.x / R;
    const int g = blockIdx.x, item = g / groups_per_item, y0 = (g % groups_per_item) * R;
    if (threadIdx.x == 0) {
        mbar_init(mbar, 1);
        mbar_arrive_expect_tx(mbar, (unsigned)(R * P * sizeof(float2)));
#pragma unroll 1
        for (int b = 0; b < P / BOX; ++b) tma_load_3d(sm + b * BOX * R, &wmap, mbar, y0, b * BOX, item);
    }
    __syncthreads();
    const bool ok = mbar_wait_bounded(mbar, 0, status);
    float2 v[16];
#pragma unroll
    for (int e = 0; e < 16; ++e) v[e] = sm[e * NT + threadIdx.x];
    if (__syncthreads_or(!ok)) return;         // a copy did not land: the status word says so
    const TwTable<P> twt{tw, t};
    inv1_to_stage0<P, R, Geo<P>::NST - 1>(v, sm, r, t, twt);
    twt.template apply<0, true>(v);
    stage_butterflies<P, 0, true, 16>(v);
    const long long base = item * field_item_stride + (long long)(y0 + r) * N;
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = epilogue_value<EPI>(ep, base + t + e * T, cscale(v[e], scale));
#pragma unroll
    for (int e = 8; e < 16; ++e) v[e] = make_float2(0.f, 0.f);   // zero padding of the next transform
    // forward: the first exchange writes the positions this thread read in the last one
    fwd1_from<P, R, 0, 8>(v, sm, r, t, twt);
    __syncthreads();   // every exchange read done before the tile (which aliases the region) is written
#pragma unroll
    for (int e = 0; e < 16; ++e) sm[e * NT + threadIdx.x] = v[e];
    fence_proxy_async_smem();
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll 1
        for (int b = 0; b < P / BOX; ++b) tma_store_3d(&wmap, sm + b * BOX * R, y0, b * BOX, item);
        tma_store_commit_and_drain();
    }
}

template <int P, int EPI>
static cudaError_t row_turn_impl(const CUtensorMap* wmap, int ny, int items, long long field_item_stride, float scale,
                                 const float4* tw, int* status, const Epilogue& ep, cudaStream_t st) {
    static_assert(P >= 64 && P <= 2048, "row_turn_supported");
    constexpr int R = rows_fwd<P>();
    constexpr int T = P / 16;
    if (ny % R || items < 1 || !status) return cudaErrorInvalidValue;
    const size_t smem = row_smem_words<P, R>() * sizeof(float2) + sizeof(uint64_t);
    cudaError_t e = kernel_setup<k_row_turn<P, R, EPI>>(smem, R * T, nullptr);
    if (e != cudaSuccess) return e;
    const int groups = ny / R;
    return pdl_launch(k_row_turn<P, R, EPI>, dim3((unsigned)(groups * items)), dim3(R * T), smem, st, *wmap, groups,
                      field_item_stride, scale, tw, status, ep);
}

template <int P, bool PRE>
static cudaError_t row_fwd_impl_t(const float2* in, long long in_item_stride, const CUtensorMap* wmap,
                                  int item_off, int ny, int items, const float4* tw, int* status, const Prefactor& pre,
                                  cudaStream_t st) {
    constexpr int R = rows_fwd<P>();
    constexpr int T = P / 16;
    if (ny % R) return cudaErrorInvalidValue;
    if constexpr (P >= 8192) {
        const size_t smem = row_smem_words<P / 2, R>() * sizeof(float2);
        int resident = 0;
        cudaError_t e = kernel_setup<k_row_fwd_s<P, R, PRE>>(smem, R * T / 2, &resident);
        if (e != cudaSuccess) return e;
        const int groups = (ny / R) * items;
        const int grid = std::min(groups, resident);
        if (grid < 1) return cudaErrorInvalidConfiguration;
        return pdl_launch(k_row_fwd_s<P, R, PRE>, dim3(grid), dim3(R * T / 2), smem, st, in, in_item_stride, *wmap, item_off,
                          ny / R, groups, tw, pre);
    } else {
    // persistent pipelined kernel where its bulk copies are legal: rows start on 16-byte boundaries
    const bool aligned = ((uintptr_t)in % 16 == 0) && (in_item_stride % 2 == 0);
    if (P >= 512 && aligned) {
        const size_t smem = row_fwd_p_smem_bytes<P, R>();
        int resident = 0;
        cudaError_t e = kernel_setup<k_row_fwd_p<P, R, PRE>>(smem, R * T, &resident);
        if (e != cudaSuccess) return e;
        const int groups = (ny / R) * items;
        const int grid = std::min(groups, resident);
        if (grid > 0) {
            return pdl_launch(k_row_fwd_p<P, R, PRE>, dim3(grid), dim3(R * T), smem, st, in, in_item_stride, *wmap,
                              item_off, ny / R, groups, tw, status, pre);
        }
    }
    const size_t smem = row_smem_words<P, R>() * sizeof(float2);
    cudaError_t e = kernel_setup<k_row_fwd<P, R, PRE>>(smem, R * T, nullptr);
    if (e != cudaSuccess) return e;
    dim3 grid(ny / R, items);
    return pdl_launch(k_row_fwd<P, R, PRE>, grid, dim3(R * T), smem, st, in, in_item_stride, *wmap, item_off, tw, pre);
    }
}

template <int P>
static cudaError_t row_fwd_impl(const float2* in, long long in_item_stride, const CUtensorMap* wmap,
                                int item_off, int ny, int items, const float4* tw, int* status, const Prefactor& pre,
                                cudaStream_t st) {
    if (pre.fx || pre.fy) {
        if (!pre.fx || !pre.fy) return cudaErrorInvalidValue;
        return row_fwd_impl_t<P, true>(in, in_item_stride, wmap, item_off, ny, items, tw, status, pre, st);
    }
    return row_fwd_impl_t<P, false>(in, in_item_stride, wmap, item_off, ny, items, tw, status, pre, st);
}

template <int P, int EPI>
static cudaError_t row_inv_impl_e(const CUtensorMap* wmap, int item_off, float2* out, long long out_item_stride,
                                  int ny, int items, float scale, const float4* tw, int* status, const Epilogue& ep,
                                  cudaStream_t st) {
    constexpr int R = rows_inv<P>();
    constexpr int T = P / 16;
    const size_t smem = row_smem_words<P, R>() * sizeof(float2) + sizeof(uint64_t);   // tile + mbarrier
    if (ny % R) return cudaErrorInvalidValue;
    if constexpr (P >= 8192) {
        const size_t ssmem = row_inv_s_smem_bytes<P, R>();
        int resident = 0;
        cudaError_t e = kernel_setup<k_row_inv_s<P, R, EPI>>(ssmem, R * T / 2, &resident);
        if (e != cudaSuccess) return e;
        const int groups = (ny / R) * items;
        const int grid = std::min(groups, resident);
        if (grid < 1) return cudaErrorInvalidConfiguration;
        return pdl_launch(k_row_inv_s<P, R, EPI>, dim3(grid), dim3(R * T / 2), ssmem, st, *wmap, item_off, out,
                          out_item_stride, ny / R, groups, scale, tw, status, ep);
    } else {
    if constexpr (kRowInvPersistent && P >= 512) {
        int resident = 0;
        cudaError_t e = kernel_setup<k_row_inv_p<P, R, EPI>>(smem, R * T, &resident);
        if (e != cudaSuccess) return e;
        const int groups = (ny / R) * items;
        const int grid = std::min(groups, resident);
        if (grid > 0) {
            return pdl_launch(k_row_inv_p<P, R, EPI>, dim3(grid), dim3(R * T), smem, st, *wmap, item_off, out,
                              out_item_stride, ny / R, groups, scale, tw, status, ep);
        }
    }
    cudaError_t e = kernel_setup<k_row_inv<P, R, EPI>>(smem, R * T, nullptr);
    if (e != cudaSuccess) return e;
    dim3 grid(ny / R, items);
    return pdl_launch(k_row_inv<P, R, EPI>, grid, dim3(R * T), smem, st, *wmap, item_off, out, out_item_stride, scale, tw,
                      status, ep);
    }
}

template <int P>
static cudaError_t row_inv_impl(const CUtensorMap* wmap, int item_off, float2* out, long long out_item_stride,
                                int ny, int items, float scale, const float4* tw, int* status, const Epilogue& ep,
                                cudaStream_t st) {
    switch (ep.mode) {
        case EPI_NONE: return row_inv_impl_e<P, EPI_NONE>(wmap, item_off, out, out_item_stride, ny, items, scale, tw, status, ep, st);
        case EPI_PHASE: return row_inv_impl_e<P, EPI_PHASE>(wmap, item_off, out, out_item_stride, ny, items, scale, tw, status, ep, st);
        case EPI_AMPLITUDE:
            return row_inv_impl_e<P, EPI_AMPLITUDE>(wmap, item_off, out, out_item_stride, ny, items, scale, tw, status, ep, st);
        case EPI_INTENSITY:
            return row_inv_impl_e<P, EPI_INTENSITY>(wmap, item_off, out, out_item_stride, ny, items, scale, tw, status, ep, st);
        case EPI_SEPARABLE:
            return row_inv_impl_e<P, EPI_SEPARABLE>(wmap, item_off, out, out_item_stride, ny, items, scale, tw, status, ep, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace cwo

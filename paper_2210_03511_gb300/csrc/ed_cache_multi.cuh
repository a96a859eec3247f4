// Stored-structure H.x for several FP32 vectors (2 to 8, real or complex),
// instantiated per value kind in ed_cache_multi_k<K>.cu.
//
// With the vectors one after another each element gathers a 32-byte sector per
// vector.  So x is first copied to [row][NP] (NP = 2, 4 or 8 >= NV vectors): all
// vectors' x_j of an element lie in one run.  Bound by the L1 data pipe (two
// loads of up to 32 bytes per lane).  square32, copy included, against one
// one-vector pass after another: two real vectors 0.30 against 0.49 ms, five
// 0.71 against 1.22, eight 0.81 against 1.95 (at first, one kernel gathering
// vector by vector: five in 1.81 ms).  FP64 vectors take one-vector passes: they
// are bound by the FP64 pipe, and the copy won nothing (square32, three vectors:
// 0.94 against 1.00 ms real, 1.85 against 1.82 complex).
// The sums are those of the one-vector pass, entry by entry.
#pragma once

#include <string.h>

#include "ed_cache_walk.cuh"

namespace ed {

template <int NV>
constexpr int padded = NV <= 2 ? 2 : (NV <= 4 ? 4 : 8);

// The first NV of a row's NP elements, in loads of 16 bytes and a shorter last one.
template <typename T, int NV>
struct Row {
    T v[NV];
};

template <typename T, int NV>
__device__ __forceinline__ Row<T, NV> load_row(const T* __restrict__ p) {
    constexpr int bytes = NV * (int)sizeof(T);
    constexpr int full = bytes / 16, rest = bytes % 16;
    union {
        uint4 q[(bytes + 15) / 16];
        Row<T, NV> r;
    } u;
#pragma unroll
    for (int i = 0; i < full; ++i) u.q[i] = __ldg((const uint4*)p + i);
    if constexpr (rest == 4) {
        u.q[full].x = __ldg((const unsigned*)((const uint4*)p + full));
    } else if constexpr (rest == 8) {
        const uint2 e = __ldg((const uint2*)((const uint4*)p + full));
        u.q[full].x = e.x;
        u.q[full].y = e.y;
    } else if constexpr (rest == 12) {
        u.q[full] = __ldg((const uint4*)p + full);  // the fourth is the padding of NP = 4 or 8
    }
    return u.r;
}

// xi[i][NP] = row i of the vectors of all sectors (one sector: row_off null).
template <typename T, int NP>
__global__ void interleave_kernel(T* __restrict__ xi, const T* __restrict__ x, int64_t total, int nvec,
                                  const int64_t* __restrict__ row_off, int n_sec, const int* __restrict__ x_step,
                                  int64_t x_step_elems) {
    struct alignas(NP * sizeof(T) >= 16 ? 16 : NP * sizeof(T)) Out {
        T v[NP];
    };
    if (x_step) x += (int64_t)(*x_step) * x_step_elems;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        int64_t off = 0, D = total;
        if (row_off) {
            int lo = 0, hi = n_sec - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (row_off[mid] <= i) lo = mid;
                else hi = mid - 1;
            }
            off = row_off[lo];
            D = row_off[lo + 1] - off;
        }
        const T* __restrict__ src = x + (int64_t)nvec * off + (i - off);
        Out o;
        memset(&o, 0, sizeof(Out));
#pragma unroll
        for (int v = 0; v < NP; ++v)
            if (v < nvec) o.v[v] = src[(int64_t)v * D];
        *(Out*)(xi + i * NP) = o;
    }
}

// entries in flight: about 64 bytes of gathered x per lane, at most AHEAD
template <typename T, int NV>
constexpr int multi_ahead = NV * sizeof(T) > 32 ? 1 : (NV * sizeof(T) > 16 ? 2 : AHEAD);
template <typename T, int NV>
constexpr int multi_blocks = NV * sizeof(T) > 32 ? 2 : (NV * sizeof(T) > 16 ? 3 : 4);

template <int K, int NV>
__global__ void __launch_bounds__(BLOCK, multi_blocks<typename Val<K>::T, NV>) cache_pass_multi(CachePass p) {
    using V = Val<K>;
    using T = typename V::T;
    using R = typename V::R;
    using CT = typename std::conditional<V::cplx, T, R>::type;
    constexpr int NP = padded<NV>;
    __shared__ CT ctab[NCODE];
    stage_codes<K>(ctab, p.ctab);
    write_counters(p);
    __syncthreads();
    const T* __restrict__ xi = (const T*)p.xi;
    T* __restrict__ y = (T*)p.y;
    const int lane = threadIdx.x & 31;
    const int64_t D = p.D;
    const uint32_t ob = p.off_bits, om = (1u << ob) - 1u;
    const bool last = p.mode == 0 || p.mode == 3, prev = p.mode >= 2;
    const T* __restrict__ xs = xi + p.xoff * NP;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    int64_t sl = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    Ahead nx;
    if (sl < p.ns) nx.load(p, sl, lane);
    for (; sl < p.ns; sl += warps) {
        const uint32_t c = nx.c;
        const uint32_t* ent = nx.base + nx.bo;
        if (sl + warps < p.ns) nx.load(p, sl + warps, lane);
        const int64_t row = sl * NSLICE + lane;
        const bool keep = row < D && (c > 0 || last || !prev);  // the row's y is written
        RowSum<K, false> sum[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v)
            if (prev && keep) sum[v].start(y[(int64_t)v * D + row]);
        walk<Row<T, NV>, multi_ahead<T, NV>>(
            c, ent, 0u, 255u, lane, [&](uint32_t w) { return load_row<T, NV>(xs + (int64_t)(w & om) * NP); },
            [&](uint32_t w, const Row<T, NV>& xj) {
                const CT cf = ctab[w >> ob];
#pragma unroll
                for (int v = 0; v < NV; ++v) sum[v].add(cf, false, xj.v[v]);
            });
        if (!keep) continue;
        R inv = 0, dg = 0;
        Row<T, NV> xr;
        if (last) {
            inv = ((const R*)p.isq)[__ldg(p.stab + row)];
            dg = (R)__ldg(p.diag + row);
            xr = load_row<T, NV>(xi + row * NP);
        }
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            sum[v].close();
            finish<K>(y + (int64_t)v * D + row, &xr.v[v], sum[v].re, sum[v].im, last, inv, dg);
        }
    }
}

// All sectors of a batch (cache_batch_kernel of ed_cache_pass.cu for several vectors).
template <int K, int NV>
__global__ void __launch_bounds__(BLOCK, multi_blocks<typename Val<K>::T, NV>)
    cache_batch_multi(const CacheSector* __restrict__ sec, int n_sec, int64_t n_slices,
                      const int64_t* __restrict__ row_off, const void* xiv, void* yv,
                      const int* __restrict__ active) {
    using V = Val<K>;
    using T = typename V::T;
    using R = typename V::R;
    using CT = typename std::conditional<V::cplx, T, R>::type;
    constexpr int NP = padded<NV>;
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t gs = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); gs < n_slices; gs += warps) {
        int lo = 0, hi = n_sec - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (sec[mid].slice0 <= gs) lo = mid;
            else hi = mid - 1;
        }
        if (active && !active[lo]) continue;  // uniform over the warp
        const CacheSector& c = sec[lo];
        const int64_t ls = gs - c.slice0, D = c.D, row = ls * NSLICE + lane;
        const T* __restrict__ xi = (const T*)xiv + row_off[lo] * NP;
        T* __restrict__ y = (T*)yv + (int64_t)NV * row_off[lo];
        const CT* __restrict__ ctab = (const CT*)(c.ctab + (K == 0 || K == 2 ? CT_D2 : CT_F2));
        const R* __restrict__ isq;
        if constexpr (K == 0 || K == 2) isq = (const R*)c.sq + c.G1;
        else isq = (const R*)c.sqf + c.G1;
        const uint32_t ob = c.off_bits, om = (1u << ob) - 1u;
        RowSum<K, false> sum[NV];
        walk<Row<T, NV>, multi_ahead<T, NV>>(
            __ldg(c.counts + row), c.ent[ls >> c.chunk_shift] + __ldg(c.boff + ls), 0u, 255u, lane,
            [&](uint32_t w) { return load_row<T, NV>(xi + (int64_t)(w & om) * NP); },
            [&](uint32_t w, const Row<T, NV>& xj) {
                const CT cf = __ldg(ctab + (V::cplx ? 1 : 2) * (w >> ob));
#pragma unroll
                for (int v = 0; v < NV; ++v) sum[v].add(cf, false, xj.v[v]);
            });
        if (row >= D) continue;
        const R inv = isq[__ldg(c.stab + row)];
        const R dg = (R)__ldg(c.diag + row);
        const Row<T, NV> xr = load_row<T, NV>(xi + row * NP);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            sum[v].close();
            finish<K>(y + (int64_t)v * D + row, &xr.v[v], sum[v].re, sum[v].im, true, inv, dg);
        }
    }
}

template <typename F>
ed_status with_nvec(int nvec, F&& f) {
    switch (nvec) {
        case 2: return f(std::integral_constant<int, 2>{});
        case 3: return f(std::integral_constant<int, 3>{});
        case 4: return f(std::integral_constant<int, 4>{});
        case 5: return f(std::integral_constant<int, 5>{});
        case 6: return f(std::integral_constant<int, 6>{});
        case 7: return f(std::integral_constant<int, 7>{});
        case 8: return f(std::integral_constant<int, 8>{});
    }
    return fail(ED_ERR_ARG, "nvec out of range [2,8]");
}

template <int K, int NV>
void launch_interleave(void* xi, const void* x, int64_t total, const int64_t* row_off, int n_sec, const int* x_step,
                       int64_t x_step_elems, int sms, cudaStream_t s) {
    using T = typename Val<K>::T;
    const unsigned g = (unsigned)std::max<int64_t>(1, std::min<int64_t>((total + 255) / 256, (int64_t)sms * 8));
    interleave_kernel<T, padded<NV>><<<g, 256, 0, s>>>((T*)xi, (const T*)x, total, NV, row_off, n_sec, x_step,
                                                       x_step_elems);
}

template <int K>
ed_status pass_multi_kind(const CachePass& p, int sms, cudaStream_t s) {
    return with_nvec(p.nvec, [&](auto nv) -> ed_status {
        constexpr int NV = decltype(nv)::value;
        if (p.mode < 2) launch_interleave<K, NV>(p.xi, p.x, p.D, nullptr, 1, nullptr, 0, sms, s);
        const int64_t need = (p.ns + (BLOCK / 32) - 1) / (BLOCK / 32);
        const int64_t fit = (int64_t)sms * multi_blocks<typename Val<K>::T, NV>;
        const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(need, fit));
        cache_pass_multi<K, NV><<<grid, BLOCK, 0, s>>>(p);
        ED_CUDA(cudaGetLastError());
        return ED_OK;
    });
}

template <int K>
ed_status batch_multi_kind(const BatchLaunch& L, int sms, cudaStream_t s) {
    return with_nvec(L.nvec, [&](auto nv) -> ed_status {
        constexpr int NV = decltype(nv)::value;
        launch_interleave<K, NV>(L.xi, L.x, L.total_rows, L.row_off, L.n_sec, L.x_step, L.x_step_elems, sms, s);
        const int64_t need = (L.stored_slices + (BLOCK / 32) - 1) / (BLOCK / 32);
        const int64_t fit = (int64_t)sms * multi_blocks<typename Val<K>::T, NV>;
        const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(need, fit));
        cache_batch_multi<K, NV><<<grid, BLOCK, 0, s>>>(L.stored, L.n_sec, L.stored_slices, L.row_off, L.xi, L.y,
                                                        L.active);
        ED_CUDA(cudaGetLastError());
        return ED_OK;
    });
}

}  // namespace ed

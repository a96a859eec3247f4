// Stored-structure H.x for several FP32 vectors (2 to 8, real or complex),
// instantiated per value kind in ed_cache_multi_k<K>.cu.
//
// With one-vector passes each element gathers a 32-byte sector per vector.  So, where
// the sector is not small (cache_interleaved_bytes), x is first copied to [row][NP]
// (NP = 2, 4 or 8 >= NV vectors): all vectors' x_j of an element lie in one run.
// Bound by the L1 data pipe.  square32, copy included, against one-vector passes side
// by side: two real vectors 0.31 against 0.47 ms, five 0.58 against 1.11, eight 0.58
// against 1.74, five complex 1.34 against 1.49 (one lane per row: five 0.71, eight 0.81,
// five complex 1.62; at first, one kernel gathering vector by vector: five in 1.81 ms).
// FP64 vectors take one-vector passes: they are bound by the FP64 pipe, and the copy won
// nothing (square32, three vectors: 0.94 against 0.95 ms real, 1.85 against 1.75 complex).
// The sums are those of the one-vector pass, entry by entry (complex vectors too: axis-aligned
// tables where that takes them), so y does not depend on whether there was room for the copy.
#pragma once

#include <string.h>

#include "ed_cache_walk.cuh"

namespace ed {

template <int NV>
constexpr int padded = NV <= 2 ? 2 : (NV <= 4 ? 4 : 8);

// A row of more than 16 bytes is read in two halves by two neighbouring lanes, each
// taking its half of the rows of both lanes one after another: the lanes of a load
// then share sectors, where one lane reading its whole row fetches every sector
// twice and more through the L1 data pipe.  (Four lanes to a 64-byte row were
// slower: five complex vectors 2.09 against 1.34 ms.)
template <typename T, int NV>
struct Layout {
    static constexpr int NP = padded<NV>;
    static constexpr int G = NP * sizeof(T) <= 16 ? 1 : 2;
    static constexpr int P = NP / G;  // elements of a lane's part
};

template <typename T, int NV>
struct Parts {
    T v[Layout<T, NV>::G][Layout<T, NV>::P];  // [row of the group][element of this lane's part]
    uint32_t w[Layout<T, NV>::G];             // the rows' entry words
};

template <typename T, int P>
__device__ __forceinline__ void load_part(T (&v)[P], const T* __restrict__ p) {
    constexpr int n = P * (int)sizeof(T) / 16;
    union {
        uint4 q[n ? n : 1];
        uint2 d;
        T e[P];
    } u;
    if constexpr (n == 0) u.d = __ldg((const uint2*)p);
#pragma unroll
    for (int i = 0; i < n; ++i) u.q[i] = __ldg((const uint4*)p + i);
#pragma unroll
    for (int j = 0; j < P; ++j) v[j] = u.e[j];
}

// The sums of one slice: this lane's part of the rows of its group.
template <int K, int NV, bool AX>
struct GroupSum {
    using T = typename Val<K>::T;
    using R = typename Val<K>::R;
    using L = Layout<T, NV>;
    RowSum<K, AX> sum[L::G][L::P];

    template <typename Coef>
    __device__ __forceinline__ void run(uint32_t c, const uint32_t* ent, const T* __restrict__ xs, uint32_t ob,
                                        uint32_t n_re, int lane, Coef&& coef) {
        constexpr int bytes = L::NP * (int)sizeof(T);
        constexpr int ahead = bytes > 16 ? 2 : AHEAD;
        const uint32_t om = (1u << ob) - 1u;
        const int h = lane % L::G, l0 = lane - h;
        walk<Parts<T, NV>, ahead, true>(
            c, ent, 0u, 255u, lane,
            [&](uint32_t w) {
                Parts<T, NV> x;
#pragma unroll
                for (int r = 0; r < L::G; ++r) {
                    x.w[r] = L::G == 1 ? w : __shfl_sync(FULL, w, l0 + r);
                    load_part<T, L::P>(x.v[r], xs + (int64_t)(x.w[r] & om) * L::NP + h * L::P);
                }
                return x;
            },
            [&](uint32_t, const Parts<T, NV>& x, unsigned has) {
#pragma unroll
                for (int r = 0; r < L::G; ++r) {
                    if (!((has >> (l0 + r)) & 1u)) continue;
                    const uint32_t cd = x.w[r] >> ob;
                    const auto cf = coef(cd);
#pragma unroll
                    for (int j = 0; j < L::P; ++j) sum[r][j].add(cf, AX && cd >= n_re, x.v[r][j]);
                }
            });
    }
};

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

template <typename T, int NV>
constexpr int multi_blocks = Layout<T, NV>::NP * sizeof(T) > 32 ? 2 : 4;  // five real vectors 0.58 ms against 0.64 (3)

template <int K, int NV, bool AX>
__global__ void __launch_bounds__(BLOCK, multi_blocks<typename Val<K>::T, NV>) cache_pass_multi(CachePass p) {
    using V = Val<K>;
    using T = typename V::T;
    using R = typename V::R;
    using CT = typename std::conditional<V::cplx, T, R>::type;
    using L = Layout<T, NV>;
    constexpr int NP = L::NP;
    __shared__ CT ctab[NCODE];
    stage_codes<K>(ctab, p.ctab);
    write_counters(p);
    __syncthreads();
    const T* __restrict__ xi = (const T*)p.xi;
    T* __restrict__ y = (T*)p.y;
    const int lane = threadIdx.x & 31, h = lane % L::G;
    const int64_t D = p.D;
    const uint32_t ob = p.off_bits;
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
        const int64_t first = sl * NSLICE + lane - h;  // the group's rows
        bool keep[L::G];                               // whose y is written
        GroupSum<K, NV, AX> group;
#pragma unroll
        for (int r = 0; r < L::G; ++r) {
            const uint32_t cr = L::G == 1 ? c : __shfl_sync(FULL, c, lane - h + r);
            keep[r] = first + r < D && (cr > 0 || last || !prev);
#pragma unroll
            for (int j = 0; j < L::P; ++j)
                if (prev && keep[r] && h * L::P + j < NV) group.sum[r][j].start(y[(int64_t)(h * L::P + j) * D + first + r]);
        }
        group.run(c, ent, xs, ob, p.n_re, lane, [&](uint32_t cd) { return ctab[cd]; });
#pragma unroll
        for (int r = 0; r < L::G; ++r) {
            if (!keep[r]) continue;
            const int64_t row = first + r;
            R inv = 0, dg = 0;
            T xr[L::P];
            if (last) {
                inv = ((const R*)p.isq)[__ldg(p.stab + row)];
                dg = (R)__ldg(p.diag + row);
                load_part<T, L::P>(xr, xi + row * NP + h * L::P);
            }
#pragma unroll
            for (int j = 0; j < L::P; ++j) {
                if (h * L::P + j >= NV) continue;
                RowSum<K, AX>& sm = group.sum[r][j];
                sm.close();
                finish<K>(y + (int64_t)(h * L::P + j) * D + row, &xr[j], sm.re, sm.im, last, inv, dg);
            }
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
    using L = Layout<T, NV>;
    constexpr int NP = L::NP;
    const int lane = threadIdx.x & 31, h = lane % L::G;
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
        const CT* __restrict__ ctab = (const CT*)(c.ctab + ct_offset<K>);
        const R* __restrict__ isq;
        if constexpr (K == 0 || K == 2) isq = (const R*)c.sq + c.G1;
        else isq = (const R*)c.sqf + c.G1;
        GroupSum<K, NV, false> group;
        group.run(__ldg(c.counts + row), c.ent[ls >> c.chunk_shift] + __ldg(c.boff + ls), xi, c.off_bits, 0u, lane,
               [&](uint32_t cd) { return __ldg(ctab + ct_step<K> * cd); });
#pragma unroll
        for (int r = 0; r < L::G; ++r) {
            const int64_t at = row - h + r;
            if (at >= D) continue;
            const R inv = isq[__ldg(c.stab + at)];
            const R dg = (R)__ldg(c.diag + at);
            T xr[L::P];
            load_part<T, L::P>(xr, xi + at * NP + h * L::P);
#pragma unroll
            for (int j = 0; j < L::P; ++j) {
                if (h * L::P + j >= NV) continue;
                RowSum<K, false>& sm = group.sum[r][j];
                sm.close();
                finish<K>(y + (int64_t)(h * L::P + j) * D + at, &xr[j], sm.re, sm.im, true, inv, dg);
            }
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
ed_status pass_multi_kind(const CachePass& p, bool ax, int sms, cudaStream_t s) {
    return with_nvec(p.nvec, [&](auto nv) -> ed_status {
        constexpr int NV = decltype(nv)::value;
        if (p.mode < 2) launch_interleave<K, NV>(p.xi, p.x, p.D, nullptr, 1, nullptr, 0, sms, s);
        const int64_t need = (p.ns + (BLOCK / 32) - 1) / (BLOCK / 32);
        const int64_t fit = (int64_t)sms * multi_blocks<typename Val<K>::T, NV>;
        const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(need, fit));
        if constexpr (Val<K>::cplx) {
            if (ax) cache_pass_multi<K, NV, true><<<grid, BLOCK, 0, s>>>(p);
            else cache_pass_multi<K, NV, false><<<grid, BLOCK, 0, s>>>(p);
        } else {
            cache_pass_multi<K, NV, false><<<grid, BLOCK, 0, s>>>(p);
        }
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

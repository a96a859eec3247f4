// Device helpers of the stored-structure pass kernels (ed_cache_pass.cu,
// ed_cache_multi.cuh).
#pragma once

#include "ed_cache.cuh"

namespace ed {

constexpr unsigned FULL = 0xffffffffu;
constexpr int AHEAD = 4;   // entries in flight per lane (measured: ed_cache_pass.cu)

// Walk entries [k0, k1) of every row of a slice in order (c: entries of this
// lane's row; p: the slice's first entry; k0, k1 and p uniform over the warp).
// get(w) loads x for entry word w, use(w, x) adds it.  Once a row of the slice
// has ended, the places of the others' entries come from ballots.  ALL: both are
// called by the whole warp, use with the mask of the lanes that have an entry
// (the others' word is 0).
template <typename X, int U, bool ALL = false, typename Get, typename Use>
__device__ __forceinline__ void walk(uint32_t c, const uint32_t* p, uint32_t k0, uint32_t k1, int lane, Get&& get,
                                     Use&& use) {
    const uint32_t cmin = __reduce_min_sync(FULL, c);
    k1 = min(k1, __reduce_max_sync(FULL, c));
    const uint32_t* __restrict__ q = p;
    if (k0) q += __reduce_add_sync(FULL, min(c, k0));
    const uint32_t kf = min(cmin, k1);
    uint32_t k = k0;
    for (; k + U <= kf; k += U, q += 32 * U) {
        uint32_t w[U];
        X xv[U];
#pragma unroll
        for (int u = 0; u < U; ++u) w[u] = __ldg(q + 32 * u + lane);
#pragma unroll
        for (int u = 0; u < U; ++u) xv[u] = get(w[u]);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if constexpr (ALL) use(w[u], xv[u], FULL);
            else use(w[u], xv[u]);
        }
    }
    const unsigned lt = (1u << lane) - 1u;
    for (; k < k1; k += U) {
        uint32_t w[U];
        X xv[U];
        bool has[U];
        unsigned m[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            has[u] = c > k + u && k + u < k1;
            m[u] = __ballot_sync(FULL, has[u]);
            w[u] = 0;
            if (has[u]) w[u] = __ldg(q + __popc(m[u] & lt));
            q += __popc(m[u]);
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (ALL || has[u]) xv[u] = get(w[u]);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if constexpr (ALL) use(w[u], xv[u], m[u]);
            else if (has[u]) use(w[u], xv[u]);
        }
    }
}

// a b rounded, never fused with what follows
__device__ __forceinline__ double prod(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float prod(float a, float b) { return __fmul_rn(a, b); }

// Sum of one row for one vector of kind K.  AX (complex kinds): every code's
// coefficient is real or purely imaginary (real characters: Heisenberg terms
// real, chirality terms imaginary), so one entry costs two real multiply-adds
// instead of four.  The real codes come first (codes below n_re); the table
// holds (c, c) for a real c and (-c, c) for i c, and the imaginary case takes
// x_j's parts swapped.
// General complex coefficients keep the four products in sums of their own: four
// instructions per entry, where re += cr x.re - ci x.im takes three per part
// (product, fused difference, addition), in FP64 on the pipe that bounds these
// passes (kagome36: 88 -> 60 ms).  Each of the two sums of a part is rounded at
// its own size, so the rounding errors stay those of the difference added in one
// go (4.2 against 4.5 10^-16, 5.6 against 5.7 of |y| on kagome sectors); two
// multiply-adds into one sum round it twice.
// DIFF: the fused difference of products, added in one go, all the same (for
// ed_lanczos: the sign of a Ritz vector hangs on the last bits of alpha and beta,
// so its recursion keeps the arithmetic that its vectors have had).  With one warp
// per slice only: several warps per slice add their parts' sums in an order of their
// own anyway, and take the four sums there too.
template <int K, bool AX, bool DIFF = false>
struct RowSum {
    using T = typename Val<K>::T;
    using R = typename Val<K>::R;
    static constexpr bool four = Val<K>::cplx && !AX && !DIFF;
    R re = 0, im = 0, re2 = 0, im2 = 0;
    __device__ __forceinline__ void start(const T& y) {
        if constexpr (Val<K>::cplx) {
            re = y.x;
            im = y.y;
        } else {
            re = y;
        }
    }
    template <typename CT>
    __device__ __forceinline__ void add(const CT& cf, bool imag, const T& x) {
        if constexpr (!Val<K>::cplx) {
            re += cf * x;
        } else if constexpr (AX) {
            re += cf.x * (imag ? x.y : x.x);
            im += cf.y * (imag ? x.x : x.y);
        } else if constexpr (DIFF) {
            re += fma(cf.x, x.x, -prod(cf.y, x.y));
            im += fma(cf.y, x.x, prod(cf.x, x.y));
        } else {
            re += cf.x * x.x;
            re2 += cf.y * x.y;
            im += cf.x * x.y;
            im2 += cf.y * x.x;
        }
    }
    __device__ __forceinline__ void close() {
        if constexpr (four) {
            re -= re2;
            im += im2;
        }
    }
};

// The row's element of y from its sum, and x's with the last segment.
template <int K>
__device__ __forceinline__ void finish(typename Val<K>::T* y, const typename Val<K>::T* x, typename Val<K>::R re,
                                       typename Val<K>::R im, bool last, typename Val<K>::R inv,
                                       typename Val<K>::R dg) {
    if constexpr (!Val<K>::cplx) {
        if (last) *y = re * inv + dg * *x;
        else *y = re;
    } else {
        typename Val<K>::T out;
        if (last) {
            const typename Val<K>::T xi = *x;
            out.x = re * inv + dg * xi.x;
            out.y = im * inv + dg * xi.y;
        } else {
            out.x = re;
            out.y = im;
        }
        *y = out;
    }
}

template <int K, typename CT>
__device__ __forceinline__ void stage_codes(CT* dst, const void* src) {
    for (int i = threadIdx.x; i < NCODE; i += blockDim.x) {
        dst[i] = ((const CT*)src)[ct_step<K> * i];
    }
}

__device__ __forceinline__ void write_counters(const CachePass& p) {
    if (p.counters && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) {
        p.counters[0] = p.n_ent;
        p.counters[1] = p.n_skip;
        p.counters[2] = 0ull;
    }
}

// What the next slice's walk starts from, loaded a slice ahead (a slice's
// dependent loads count -> offset -> entry -> x_j bound short slices otherwise).
struct Ahead {
    uint32_t c, bo;
    const uint32_t* base;
    __device__ __forceinline__ void load(const CachePass& p, int64_t sl, int lane) {
        c = __ldg(p.counts + sl * NSLICE + lane);
        bo = __ldg(p.boff + sl);
        base = (const uint32_t*)__ldg((const unsigned long long*)(p.ent + (sl >> p.chunk_shift)));
    }
};

}  // namespace ed

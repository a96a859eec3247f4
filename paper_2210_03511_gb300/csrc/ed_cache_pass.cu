// Stored-structure H.x: the pass over one column segment (ed_cache.cu builds
// the structure and describes its layout).
//
// One warp per slice of 32 rows, one lane per row.  The entries of a slice are
// interleaved: entry k of all rows that have one lie side by side, so an entry
// load of a warp is one run of 4 a_k bytes (a_k: rows with more than k
// entries).  With the rows' entries one after another instead, every lane read
// its own sector, and the two loads of an element (entry, x_j) shared the L1
// data pipe, which bounded the pass (90 % of its cycles at square32 FP64).
// One vector, before and after: square32 FP64 0.519 -> 0.342 ms (now the FP64
// pipe, 84 % of its cycles), square36 FP64 (63 10^6 rows, four segments)
// 20.2 -> 14.1 ms, kagome36 complex FP32 22.6 -> 16.2 ms.
// Neighbouring rows stay on neighbouring lanes: their images are often
// neighbours too, and sorting the rows of a window by their counts, which
// keeps a warp's lanes together to the end, cost more in x_j sectors than it
// saved (square36 FP64 22.2 against 14.0 ms, kagome36 complex FP32 27.5 against
// 16.5 ms).
#include "ed_cache.cuh"

namespace ed {

namespace {

constexpr unsigned FULL = 0xffffffffu;

// Entries in flight per lane, and resident blocks per SM (register budget
// 65536 / (256 x blocks)).  Four entries at 5 blocks (4 for complex FP64) beat
// more warps with fewer entries in flight and fewer warps with eight: square36
// FP64 13.5 ms against 14.3 (4 and 2 in the ragged rest, 6 blocks), 15.1 (2, 8
// blocks) and 13.8 (8, 4 blocks); kagome36 complex FP32 14.2 against 16.2, 17.0
// and 15.3; square32 FP64 0.334 against 0.344, 0.366 and 0.329.
constexpr int AHEAD = 4;
constexpr int pass_blocks(int K, int NV) { return NV == 1 ? (K == 2 ? 4 : 5) : 2; }

// Walk entries [k0, k1) of every row of a slice in order (c: entries of this
// lane's row; p: the slice's first entry; k0, k1 and p uniform over the warp).
// get(w) loads x for entry word w, use(w, x) adds it.  Once a row of the slice
// has ended, the places of the others' entries come from ballots.
template <typename X, typename Get, typename Use>
__device__ __forceinline__ void walk(uint32_t c, const uint32_t* p, uint32_t k0, uint32_t k1, int lane, Get&& get,
                                     Use&& use) {
    const uint32_t cmin = __reduce_min_sync(FULL, c);
    k1 = min(k1, __reduce_max_sync(FULL, c));
    const uint32_t* __restrict__ q = p;
    if (k0) q += __reduce_add_sync(FULL, min(c, k0));
    const uint32_t kf = min(cmin, k1);
    uint32_t k = k0;
    for (; k + AHEAD <= kf; k += AHEAD, q += 32 * AHEAD) {
        uint32_t w[AHEAD];
        X xv[AHEAD];
#pragma unroll
        for (int u = 0; u < AHEAD; ++u) w[u] = __ldg(q + 32 * u + lane);
#pragma unroll
        for (int u = 0; u < AHEAD; ++u) xv[u] = get(w[u]);
#pragma unroll
        for (int u = 0; u < AHEAD; ++u) use(w[u], xv[u]);
    }
    const unsigned lt = (1u << lane) - 1u;
    for (; k < k1; k += AHEAD) {
        uint32_t w[AHEAD];
        X xv[AHEAD];
        bool has[AHEAD];
#pragma unroll
        for (int u = 0; u < AHEAD; ++u) {
            has[u] = c > k + u && k + u < k1;
            const unsigned m = __ballot_sync(FULL, has[u]);
            w[u] = 0;
            if (has[u]) w[u] = __ldg(q + __popc(m & lt));
            q += __popc(m);
        }
#pragma unroll
        for (int u = 0; u < AHEAD; ++u)
            if (has[u]) xv[u] = get(w[u]);
#pragma unroll
        for (int u = 0; u < AHEAD; ++u)
            if (has[u]) use(w[u], xv[u]);
    }
}

// acc += (coefficient of w) x for one vector of kind K.  AX (complex kinds):
// every code's coefficient is real or purely imaginary (real characters:
// Heisenberg terms real, chirality terms imaginary), so one entry costs two real
// multiply-adds instead of four.  The real codes come first (codes below n_re);
// the table holds (c, c) for a real c and (-c, c) for i c, and the imaginary
// case takes x_j's parts swapped.
template <int K, bool AX, typename CT, typename T, typename R>
__device__ __forceinline__ void accumulate(R& re, R& im, const CT& cf, bool imag, const T& x) {
    if constexpr (!Val<K>::cplx) {
        re += cf * x;
    } else if constexpr (AX) {
        re += cf.x * (imag ? x.y : x.x);
        im += cf.y * (imag ? x.x : x.y);
    } else {
        cmadd(re, im, cf.x, cf.y, x);
    }
}

template <int K>
__device__ __forceinline__ void finish(typename Val<K>::T* y, const typename Val<K>::T* x, int64_t o,
                                       typename Val<K>::R re, typename Val<K>::R im, bool last,
                                       typename Val<K>::R inv, typename Val<K>::R dg) {
    if constexpr (!Val<K>::cplx) {
        if (last) y[o] = re * inv + dg * x[o];
        else y[o] = re;
    } else {
        typename Val<K>::T out;
        if (last) {
            const typename Val<K>::T xi = x[o];
            out.x = re * inv + dg * xi.x;
            out.y = im * inv + dg * xi.y;
        } else {
            out.x = re;
            out.y = im;
        }
        y[o] = out;
    }
}

template <int K, typename CT>
__device__ __forceinline__ void stage_codes(CT* dst, const void* src) {
    for (int i = threadIdx.x; i < NCODE; i += blockDim.x) {
        if constexpr (Val<K>::cplx) dst[i] = ((const CT*)src)[i];
        else dst[i] = ((const CT*)src)[2 * i];  // real part of the complex table
    }
}

__device__ __forceinline__ void write_counters(const CachePass& p) {
    if (p.counters && blockIdx.x == 0 && threadIdx.x == 0) {
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

// PREV: modes 2 and 3 (a partial sum from earlier segments exists in y), a
// compile-time flag so that the one-segment pass carries no such register.  A
// row's sum continues from that partial sum; a row without entries in an inner
// segment is left alone.
template <int K, int NV, bool AX, bool PREV>
__global__ void __launch_bounds__(BLOCK, pass_blocks(K, NV)) cache_pass_kernel(CachePass p) {
    using V = Val<K>;
    using T = typename V::T;
    using R = typename V::R;
    using CT = typename std::conditional<V::cplx, T, R>::type;
    __shared__ CT ctab[NCODE];
    stage_codes<K>(ctab, p.ctab);
    write_counters(p);
    __syncthreads();
    const T* __restrict__ x = (const T*)p.x;
    T* __restrict__ y = (T*)p.y;
    const int lane = threadIdx.x & 31;
    const int nvec = NV == 1 ? 1 : p.nvec;
    const int64_t D = p.D;
    const uint32_t ob = p.off_bits, om = (1u << ob) - 1u, n_re = p.n_re;
    const bool last = p.mode == 0 || p.mode == 3;
    const T* __restrict__ xs = x + p.xoff;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    int64_t sl = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    Ahead nx;
    if (sl < p.ns) nx.load(p, sl, lane);
    for (; sl < p.ns; sl += warps) {
        const uint32_t c = nx.c;
        const uint32_t* ent = nx.base + nx.bo;
        if (sl + warps < p.ns) nx.load(p, sl + warps, lane);
        const int64_t row = sl * NSLICE + lane;
        const bool keep = row < D && (c > 0 || last || !PREV);  // the row's y is written
        R re[NV], im[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            re[v] = im[v] = 0;
            if (PREV && v < nvec && keep) {
                const T pv = y[(int64_t)v * D + row];
                if constexpr (V::cplx) { re[v] = pv.x; im[v] = pv.y; }
                else re[v] = pv;
            }
        }
        if constexpr (NV == 1) {
            walk<T>(
                c, ent, 0u, 255u, lane, [&](uint32_t w) { return xs[w & om]; },
                [&](uint32_t w, const T& xj) {
                    const uint32_t cd = w >> ob;
                    accumulate<K, AX>(re[0], im[0], ctab[cd], cd >= n_re, xj);
                });
        } else {
            walk<char>(
                c, ent, 0u, 255u, lane, [&](uint32_t) { return (char)0; },
                [&](uint32_t w, char) {
                    const uint32_t cd = w >> ob;
                    const CT cf = ctab[cd];
#pragma unroll
                    for (int v = 0; v < NV; ++v)
                        if (v < nvec) accumulate<K, AX>(re[v], im[v], cf, cd >= n_re, xs[(int64_t)v * D + (w & om)]);
                });
        }
        if (!keep) continue;
        R inv = 0, dg = 0;
        if (last) {
            inv = ((const R*)p.isq)[__ldg(p.stab + row)];
            dg = (R)__ldg(p.diag + row);
        }
#pragma unroll
        for (int v = 0; v < NV; ++v)
            if (v < nvec) finish<K>(y, x, (int64_t)v * D + row, re[v], im[v], last, inv, dg);
    }
}

// One vector with L (2, 4 or 8) warps per slice: warp q of a group takes the
// q-th part of every row's entries, and the parts' sums are added in order in
// shared memory (ed_hamiltonian_store_set_lanes; results differ from one lane
// per row by summation order only).  For sectors with too few slices to fill
// the GPU.
template <int K, int L>
__global__ void __launch_bounds__(BLOCK, pass_blocks(K, 1)) cache_pass_split(CachePass p) {
    using V = Val<K>;
    using T = typename V::T;
    using R = typename V::R;
    using CT = typename std::conditional<V::cplx, T, R>::type;
    constexpr int G = BLOCK / 32 / L;  // slices a block works on at a time
    __shared__ CT ctab[NCODE];
    __shared__ T part[BLOCK];
    stage_codes<K>(ctab, p.ctab);
    write_counters(p);
    __syncthreads();
    const T* __restrict__ x = (const T*)p.x;
    T* __restrict__ y = (T*)p.y;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, q = warp % L;
    const uint32_t ob = p.off_bits, om = (1u << ob) - 1u;
    const bool last = p.mode == 0 || p.mode == 3;
    const T* __restrict__ xs = x + p.xoff;
    for (int64_t s0 = (int64_t)blockIdx.x * G; s0 < p.ns; s0 += (int64_t)gridDim.x * G) {  // uniform over the block
        const int64_t sl = s0 + warp / L;
        const int64_t row = sl * NSLICE + lane;
        R re = 0, im = 0;
        if (sl < p.ns) {
            Ahead a;
            a.load(p, sl, lane);
            const uint32_t n = __reduce_max_sync(FULL, a.c);
            walk<T>(
                a.c, a.base + a.bo, n * q / L, n * (q + 1) / L, lane, [&](uint32_t w) { return xs[w & om]; },
                [&](uint32_t w, const T& xj) { accumulate<K, false>(re, im, ctab[w >> ob], false, xj); });
        }
        if constexpr (V::cplx) part[threadIdx.x] = T{re, im};
        else part[threadIdx.x] = re;
        __syncthreads();
        if (q == 0 && row < p.D) {
            re = im = 0;
            if (p.mode >= 2) {
                const T pv = y[row];
                if constexpr (V::cplx) { re = pv.x; im = pv.y; }
                else re = pv;
            }
#pragma unroll
            for (int u = 0; u < L; ++u) {
                const T v = part[threadIdx.x + 32 * u];
                if constexpr (V::cplx) { re += v.x; im += v.y; }
                else re += v;
            }
            R inv = 0, dg = 0;
            if (last) {
                inv = ((const R*)p.isq)[__ldg(p.stab + row)];
                dg = (R)__ldg(p.diag + row);
            }
            finish<K>(y, x, row, re, im, last, inv, dg);
        }
        __syncthreads();
    }
}

// All sectors of a batch from their stored structures (one segment each),
// in one launch: warp w takes slice w of the concatenated slice list, finds
// its sector from the slices' first indices, and processes it as the mode-0
// pass of cache_pass_kernel (same sums, same order).  Vectors are those of a
// batch: sector s's nvec columns start at element nvec * row_off[s].  x may
// advance by x_step_elems per device-side step (block Lanczos graphs);
// sectors with active[s] == 0 are skipped.
template <int K, int NV>
__global__ void __launch_bounds__(BLOCK, pass_blocks(K, NV))
    cache_batch_kernel(const CacheSector* __restrict__ sec, int n_sec, int64_t n_slices,
                       const int64_t* __restrict__ row_off, const void* xv, void* yv, int nvec,
                       const int* __restrict__ x_step, int64_t x_step_elems, const int* __restrict__ active) {
    using V = Val<K>;
    using T = typename V::T;
    using R = typename V::R;
    using CT = typename std::conditional<V::cplx, T, R>::type;
    const T* __restrict__ xb = (const T*)xv;
    if (x_step) xb += (int64_t)(*x_step) * x_step_elems;
    T* __restrict__ yb = (T*)yv;
    const int lane = threadIdx.x & 31;
    const int nv = NV == 1 ? 1 : nvec;
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
        const int64_t ls = gs - c.slice0, D = c.D;
        const T* __restrict__ x = xb + (int64_t)nv * row_off[lo];
        T* __restrict__ y = yb + (int64_t)nv * row_off[lo];
        const CT* __restrict__ ctab = (const CT*)(c.ctab + (K == 0 || K == 2 ? CT_D2 : CT_F2));
        const R* __restrict__ isq;
        if constexpr (K == 0 || K == 2) isq = (const R*)c.sq + c.G1;
        else isq = (const R*)c.sqf + c.G1;
        const uint32_t ob = c.off_bits, om = (1u << ob) - 1u;
        const int64_t row = ls * NSLICE + lane;
        const uint32_t n = __ldg(c.counts + row);
        const uint32_t* ent = c.ent[ls >> c.chunk_shift] + __ldg(c.boff + ls);
        auto coef = [&](uint32_t w) { return __ldg(ctab + (V::cplx ? 1 : 2) * (w >> ob)); };
        R re[NV], im[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) re[v] = im[v] = 0;
        if constexpr (NV == 1) {
            walk<T>(
                n, ent, 0u, 255u, lane, [&](uint32_t w) { return x[w & om]; },
                [&](uint32_t w, const T& xj) { accumulate<K, false>(re[0], im[0], coef(w), false, xj); });
        } else {
            walk<char>(
                n, ent, 0u, 255u, lane, [&](uint32_t) { return (char)0; },
                [&](uint32_t w, char) {
                    const CT cf = coef(w);
#pragma unroll
                    for (int v = 0; v < NV; ++v)
                        if (v < nv) accumulate<K, false>(re[v], im[v], cf, false, x[(int64_t)v * D + (w & om)]);
                });
        }
        if (row >= D) continue;
        const R inv = isq[__ldg(c.stab + row)];
        const R dg = (R)__ldg(c.diag + row);
#pragma unroll
        for (int v = 0; v < NV; ++v)
            if (v < nv) finish<K>(y, x, (int64_t)v * D + row, re[v], im[v], true, inv, dg);
    }
}

template <int K, bool AX>
ed_status launch_pass(const CachePass& p, int sms, cudaStream_t s) {
    const int64_t blocks_needed = (p.ns + (BLOCK / 32) - 1) / (BLOCK / 32);
    const int per_sm = pass_blocks(K, p.nvec == 1 ? 1 : MAXV);
    const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(blocks_needed, (int64_t)sms * per_sm));
    if (p.mode >= 2) {
        if (p.nvec == 1) cache_pass_kernel<K, 1, AX, true><<<grid, BLOCK, 0, s>>>(p);
        else cache_pass_kernel<K, MAXV, AX, true><<<grid, BLOCK, 0, s>>>(p);
    } else {
        if (p.nvec == 1) cache_pass_kernel<K, 1, AX, false><<<grid, BLOCK, 0, s>>>(p);
        else cache_pass_kernel<K, MAXV, AX, false><<<grid, BLOCK, 0, s>>>(p);
    }
    ED_CUDA(cudaGetLastError());
    return ED_OK;
}

template <int K, int L>
ed_status launch_split(const CachePass& p, int sms, cudaStream_t s) {
    constexpr int G = BLOCK / 32 / L;
    const unsigned grid =
        (unsigned)std::max<int64_t>(1, std::min<int64_t>((p.ns + G - 1) / G, (int64_t)sms * pass_blocks(K, 1)));
    cache_pass_split<K, L><<<grid, BLOCK, 0, s>>>(p);
    ED_CUDA(cudaGetLastError());
    return ED_OK;
}

template <int K>
ed_status launch_kind(const CachePass& p, bool ax, int lanes, int sms, cudaStream_t s) {
    if (lanes > 1 && p.nvec == 1) {
        switch (lanes) {
            case 2: return launch_split<K, 2>(p, sms, s);
            case 4: return launch_split<K, 4>(p, sms, s);
            case 8: return launch_split<K, 8>(p, sms, s);
        }
        return fail(ED_ERR_ARG, "lanes per row must be 1, 2, 4 or 8");
    }
    if constexpr (Val<K>::cplx)
        if (ax) return launch_pass<K, true>(p, sms, s);
    return launch_pass<K, false>(p, sms, s);
}

}  // namespace

ed_status launch_cache_pass(const CachePass& p, int K, bool ax, int lanes, int sms, cudaStream_t s) {
    switch (K) {
        case 0: return launch_kind<0>(p, ax, lanes, sms, s);
        case 1: return launch_kind<1>(p, ax, lanes, sms, s);
        case 2: return launch_kind<2>(p, ax, lanes, sms, s);
        case 3: return launch_kind<3>(p, ax, lanes, sms, s);
    }
    return fail(ED_ERR_ARG, "bad value kind");
}

ed_status cache_batch_launch(const BatchLaunch& L, cudaStream_t s) {
    int dev = 0, sms = 0;
    ED_CUDA(cudaGetDevice(&dev));
    ED_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int64_t blocks_needed = (L.stored_slices + (BLOCK / 32) - 1) / (BLOCK / 32);
    auto go = [&](auto ktag) -> ed_status {
        constexpr int K = decltype(ktag)::value;
        const int64_t fit = (int64_t)sms * pass_blocks(K, L.nvec == 1 ? 1 : MAXV);
        const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(blocks_needed, fit));
        if (L.nvec == 1)
            cache_batch_kernel<K, 1><<<grid, BLOCK, 0, s>>>(L.stored, L.n_sec, L.stored_slices, L.row_off, L.x, L.y,
                                                            L.nvec, L.x_step, L.x_step_elems, L.active);
        else
            cache_batch_kernel<K, MAXV><<<grid, BLOCK, 0, s>>>(L.stored, L.n_sec, L.stored_slices, L.row_off, L.x,
                                                               L.y, L.nvec, L.x_step, L.x_step_elems, L.active);
        ED_CUDA(cudaGetLastError());
        return ED_OK;
    };
    switch (L.dtype) {
        case ED_F64: return go(std::integral_constant<int, 0>{});
        case ED_F32: return go(std::integral_constant<int, 1>{});
        case ED_C128: return go(std::integral_constant<int, 2>{});
        case ED_C64: return go(std::integral_constant<int, 3>{});
    }
    return fail(ED_ERR_ARG, "bad dtype");
}

}  // namespace ed

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
#include "ed_cache_walk.cuh"

namespace ed {

template <int K> ed_status pass_multi_kind(const CachePass& p, bool ax, int sms, cudaStream_t s);
template <int K> ed_status batch_multi_kind(const BatchLaunch& L, int sms, cudaStream_t s);
#define ED_MULTI(K)                                                                                  \
    extern template ed_status pass_multi_kind<K>(const CachePass&, bool, int, cudaStream_t);              \
    extern template ed_status batch_multi_kind<K>(const BatchLaunch&, int, cudaStream_t);
ED_MULTI(1) ED_MULTI(3)
#undef ED_MULTI

namespace {

// Resident blocks per SM of the pass kernels (register budget
// 65536 / (256 x blocks)).  Four entries in flight at 5 blocks beat more warps
// with fewer entries in flight and fewer warps with eight: square36 FP64 13.5 ms
// against 14.3 (four, two in the ragged rest, 6 blocks), 15.1 (two, 8 blocks) and
// 13.8 (eight, 4 blocks); square32 FP64 0.334 against 0.344, 0.366 and 0.329.
// Complex FP64 needs the registers of 3 blocks: the triangular24 sectors 1.57 ms
// against 1.66 (4 blocks), square32's complex sector 1.19 against 1.21.
constexpr int pass_blocks(int K) { return K == 2 ? 3 : 5; }

// Real FP32 vectors over several segments: a row has few entries per segment, so a
// warp spends its time on starting slices, and eight blocks (32 registers, nothing
// spilled, the same four entries in flight) hide that better than five.  Against
// five blocks, by entries per row and segment: square40 138.7 -> 126.3 ms (3.2) and
// 126.9 -> 118.5 (6.3), square36 12.3 -> 12.0 (4.6), 10.4 -> 9.6 (9.3) and
// 9.26 -> 8.90 (18.5), square32 0.652 -> 0.654 (3.7), 0.449 -> 0.430 (7.3) and
// 0.309 -> 0.304 (22).  Below three it loses: square36 16.9 -> 17.6 (2.4), square32
// 1.00 -> 1.06 (1.8).
constexpr int MANY_BLOCKS = 8;
constexpr uint64_t MANY_ROW_ENTRIES = 3;

// Launches of one segment with no more blocks than this per SM, and rows of twice as
// many entries as these on average: no warp waits for its turn, so a row's chain of
// entry and x_j loads bounds the call, and twice the entries in flight shorten it.
// Against four in flight, triangular24 (28,699 rows of 75 entries): real FP32 14.4 ->
// 12.3 us, FP64 16.8 -> 14.4, complex FP32 20.6 -> 16.4, FP64 24.6 -> 18.5; two complex
// FP32 vectors 20.6 -> 16.5; a batch of 2,506 real rows 10.3 -> 9.1, 12.3 -> 10.3 (FP64).
// The same sums in the same order.  Shorter rows have nothing to load ahead (chain16,
// 8.5 entries: 7.2 -> 7.6 us), and with more blocks the registers cost residents that
// the call needs.  Sixteen in flight at two blocks gained no more in these sectors
// (FP64 16.7 us).
constexpr int few_blocks(int K) { return K == 2 ? 2 : 3; }
constexpr int FEW_AHEAD = 8;
template <int K>
bool few(int64_t slices, int nvec, uint64_t entries, int64_t rows, int sms) {
    const int64_t blocks = (slices + (BLOCK / 32) - 1) / (BLOCK / 32) * nvec;
    return blocks <= (int64_t)sms * few_blocks(K) && entries >= 2 * FEW_AHEAD * (uint64_t)rows;
}

// PREV: modes 2 and 3 (a partial sum from earlier segments exists in y), a
// compile-time flag so that the one-segment pass carries no such register.  A
// row's sum continues from that partial sum; a row without entries in an inner
// segment is left alone.  MV: vector blockIdx.y of p.nvec; one vector goes without, as
// its offset costs the registers that the passes over several segments need (square36
// FP64 13.35 -> 13.73 ms, kagome36 complex FP32 14.51 -> 14.71).
template <int K, bool AX, bool PREV, bool DIFF, bool MV, int BLOCKS, int U>
__global__ void __launch_bounds__(BLOCK, BLOCKS) cache_pass_kernel(CachePass p) {
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
    const int64_t D = p.D;
    if constexpr (MV) {
        x += (int64_t)blockIdx.y * D;
        y += (int64_t)blockIdx.y * D;
    }
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
        RowSum<K, AX, DIFF> sum;
        if (PREV && keep) sum.start(y[row]);
        walk<T, U>(
            c, ent, 0u, 255u, lane, [&](uint32_t w) { return xs[w & om]; },
            [&](uint32_t w, const T& xj) {
                const uint32_t cd = w >> ob;
                sum.add(ctab[cd], cd >= n_re, xj);
            });
        if (!keep) continue;
        R inv = 0, dg = 0;
        if (last) {
            inv = ((const R*)p.isq)[__ldg(p.stab + row)];
            dg = (R)__ldg(p.diag + row);
        }
        sum.close();
        finish<K>(y + row, x + row, sum.re, sum.im, last, inv, dg);
    }
}

// One vector with L (2, 4 or 8) warps per slice: warp q of a group takes the
// q-th part of every row's entries, and the parts' sums are added in order in
// shared memory (ed_hamiltonian_store_set_lanes; results differ from one lane
// per row by summation order only).  For sectors with too few slices to fill
// the GPU.
template <int K, int L>
__global__ void __launch_bounds__(BLOCK, pass_blocks(K)) cache_pass_split(CachePass p) {
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
        RowSum<K, false> sum;
        if (sl < p.ns) {
            Ahead a;
            a.load(p, sl, lane);
            const uint32_t n = __reduce_max_sync(FULL, a.c);
            walk<T, AHEAD>(
                a.c, a.base + a.bo, n * q / L, n * (q + 1) / L, lane, [&](uint32_t w) { return xs[w & om]; },
                [&](uint32_t w, const T& xj) { sum.add(ctab[w >> ob], false, xj); });
        }
        sum.close();
        if constexpr (V::cplx) part[threadIdx.x] = T{sum.re, sum.im};
        else part[threadIdx.x] = sum.re;
        __syncthreads();
        if (q == 0 && row < p.D) {
            R re = 0, im = 0;
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
            finish<K>(y + row, x + row, re, im, last, inv, dg);
        }
        __syncthreads();
    }
}

// All sectors of a batch from their stored structures (one segment each),
// in one launch: warp w takes slice w of the concatenated slice list, finds
// its sector from the slices' first indices, and processes it as the mode-0
// pass of cache_pass_kernel (same sums, same order) for vector blockIdx.y of nvec.
// Vectors are those of a batch: sector s's nvec columns start at element
// nvec * row_off[s].  x may advance by x_step_elems per device-side step (block Lanczos graphs);
// sectors with active[s] == 0 are skipped.
template <int K, int BLOCKS, int U>
__global__ void __launch_bounds__(BLOCK, BLOCKS)
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
        const T* __restrict__ x = xb + (int64_t)nvec * row_off[lo] + (int64_t)blockIdx.y * D;
        T* __restrict__ y = yb + (int64_t)nvec * row_off[lo] + (int64_t)blockIdx.y * D;
        const CT* __restrict__ ctab = (const CT*)(c.ctab + ct_offset<K>);
        const R* __restrict__ isq;
        if constexpr (K == 0 || K == 2) isq = (const R*)c.sq + c.G1;
        else isq = (const R*)c.sqf + c.G1;
        const uint32_t ob = c.off_bits, om = (1u << ob) - 1u;
        const int64_t row = ls * NSLICE + lane;
        const uint32_t n = __ldg(c.counts + row);
        const uint32_t* ent = c.ent[ls >> c.chunk_shift] + __ldg(c.boff + ls);
        auto coef = [&](uint32_t w) { return __ldg(ctab + ct_step<K> * (w >> ob)); };
        RowSum<K, false> sum;
        walk<T, U>(
            n, ent, 0u, 255u, lane, [&](uint32_t w) { return x[w & om]; },
            [&](uint32_t w, const T& xj) { sum.add(coef(w), false, xj); });
        if (row >= D) continue;
        const R inv = isq[__ldg(c.stab + row)];
        const R dg = (R)__ldg(c.diag + row);
        sum.close();
        finish<K>(y + row, x + row, sum.re, sum.im, true, inv, dg);
    }
}

// The vectors side by side (MV), or one launch for each.
template <int K, bool AX, bool DIFF, bool MV, int BLOCKS, int U>
ed_status launch_blocks(const CachePass& p, int sms, cudaStream_t s) {
    using T = typename Val<K>::T;
    const int64_t need = (p.ns + (BLOCK / 32) - 1) / (BLOCK / 32);
    const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(need, (int64_t)sms * BLOCKS));
    CachePass q = p;
    for (int v = 0; v < p.nvec; v += MV ? p.nvec : 1) {
        const dim3 g(grid, MV ? (unsigned)p.nvec : 1u);
        q.x = (const T*)p.x + (int64_t)v * p.D;
        q.y = (T*)p.y + (int64_t)v * p.D;
        if constexpr (U == AHEAD) {
            if (p.mode >= 2) {
                cache_pass_kernel<K, AX, true, DIFF, MV, BLOCKS, U><<<g, BLOCK, 0, s>>>(q);
                continue;
            }
        }
        cache_pass_kernel<K, AX, false, DIFF, MV, BLOCKS, U><<<g, BLOCK, 0, s>>>(q);
    }
    ED_CUDA(cudaGetLastError());
    return ED_OK;
}

template <int K, bool AX, bool DIFF = false>
ed_status launch_pass(const CachePass& p, int sms, cudaStream_t s) {
    if constexpr (K == 1)  // no register left for a vector's offset: one launch per vector
        if (p.mode != 0 && p.n_ent >= MANY_ROW_ENTRIES * (uint64_t)p.D * (uint64_t)p.nb)
            return launch_blocks<K, AX, DIFF, false, MANY_BLOCKS, AHEAD>(p, sms, s);
    if (p.mode == 0 && few<K>(p.ns, p.nvec, p.n_ent, p.D, sms))
        return launch_blocks<K, AX, DIFF, true, few_blocks(K), FEW_AHEAD>(p, sms, s);
    const bool fills = p.ns > (int64_t)sms * pass_blocks(K) * (BLOCK / 32);
    return p.nvec == 1 || (p.mode != 0 && fills) ? launch_blocks<K, AX, DIFF, false, pass_blocks(K), AHEAD>(p, sms, s)
                                                 : launch_blocks<K, AX, DIFF, true, pass_blocks(K), AHEAD>(p, sms, s);
}

template <int K, int L>
ed_status launch_split(const CachePass& p, int sms, cudaStream_t s) {
    constexpr int G = BLOCK / 32 / L;
    const unsigned grid =
        (unsigned)std::max<int64_t>(1, std::min<int64_t>((p.ns + G - 1) / G, (int64_t)sms * pass_blocks(K)));
    cache_pass_split<K, L><<<grid, BLOCK, 0, s>>>(p);
    ED_CUDA(cudaGetLastError());
    return ED_OK;
}

template <int K>
ed_status launch_kind(const CachePass& p, bool ax, int lanes, int sms, cudaStream_t s) {
    if constexpr (K == 1 || K == 3)
        if (p.nvec > 1 && p.xi) return pass_multi_kind<K>(p, ax, sms, s);
    if (lanes > 1 && p.nvec == 1) {
        switch (lanes) {
            case 2: return launch_split<K, 2>(p, sms, s);
            case 4: return launch_split<K, 4>(p, sms, s);
            case 8: return launch_split<K, 8>(p, sms, s);
        }
        return fail(ED_ERR_ARG, "lanes per row must be 1, 2, 4 or 8");
    }
    // Several FP64 vectors (their passes are bound by the FP64 pipe, not by the gathers), or no
    // room for the interleaved copy: the one-vector passes, side by side in one launch (over
    // several segments only where one vector does not fill the GPU).  A launch per vector leaves
    // most of the GPU idle in a small sector: eight FP64 vectors of 12,870 rows 49 -> 8.1 us, of
    // 28,699 rows 131 -> 44 us, of 2.4 million rows 2.69 -> 2.47 ms.
    if constexpr (Val<K>::cplx)
        return ax ? launch_pass<K, true>(p, sms, s)
                  : (p.diff ? launch_pass<K, false, true>(p, sms, s) : launch_pass<K, false>(p, sms, s));
    else return launch_pass<K, false>(p, sms, s);
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

// Several FP32 vectors are copied unless the blocks of all their one-vector passes are
// resident at once: side by side these then take about as long as one, without scratch
// (whose pool takes 0.1 ms to make on an owner's first call) and without a launch for
// the copy.  triangular24 (28,699 rows, 112 blocks a vector), five vectors: real 35 -> 18 us,
// complex 38 -> 25 us; square16 (153 rows) 20.6 -> 8.3 us.  Just above the line the copy is
// as good or better: 56,682 rows of triangular24, four complex vectors 44 us side by side
// against 35, two complex ones of square26 (784 blocks) 36 against 27, two real ones 23
// against 25.
size_t cache_interleaved_bytes(ed_dtype dt, int nvec, int64_t rows, int64_t slices, int sms) {
    if (nvec < 2 || dt == ED_F64 || dt == ED_C128) return 0;
    const int K = dt == ED_F32 ? 1 : 3;
    if ((slices + (BLOCK / 32) - 1) / (BLOCK / 32) * nvec <= (int64_t)sms * pass_blocks(K)) return 0;
    return (size_t)(nvec <= 2 ? 2 : (nvec <= 4 ? 4 : 8)) * (size_t)rows * (dt == ED_F32 ? 4 : 8);
}

ed_status cache_batch_launch(const BatchLaunch& L, cudaStream_t s) {
    int dev = 0, sms = 0;
    ED_CUDA(cudaGetDevice(&dev));
    ED_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int64_t need = (L.stored_slices + (BLOCK / 32) - 1) / (BLOCK / 32);
    auto go = [&](auto ktag) -> ed_status {
        constexpr int K = decltype(ktag)::value;
        if constexpr (K == 1 || K == 3)
            if (L.nvec > 1 && L.xi) return batch_multi_kind<K>(L, sms, s);
        auto launch = [&](auto btag, auto utag) {
            constexpr int B = decltype(btag)::value;
            const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(need, (int64_t)sms * B));
            cache_batch_kernel<K, B, decltype(utag)::value><<<dim3(grid, (unsigned)L.nvec), BLOCK, 0, s>>>(
                L.stored, L.n_sec, L.stored_slices, L.row_off, L.x, L.y, L.nvec, L.x_step, L.x_step_elems, L.active);
        };
        if (few<K>(L.stored_slices, L.nvec, L.stored_entries, L.total_rows, sms))
            launch(std::integral_constant<int, few_blocks(K)>{}, std::integral_constant<int, FEW_AHEAD>{});
        else
            launch(std::integral_constant<int, pass_blocks(K)>{}, std::integral_constant<int, AHEAD>{});
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

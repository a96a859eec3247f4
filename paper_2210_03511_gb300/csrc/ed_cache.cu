// Stored structure of H for repeated H.x (the Lanczos loop applies one H
// tens to hundreds of times).
//
// The matrix-free kernel (ed_apply_impl.cuh) repeats, for every gather, the
// representative search of Alg. "Sublattice coding algorithm for finding the
// representative" and the Limits + binary search of section "Distributed and
// hybrid memory parallelization".  On sectors whose basis exceeds L2 both the
// Limits entry and x_j are random DRAM accesses.  Here both searches run
// once: the row walk records, for every row i and every gather of the pull form
// y_i = sum_j conj(H_ji) x_j, the column j and a one-byte code of its
// coefficient conj(h) chi(g_tau) sqrt(|Stab tau~|) (the row factor
// 1/sqrt(|Stab sigma_i|) and the Ising diagonal are kept per row).  H.x then
// streams this structure and gathers x (ed_cache_pass.cu).
//
// Column segments.  x is cut into segments of 2^seg_bits elements (chosen so
// one segment of the vector type fits comfortably in L2); the entries of each
// row are stored per segment, and H.x runs one pass per segment, so every
// pass gathers from an L2-resident slice of x instead of from all of HBM.
//
// Layout.  Rows form slices of 32 (one warp of the pass):
//   counts[b][row]  (u8)  entries of row `row` in segment b
//   boff[b][slice]  (u32) first entry of the slice's segment-b entries, relative
//                         to its chunk's entries
//   ent[chunk][...] (u32) (code << off_bits) | (j - b 2^seg_bits); inside a slice
//                         entry k of all rows that have one side by side, then
//                         entry k + 1; of a row in flip order
//   diag[row]       (f64) Ising part of row `row`
// The coefficient of code c is ctab[c] (built once per Hamiltonian from the
// codes that occur: distinct (h, chi(g), |Stab tau~|) combinations; real ones
// count up from 0, the others down from the largest code).
//
// Build.  Rows are taken in chunks: one search pass writes every entry of the
// chunk as (column, coefficient key) to scratch (in one word of 32 bits where both
// fit) and counts entries per row and
// segment; the slices' offsets are scanned, the chunk's entries allocated and
// packed.  Searching costs far more than the 16 bytes of scratch traffic per
// entry, so one search and a pack (36-site kagome sector, 4.7 10^9 entries: 159
// and 30 ms) replace the two searches (count, then fill) that a layout without
// scratch needs.
#include <math.h>

#include <algorithm>
#include <vector>

#include "ed_cache.cuh"

namespace ed {

namespace {

constexpr int CMAXNB = 128;   // column segments at most

struct CacheSearch {
    HxArgs a;                      // basis and terms (x, y unused)
    int seg_bits, nb;
    int64_t r0, r1, R;             // rows of the chunk, its scratch stride
    void* raw;                     // [n_flip][R] (column, key) of the row's k-th entry: uint2, or
    int key_shift;                 // one word, key << key_shift | column, when key_shift > 0
    uint8_t* rowtot;               // [R] entries of the row
    uint8_t* counts;               // [nb][Dpad] entries of the row per segment
    int64_t Dpad;
    double* diag;                  // [D]
    const uint16_t* hmap;          // [n_flip][8] h-value id by the spins at (a, c0, c1)
    const uint16_t* chi_id;        // [G] id of the exact value chi(g)
    uint32_t n_chi, Gp1;           // code key = (h id * n_chi + chi id) * (G+1) + |Stab tau~|
    uint64_t dmask;                // bits of one site's state: 1 (spin-1/2) or 2^b - 1 (SU(N) colours)
    double diag_off;               // Ising part per pair class: jhs(1) (diag_off n_pairs - n_acting): 1/2 spin, 1 SU(N)
    uint32_t* seen;                // bit set of keys that occur
    unsigned long long* counters;  // [0] entries, [1] incompatible images, [2] missing, [3] overflow
};

// The search over one chunk of rows, one thread per row.  The row walk
// (activity mask, representative, index search) is that of hx_body.
template <typename W, bool CH, int NS>
__global__ void __launch_bounds__(BLOCK, hx_min_blocks(sizeof(W), 1, 0)) cache_search_kernel(CacheSearch c) {
    extern __shared__ __align__(16) uint8_t smem[];
    const HxArgs& a = c.a;
    constexpr bool generic = !(NS >= 2 && NS <= 4);
    const HxPlan plan = hx_plan(a.dt, 0, generic, a.blocks, a.n_flip, a.n_jc, a.S);
    const SmemLayout lay = plan.lay;
    const TabView<CH> t = stage_sections<CH>(a.dt, smem, 0, plan.mask);
    stage_blob(smem + lay.flip, (const uint8_t*)a.flips, (size_t)a.n_flip * sizeof(FlipTerm));
    stage_blob(smem + lay.jhs, (const uint8_t*)a.jhs, (size_t)a.n_jc * (a.dt.G + 1) * 8);
    uint16_t* pab = (uint16_t*)(smem + lay.pab);
    uint32_t* cmask = (uint32_t*)(smem + lay.cmask);
    for (int i = threadIdx.x; i < a.n_jc * MAXW; i += blockDim.x) cmask[i] = 0u;
    __syncthreads();
    for (int i = threadIdx.x; i < a.n_flip; i += blockDim.x) {
        const FlipTerm& f = ((const FlipTerm*)(smem + lay.flip))[i];
        pab[i] = (uint16_t)((uint8_t)f.pa | ((uint16_t)(uint8_t)f.pb << 8));
        atomicOr(&cmask[a.jcls[i] * MAXW + (i >> 5)], 1u << (i & 31));
    }
    const uint32_t* dir_base = a.dir_base;
    const uint8_t* dir_q = a.dir_q;
    if (plan.dir) {
        uint32_t* db = (uint32_t*)(smem + lay.dir);
        uint8_t* dq = (uint8_t*)(db + a.S + 1);
        for (int i = threadIdx.x; i <= a.S; i += blockDim.x) db[i] = a.dir_base[i];
        for (int i = threadIdx.x; i < a.S; i += blockDim.x) dq[i] = a.dir_q[i];
        dir_base = db;
        dir_q = dq;
    }
    __syncthreads();
    const FlipTerm* flips = (const FlipTerm*)(smem + lay.flip);
    const double* jhs = (const double*)(smem + lay.jhs);
    const W* __restrict__ reps = (const W*)a.reps;
    const int64_t D = a.D;
    const int G1 = a.dt.G + 1;
    const int nw = (a.n_flip + 31) >> 5;
    unsigned long long n_gather = 0, n_skip = 0, n_miss = 0;
    uint8_t cnt[CMAXNB];
    for (int64_t row = c.r0 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; row < c.r1;
         row += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = row - c.r0;
        if (row >= D) {  // the last slice's empty lanes
            c.rowtot[r] = 0;
            for (int b = 0; b < c.nb; ++b) c.counts[(int64_t)b * c.Dpad + row] = 0;
            continue;
        }
        for (int b = 0; b < c.nb; ++b) cnt[b] = 0;
        const W s = reps[row];
        uint32_t mask[MAXW];
#pragma unroll
        for (int w = 0; w < MAXW; ++w) mask[w] = 0u;
#pragma unroll
        for (int w = 0; w < MAXW; ++w) {
            if (w < nw) {
                const int tn = min(32, a.n_flip - 32 * w);
                uint32_t mw = 0u;
                for (int bb = 0; bb < tn; ++bb) {
                    // a term acts iff the two sites' states differ (spins, or packed colours)
                    const uint32_t e = pab[32 * w + bb];
                    mw |= (uint32_t)((((s >> (e & 0xFFu)) ^ (s >> (e >> 8))) & (W)c.dmask) != 0) << bb;
                }
                mask[w] = mw;
            }
        }
        // Ising part, as in hx_body
        double diag = 0.0;
        for (int cc = 0; cc < a.n_jc; ++cc) {
            int nact = 0, ntot = 0;
#pragma unroll
            for (int w = 0; w < MAXW; ++w) {
                if (w < nw) {
                    const uint32_t cm = cmask[cc * MAXW + w];
                    nact += __popc(mask[w] & cm);
                    ntot += __popc(cm);
                }
            }
            diag += jhs[cc * G1 + 1] * (c.diag_off * (double)ntot - (double)nact);
        }
        c.diag[row] = diag;
        uint32_t k = 0;
#pragma unroll
        for (int w = 0; w < MAXW; ++w) {
            if (w >= nw) continue;
            uint32_t mw = mask[w];
            while (mw) {
                const int tt = 32 * w + ctz32(mw);
                mw &= mw - 1u;
                const uint32_t e = pab[tt];
                // exchange the two sites' states: flip both spins, or swap two packed colours
                const W dd = ((s >> (e & 0xFFu)) ^ (s >> (e >> 8))) & (W)c.dmask;
                const W tau = s ^ ((dd << (e & 0xFFu)) | (dd << (e >> 8)));
                W rp;
                int g, nst;
                bool cp;
                rep_of<W, CH, NS>(tau, t, rp, g, nst, cp);
                if (!cp) {
                    ++n_skip;
                    continue;
                }
                const int64_t jx = find_index<W>(rp, reps, dir_base, dir_q, a.limits, a.L);
                if (jx < 0) {
                    ++n_miss;
                    continue;
                }
                const FlipTerm& ft = flips[tt];
                uint32_t hb = (uint32_t)((s >> ft.pa) & 1);
                if (ft.pc0 >= 0) hb |= (uint32_t)((s >> ft.pc0) & 1) << 1;
                if (ft.pc1 >= 0) hb |= (uint32_t)((s >> ft.pc1) & 1) << 2;
                const uint32_t key = ((uint32_t)__ldg(c.hmap + tt * 8 + hb) * c.n_chi + __ldg(c.chi_id + g)) * c.Gp1 +
                                     (uint32_t)nst;
                ++cnt[(uint64_t)jx >> c.seg_bits];
                const uint32_t bit = 1u << (key & 31);
                if (!(c.seen[key >> 5] & bit)) atomicOr(&c.seen[key >> 5], bit);
                if (sizeof(W) == 4 && c.key_shift)
                    ((uint32_t*)c.raw)[(int64_t)k * c.R + r] = key << c.key_shift | (uint32_t)jx;
                else ((uint2*)c.raw)[(int64_t)k * c.R + r] = make_uint2((uint32_t)jx, key);
                ++k;
            }
        }
        n_gather += k;
        c.rowtot[r] = (uint8_t)k;
        for (int b = 0; b < c.nb; ++b) c.counts[(int64_t)b * c.Dpad + row] = cnt[b];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        n_gather += __shfl_xor_sync(0xffffffffu, n_gather, o);
        n_skip += __shfl_xor_sync(0xffffffffu, n_skip, o);
        n_miss += __shfl_xor_sync(0xffffffffu, n_miss, o);
    }
    if ((threadIdx.x & 31) == 0) {
        if (n_gather) atomicAdd(c.counters + 0, n_gather);
        if (n_skip) atomicAdd(c.counters + 1, n_skip);
        if (n_miss) atomicAdd(c.counters + 2, n_miss);
    }
}

// Entries of each slice of the chunk: tot[b][i], i < nsl, of slice s0 + i.
__global__ void slice_totals(const uint8_t* counts, int64_t Dpad, int64_t s0, int64_t nsl, int nb, uint32_t* tot) {
    const int64_t n = nsl * nb;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const uint4* p = (const uint4*)(counts + (i / nsl) * Dpad + (s0 + i % nsl) * NSLICE);  // 32 bytes, 16-aligned
        uint32_t acc = 0;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const uint4 v = p[q];
            acc = __vsadu4(v.x, 0u) + __vsadu4(v.y, 0u) + __vsadu4(v.z, 0u) + __vsadu4(v.w, 0u) + acc;
        }
        tot[i] = acc;
    }
}

// boff[b][s0 + i] = abs[b][i] (entries of one chunk, segment after segment).
__global__ void slice_offsets(const uint64_t* abs_off, int64_t nsl, int nb, int64_t s0, int64_t ns, uint32_t* boff) {
    const int64_t n = nsl * nb;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        boff[(i / nsl) * ns + s0 + i % nsl] = (uint32_t)abs_off[i];
}

struct CachePack {
    int seg_bits, nb, off_bits;
    int64_t r0, r1, R, Dpad, ns;
    const void* raw;               // [n_flip][R], as CacheSearch
    int key_shift;
    const uint8_t* rowtot;         // [R]
    const uint8_t* counts;         // [nb][Dpad]
    const uint32_t* boff;          // [nb][ns]
    const uint8_t* code;           // key -> code
    uint32_t* ent;                 // the chunk's entries
    unsigned long long* counters;  // [3] overflow
};

// Entries of the chunk from scratch into their places, one warp per slice, one
// lane per row.  Before entry k of lane l lie min(c_i, k + 1) entries of the
// lanes i < l and min(c_i, k) of the others (c_i: the lanes' counts in the
// segment, four to a word).  With one segment all lanes are at the same k and a
// ballot gives the place.
template <bool WORD, bool ONE>  // entries of one word; one segment
__global__ void __launch_bounds__(BLOCK) cache_pack_kernel(CachePack a) {
    auto load = [&](int64_t at) -> uint2 {
        if constexpr (WORD) {
            const uint32_t w = __ldg((const uint32_t*)a.raw + at);
            return make_uint2(w & ((1u << a.key_shift) - 1u), w >> a.key_shift);
        } else {
            return __ldg((const uint2*)a.raw + at);
        }
    };
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const uint32_t segmask = (uint32_t)(((uint64_t)1 << a.seg_bits) - 1);
    uint32_t before[NSLICE / 4];   // byte i: 1 for the lanes before this one
#pragma unroll
    for (int q = 0; q < NSLICE / 4; ++q) {
        const int n = min(4, max(0, lane - 4 * q));
        before[q] = n == 4 ? 0x01010101u : (0x01010101u & ((1u << (8 * n)) - 1u));
    }
    uint8_t kb[CMAXNB];
    unsigned long long over = 0;
    const int64_t warps = (int64_t)gridDim.x * (BLOCK / 32);
    for (int64_t sl = a.r0 / NSLICE + (int64_t)blockIdx.x * (BLOCK / 32) + (threadIdx.x >> 5);
         sl < a.r1 / NSLICE; sl += warps) {
        const int64_t row = sl * NSLICE + lane, r = row - a.r0;
        const int n = a.rowtot[r];
        if constexpr (ONE) {
            uint32_t* out = a.ent + a.boff[sl];
            const int m = __reduce_max_sync(0xffffffffu, n);
            constexpr int U = 4;  // entries in flight: a slice is one chain of entry and code loads (0.01 ms of 0.3)
            for (int k = 0; k < m; k += U) {
                uint2 e[U];
                uint32_t w[U];
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (n > k + u) e[u] = load((int64_t)(k + u) * a.R + r);
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (n > k + u) w[u] = ((uint32_t)__ldg(a.code + e[u].y) << a.off_bits) | e[u].x;
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const unsigned has = __ballot_sync(0xffffffffu, n > k + u);
                    if (n > k + u) out[__popc(has & lt)] = w[u];
                    out += __popc(has);
                }
            }
        } else {
            for (int b = 0; b < a.nb; ++b) kb[b] = 0;
            for (int i = 0; i < n; ++i) {
                const uint2 e = load((int64_t)i * a.R + r);
                const int b = (int)(e.x >> a.seg_bits);
                const uint32_t k = kb[b];
                kb[b] = (uint8_t)(k + 1);
                const uint4* cw = (const uint4*)(a.counts + (int64_t)b * a.Dpad + sl * NSLICE);
                const uint4 lo = cw[0], hi = cw[1];
                const uint32_t c[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
                const uint32_t kk = k * 0x01010101u;
                uint32_t o = 0;
#pragma unroll
                for (int q = 0; q < 8; ++q) o += __vsadu4(__vminu4(c[q], kk + before[q]), 0u);
                if (k >= ((const uint8_t*)cw)[lane]) {
                    ++over;
                    continue;
                }
                a.ent[(int64_t)a.boff[(int64_t)b * a.ns + sl] + o] =
                    ((uint32_t)__ldg(a.code + e.y) << a.off_bits) | (e.x & segmask);
            }
        }
    }
    if (over) atomicAdd(a.counters + 3, over);
}

template <typename W, bool CH, int NS>
static ed_status launch_search(const CacheSearch& c, size_t smem, cudaStream_t s) {
    auto k = cache_search_kernel<W, CH, NS>;
    static int cfg_smem = -1, cfg_per_sm = 0, cfg_sms = 0;
    const ed_status st = occupancy(k, smem, cfg_smem, cfg_per_sm, cfg_sms);
    if (st != ED_OK) return st;
    const int per_sm = std::min(cfg_per_sm, std::max(1, c.a.blocks));
    int64_t grid = std::min<int64_t>((int64_t)cfg_sms * per_sm, (c.r1 - c.r0 + BLOCK - 1) / BLOCK);
    if (grid < 1) grid = 1;
    k<<<(unsigned)grid, BLOCK, smem, s>>>(c);
    ED_CUDA(cudaGetLastError());
    return ED_OK;
}

static ed_status search_dispatch(const CacheSearch& c, size_t smem, int n_sub, bool ns_ok, bool w8, bool ch,
                                 cudaStream_t s) {
    auto go = [&](auto wtag, auto chtag) -> ed_status {
        using W = decltype(wtag);
        constexpr bool CH = decltype(chtag)::value;
        if (ns_ok) {
            if (n_sub == 2) return launch_search<W, CH, 2>(c, smem, s);
            if (n_sub == 3) return launch_search<W, CH, 3>(c, smem, s);
            if (n_sub == 4) return launch_search<W, CH, 4>(c, smem, s);
        }
        return launch_search<W, CH, 0>(c, smem, s);
    };
    if (w8) return ch ? go(uint64_t{}, std::true_type{}) : go(uint64_t{}, std::false_type{});
    return ch ? go(uint32_t{}, std::true_type{}) : go(uint32_t{}, std::false_type{});
}

// Freed together with the structure.
struct BuildScratch {
    const Alloc* A;
    cudaStream_t s;
    std::vector<std::pair<void*, size_t>> bufs;
    void* get(size_t n) {
        void* p = A->get(n, s);
        if (p) bufs.push_back({p, n});
        return p;
    }
    void clear() {
        cudaStreamSynchronize(s);
        for (auto& b : bufs) A->put(b.first, b.second, s);
        bufs.clear();
    }
    ~BuildScratch() { clear(); }
};

}  // namespace

bool cache_sector_desc(const ed_hamiltonian* h, CacheSector& d) {
    const HCache& c = h->cache;
    if (!c.valid || c.nb != 1) return false;
    const ed_basis* b = h->basis;
    d.counts = (const uint8_t*)c.counts.p;
    d.boff = (const uint32_t*)c.boff.p;
    d.ent = (const uint32_t* const*)c.base.p;
    d.chunk_shift = c.chunk_shift;
    d.diag = (const double*)c.diag.p;
    d.stab = (const uint16_t*)b->stab.p;
    d.ctab = (const uint8_t*)c.ctab.p;
    d.sq = b->dt.blob + b->dt.off_sqrt;
    d.sqf = b->dt.blob + b->dt.off_sqrtf;
    d.D = b->dim;
    d.ns = c.ns;
    d.slice0 = 0;
    d.G1 = b->ht.G + 1;
    d.off_bits = (uint32_t)c.off_bits;
    return true;
}

void cache_free(ed_hamiltonian* h) {
    HCache& c = h->cache;
    const Alloc& A = h->basis->alloc;
    for (DevBuf* d : {&c.counts, &c.boff, &c.diag, &c.ctab, &c.base}) A.put(d->p, d->bytes, 0);
    for (DevBuf& d : c.ent) A.put(d.p, d.bytes, 0);
    c = HCache{};
}

// Default column segment: 128 MB of the vector type, at most 2^24 elements.
static int default_seg_bits(ed_dtype dtype) {
    const int sx = dtype == ED_F32 ? 4 : dtype == ED_C128 ? 16 : 8;
    const uint64_t elems = (uint64_t)(128u << 20) / (uint64_t)sx;
    int bits = 0;
    while (((uint64_t)2 << bits) <= elems) ++bits;
    return std::min(bits, 24);
}

namespace {

// Coefficient keys of a Hamiltonian (ids of the distinct values of h and chi)
// and the codes of the keys that have occurred.
struct Codes {
    std::vector<std::pair<double, double>> hval, cval;
    std::vector<uint16_t> hmap, chi_id;
    uint64_t G1 = 0, n_keys = 0;
    std::vector<uint32_t> seen;      // keys that have a code
    std::vector<uint8_t> code;
    std::vector<double> d1;          // [NCODE] coefficients of real Hamiltonians, FP64
    std::vector<double> d2;          // [NCODE][2] coefficients, FP64
    std::vector<float> f2;           // and FP32
    int cap = NCODE, n_re = 0, n_im = 0;

    void init(const ed_hamiltonian* h) {
        const HostTables& t = h->basis->ht;
        hmap.resize((size_t)std::max(h->n_flip, 1) * 8);
        for (int f = 0; f < h->n_flip; ++f) {
            const FlipTerm& ft = h->flips[f];
            for (int hb = 0; hb < 8; ++hb) {
                double him = 0.0;
                if (ft.pc0 >= 0) him += ft.k0 * ((hb & 2) ? 0.5 : -0.5);
                if (ft.pc1 >= 0) him += ft.k1 * ((hb & 4) ? 0.5 : -0.5);
                if (hb & 1) him = -him;
                const std::pair<double, double> v{ft.jhalf, him};
                const size_t id = std::find(hval.begin(), hval.end(), v) - hval.begin();
                if (id == hval.size()) hval.push_back(v);
                hmap[(size_t)f * 8 + hb] = (uint16_t)id;
            }
        }
        chi_id.resize(t.G);
        for (int g = 0; g < t.G; ++g) {
            const std::pair<double, double> v{t.chi[2 * g], t.chi[2 * g + 1]};
            const size_t id = std::find(cval.begin(), cval.end(), v) - cval.begin();
            if (id == cval.size()) cval.push_back(v);
            chi_id[g] = (uint16_t)id;
        }
        G1 = (uint64_t)(t.G + 1);
        n_keys = (uint64_t)hval.size() * cval.size() * G1;
    }
    void reset(int capacity) {
        cap = capacity;
        n_re = n_im = 0;
        seen.assign((n_keys + 31) / 32, 0u);
        code.assign((size_t)n_keys, 0);
        d1.assign(NCODE, 0.0);
        d2.assign(2 * NCODE, 0.0);
        f2.assign(2 * NCODE, 0.f);
    }
    // Give the keys of `now` that have none a code; false if they run out.
    bool add(const std::vector<uint32_t>& now, bool& grew) {
        grew = false;
        for (size_t w = 0; w < now.size(); ++w) {
            for (uint32_t m = now[w] & ~seen[w]; m; m &= m - 1) {
                const uint64_t key = w * 32 + (uint64_t)__builtin_ctz(m);
                if (n_re + n_im >= cap) return false;
                const int nst = (int)(key % G1);
                const uint64_t hc = key / G1;
                const auto& cv = cval[hc % cval.size()];
                const auto& hv = hval[hc / cval.size()];
                // conj(h) chi sqrt(n), h = jhalf + i him: the matrix-free kernel's coefficient of
                // this gather in each precision (real FP32: its real part; real FP64: jhalf sqrt(n)
                // with the sign of chi, which may differ from -1 and 1 by rounding)
                const double sq = sqrt((double)nst);
                const double re = (hv.first * cv.first + hv.second * cv.second) * sq;
                const double im = (hv.first * cv.second - hv.second * cv.first) * sq;
                const int id = im == 0.0 ? n_re++ : cap - 1 - n_im++;
                d1[id] = cv.first < 0.0 ? -(hv.first * sq) : hv.first * sq;
                d2[2 * id] = re;
                d2[2 * id + 1] = im;
                const float jf = (float)hv.first, hf = (float)hv.second, cx = (float)cv.first, cy = (float)cv.second;
                f2[2 * id] = (jf * cx + hf * cy) * (float)sq;
                f2[2 * id + 1] = (jf * cy - hf * cx) * (float)sq;
                code[key] = (uint8_t)id;
                seen[w] |= 1u << (key & 31);
                grew = true;
            }
        }
        return true;
    }
};

// Scratch of these sizes comes from the device's pool: an allocation of more than 1 MB takes
// 0.13 ms to map and free, as much as the search of a small sector (kagome18 without rotations,
// 8,110 rows: 0.44 -> 0.36 ms, triangular24 0.75 -> 0.65); smaller ones are cheap, and large
// sectors do not notice.
constexpr size_t POOLED_MIN = (size_t)1 << 20, POOLED_MAX = (size_t)16 << 20;

// Builds the structure into h->cache, its chunks' scratch limited to about
// `scratch` bytes.  On an error the parts stay in h->cache for cache_free;
// smaller: the scratch of another try, where the memory had no room for this one's
// and less scratch may make some (0: it may not).
static ed_status build_once(ed_hamiltonian* h, int bits, size_t max_bytes, size_t scratch, Codes& codes,
                            cudaStream_t s, size_t& smaller) {
    const ed_basis* b = h->basis;
    const HostTables& t = b->ht;
    const Alloc& A = b->alloc;
    const int64_t D = b->dim;
    const int nb = (int)(((uint64_t)D + ((uint64_t)1 << bits) - 1) >> bits);
    HCache& c = h->cache;
    smaller = 0;
    BuildScratch sc{&A, s, {}};
    c.seg_bits = bits;
    c.nb = nb;
    c.ns = (D + NSLICE - 1) / NSLICE;
    c.off_bits = std::max(24, bits);
    const int64_t ns = c.ns, Dpad = ns * NSLICE;
    // chunk: a power of two of rows whose raw entries fit the scratch; the only chunk: all rows.
    // Column and key in one word where they fit (32-bit states; sectors of 64-bit states are large,
    // and the choice cost their search 4 %, square36 219 -> 229 ms): half the scratch, which in a
    // small sector then stays below what an allocation of its own takes (chain16, 12,870 rows:
    // 0.30 -> 0.16 ms), and half its traffic (square32 7.0 -> 5.8 ms)
    auto width = [](uint64_t n) {
        int k = 1;
        while (((uint64_t)1 << k) < n) ++k;
        return k;
    };
    const int col_bits = width((uint64_t)D);
    const int key_shift = b->word == 4 && col_bits + width(codes.n_keys) <= 32 ? col_bits : 0;
    const size_t raw_bytes = key_shift ? sizeof(uint32_t) : sizeof(uint2);
    const int64_t row_bytes = (int64_t)raw_bytes * std::max(h->n_flip, 1) + 1;
    int64_t chunk = NSLICE;
    while (chunk * 2 * row_bytes <= (int64_t)scratch && chunk < (1 << 22) && chunk < Dpad) chunk *= 2;
    c.chunk_shift = 0;
    while (((int64_t)NSLICE << c.chunk_shift) < chunk) ++c.chunk_shift;
    const int64_t n_chunks = (Dpad + chunk - 1) / chunk;
    const int64_t R = std::min(chunk, Dpad), Rsl = R / NSLICE;
    codes.reset(1 << (32 - c.off_bits));
    auto get = [&](DevBuf& d, size_t bytes) {
        d.bytes = bytes;
        d.p = A.get(bytes, s);
        return d.p != nullptr;
    };
    const bool ok = get(c.counts, (size_t)nb * Dpad) && get(c.diag, (size_t)D * 8) && get(c.boff, (size_t)nb * ns * 4) &&
              get(c.ctab, CT_BYTES) && get(c.base, (size_t)n_chunks * 8);
    const size_t seen_bytes = codes.seen.size() * 4;
    // one allocation for the scratch: allocations cost more than the build of a small sector
    size_t at = 0;
    auto part = [&](size_t n) {
        const size_t o = at;
        at += (n + 255) & ~(size_t)255;
        return o;
    };
    const size_t o_hmap = part(codes.hmap.size() * 2), o_chi = part(codes.chi_id.size() * 2), o_cnt = part(64),
                 o_seen = part(seen_bytes), o_code = part((size_t)codes.n_keys),
                 o_raw = part((size_t)std::max(h->n_flip, 1) * R * raw_bytes), o_tot1 = part((size_t)R),
                 o_tot = part((size_t)nb * Rsl * 4), o_abs = part(((size_t)nb * Rsl + 1) * 8),
                 o_tiles = part(scan_scratch_words((uint64_t)nb * Rsl) * 8);
    struct Pooled {
        void* p;
        cudaStream_t s;
        ~Pooled() {
            if (p) StreamPool::put(p, s);
        }
    } pooled{at > POOLED_MIN && at <= POOLED_MAX ? h->scratch.get(A, b->device, at, s) : nullptr, s};
    uint8_t* scr = (uint8_t*)(pooled.p ? pooled.p : sc.get(at));
    uint16_t* d_hmap = (uint16_t*)(scr + o_hmap);
    uint16_t* d_chi = (uint16_t*)(scr + o_chi);
    unsigned long long* d_cnt = (unsigned long long*)(scr + o_cnt);
    uint32_t* d_seen = (uint32_t*)(scr + o_seen);
    uint8_t* d_code = scr + o_code;
    void* d_raw = scr + o_raw;
    uint8_t* d_rowtot = scr + o_tot1;
    uint32_t* d_tot = (uint32_t*)(scr + o_tot);
    uint64_t* d_abs = (uint64_t*)(scr + o_abs);
    uint64_t* d_tiles = (uint64_t*)(scr + o_tiles);
    if (!ok || !scr) {
        if (ok && chunk > NSLICE) smaller = std::min(scratch, at) / 32;
        return fail(ED_ERR_NOMEM, "structure build: allocation failed");
    }
    ED_CUDA(cudaMemcpyAsync(d_hmap, codes.hmap.data(), codes.hmap.size() * 2, cudaMemcpyHostToDevice, s));
    ED_CUDA(cudaMemcpyAsync(d_chi, codes.chi_id.data(), codes.chi_id.size() * 2, cudaMemcpyHostToDevice, s));
    ED_CUDA(cudaMemsetAsync(d_cnt, 0, o_code - o_cnt, s));  // counters and seen bits
    ED_CUDA(cudaDeviceGetAttribute(&c.sms, cudaDevAttrMultiProcessorCount, b->device));
    CacheSearch q{};
    q.a = make_args(h);
    q.seg_bits = bits;
    q.nb = nb;
    q.R = R;
    q.raw = d_raw;
    q.key_shift = key_shift;
    q.rowtot = d_rowtot;
    q.counts = (uint8_t*)c.counts.p;
    q.Dpad = Dpad;
    q.diag = (double*)c.diag.p;
    q.hmap = d_hmap;
    q.chi_id = d_chi;
    q.n_chi = (uint32_t)codes.cval.size();
    q.Gp1 = (uint32_t)codes.G1;
    q.dmask = h->sun ? (((uint64_t)1 << b->sun_b) - 1) : 1ull;
    q.diag_off = h->sun ? 1.0 : 0.5;
    q.seen = d_seen;
    q.counters = d_cnt;
    const bool w8 = b->word == 8, ch = b->dt.chunk_lo > 0, ns_ok = b->dt.dl_stride == 4;
    const bool generic = !(ns_ok && t.n_sub >= 2 && t.n_sub <= 4);
    q.a.blocks = hx_min_blocks(b->word, 1, 0);
    const size_t smem = hx_plan(b->dt, 0, generic, q.a.blocks, h->n_flip, h->n_jc, 1 << t.m).lay.total;
    size_t need = c.counts.bytes + c.diag.bytes + c.boff.bytes + c.ctab.bytes + c.base.bytes;
    std::vector<uint64_t> seg_total(nb, 0), edge(nb + 1);
    std::vector<uint32_t> now(codes.seen.size());
    std::vector<uint64_t> base((size_t)n_chunks, 0);
    unsigned long long cnt[4] = {};
    for (int64_t k = 0; k < n_chunks; ++k) {
        q.r0 = k * chunk;
        q.r1 = std::min<int64_t>(q.r0 + chunk, Dpad);
        ed_status st = search_dispatch(q, smem, t.n_sub, ns_ok, w8, ch, s);
        if (st != ED_OK) return st;
        const int64_t nsl = (q.r1 - q.r0) / NSLICE, n = nsl * nb;
        const unsigned g = (unsigned)std::min<int64_t>((n + 255) / 256, (int64_t)c.sms * 16);
        slice_totals<<<g, 256, 0, s>>>(q.counts, Dpad, q.r0 / NSLICE, nsl, nb, d_tot);
        ED_CUDA(cudaGetLastError());
        st = exclusive_scan_u32(d_tot, (uint64_t)n, d_abs, d_tiles, d_abs + n, s);
        if (st != ED_OK) return st;
        slice_offsets<<<g, 256, 0, s>>>(d_abs, nsl, nb, q.r0 / NSLICE, ns, (uint32_t*)c.boff.p);
        ED_CUDA(cudaGetLastError());
        // the first entry of every segment in the chunk, and the chunk's total
        ED_CUDA(cudaMemcpy2DAsync(edge.data(), 8, d_abs, (size_t)nsl * 8, 8, nb, cudaMemcpyDeviceToHost, s));
        ED_CUDA(cudaMemcpyAsync(&edge[nb], d_abs + n, 8, cudaMemcpyDeviceToHost, s));
        ED_CUDA(cudaMemcpyAsync(now.data(), d_seen, seen_bytes, cudaMemcpyDeviceToHost, s));
        ED_CUDA(cudaMemcpyAsync(cnt, d_cnt, 32, cudaMemcpyDeviceToHost, s));
        ED_CUDA(cudaStreamSynchronize(s));
        if (cnt[2]) return fail(ED_ERR_INDEX_NOT_FOUND, "%llu representatives missing from the basis", cnt[2]);
        bool grew = false;
        if (!codes.add(now, grew))
            return fail(ED_ERR_TABLE_TOO_LARGE, "more than %d distinct coefficients beside %d bits of column offset",
                        codes.cap, c.off_bits);
        if (grew || k == 0)
            ED_CUDA(cudaMemcpyAsync(d_code, codes.code.data(), codes.code.size(), cudaMemcpyHostToDevice, s));
        // At most 2^32 - 2 entries to a segment: not for the offsets' sake, which count from the
        // chunk's first entry, but a structure that was refused stays refused
        for (int i = 0; i < nb; ++i) {
            seg_total[i] += edge[i + 1] - edge[i];
            if (seg_total[i] >= 0xFFFFFFFFull)
                return fail(ED_ERR_ARG, "segment %d holds 2^32 or more entries; use smaller segments", i);
        }
        c.n_ent += edge[nb];
        DevBuf e;
        e.bytes = std::max<size_t>((size_t)edge[nb] * 4, 16);
        need += e.bytes;
        if (need > max_bytes)
            return fail(ED_ERR_NOMEM, "the stored structure needs %zu bytes or more, over the limit of %zu", need,
                        max_bytes);
        e.p = A.get(e.bytes, s);
        if (!e.p) {
            if (chunk > NSLICE && at > need / 32) smaller = std::min(scratch, at) / 32;
            return fail(ED_ERR_NOMEM, "structure entries (%zu bytes)", e.bytes);
        }
        c.ent.push_back(e);
        base[k] = (uint64_t)(uintptr_t)e.p;
        CachePack pk{};
        pk.seg_bits = bits;
        pk.nb = nb;
        pk.off_bits = c.off_bits;
        pk.r0 = q.r0;
        pk.r1 = q.r1;
        pk.R = R;
        pk.Dpad = Dpad;
        pk.ns = ns;
        pk.raw = d_raw;
        pk.key_shift = key_shift;
        pk.rowtot = d_rowtot;
        pk.counts = q.counts;
        pk.boff = (const uint32_t*)c.boff.p;
        pk.code = d_code;
        pk.ent = (uint32_t*)e.p;
        pk.counters = d_cnt;
        const unsigned pg = (unsigned)std::min<int64_t>((nsl + 7) / 8, (int64_t)c.sms * 8);
        auto pack = key_shift ? (nb == 1 ? cache_pack_kernel<true, true> : cache_pack_kernel<true, false>)
                              : (nb == 1 ? cache_pack_kernel<false, true> : cache_pack_kernel<false, false>);
        pack<<<pg, BLOCK, 0, s>>>(pk);
        ED_CUDA(cudaGetLastError());
    }
    // coefficient tables; axis-aligned ones: (c, c) for a real c, (-c, c) for i c
    const int n_code = codes.n_re + codes.n_im;
    c.n_code = n_code;
    c.n_re = codes.cap - codes.n_im;
    std::vector<double> a_d2(2 * NCODE, 0.0);
    std::vector<float> a_f2(2 * NCODE, 0.f);
    c.axis_d = c.axis_f = true;
    for (int k = 0; k < codes.cap; ++k) {
        const bool re = k < c.n_re;
        const double dr = codes.d2[2 * k], di = codes.d2[2 * k + 1];
        const float fr = codes.f2[2 * k], fi = codes.f2[2 * k + 1];
        c.axis_d = c.axis_d && (re || dr == 0.0);
        c.axis_f = c.axis_f && (re ? fi == 0.f : fr == 0.f);
        a_d2[2 * k] = re ? dr : -di;
        a_d2[2 * k + 1] = re ? dr : di;
        a_f2[2 * k] = re ? fr : -fi;
        a_f2[2 * k + 1] = re ? fr : fi;
    }
    uint8_t* ct = (uint8_t*)c.ctab.p;
    ED_CUDA(cudaMemcpyAsync(ct + CT_D2, codes.d2.data(), NCODE * 16, cudaMemcpyHostToDevice, s));
    ED_CUDA(cudaMemcpyAsync(ct + CT_D1, codes.d1.data(), NCODE * 8, cudaMemcpyHostToDevice, s));
    ED_CUDA(cudaMemcpyAsync(ct + CT_F2, codes.f2.data(), NCODE * 8, cudaMemcpyHostToDevice, s));
    ED_CUDA(cudaMemcpyAsync(ct + CT_AXD, a_d2.data(), NCODE * 16, cudaMemcpyHostToDevice, s));
    ED_CUDA(cudaMemcpyAsync(ct + CT_AXF, a_f2.data(), NCODE * 8, cudaMemcpyHostToDevice, s));
    ED_CUDA(cudaMemcpyAsync(c.base.p, base.data(), (size_t)n_chunks * 8, cudaMemcpyHostToDevice, s));
    ED_CUDA(cudaMemcpyAsync(cnt, d_cnt, 32, cudaMemcpyDeviceToHost, s));
    ED_CUDA(cudaStreamSynchronize(s));
    if (cnt[0] != c.n_ent || cnt[3] != 0)
        return fail(ED_ERR_INDEX_NOT_FOUND, "structure pack mismatch (%llu entries, %llu overflow)", cnt[0], cnt[3]);
    c.n_skip = cnt[1];
    c.bytes = need;
    c.valid = true;
    return ED_OK;
}

}  // namespace

ed_status cache_build(ed_hamiltonian* h, ed_dtype dtype, int seg_log2, size_t max_bytes, cudaStream_t s) {
    if (h->cache.valid) cache_free(h);
    if (h->n_flip > 255) return fail(ED_ERR_ARG, "the stored structure needs at most 255 flip terms (%d)", h->n_flip);
    const int64_t D = h->basis->dim;
    const int bits = seg_log2 ? seg_log2 : default_seg_bits(dtype);
    if (bits < 5 || bits > 28) return fail(ED_ERR_ARG, "segment bits %d out of range [5,28]", bits);
    const int nb = (int)(((uint64_t)D + ((uint64_t)1 << bits) - 1) >> bits);
    if (nb > CMAXNB) return fail(ED_ERR_ARG, "%d column segments exceed %d; use larger segments", nb, CMAXNB);
    Codes codes;
    codes.init(h);
    if (codes.n_keys > ((uint64_t)1 << 26))
        return fail(ED_ERR_TABLE_TOO_LARGE, "coefficient key space of %llu too large", (unsigned long long)codes.n_keys);
    // about 3 GB of scratch, and less and less where the memory has no room for that beside the
    // structure, until the scratch is not what is in the way (a few per cent of the structure)
    size_t scratch = (size_t)3 << 30;
    ed_status st = build_once(h, bits, max_bytes, scratch, codes, s, scratch);
    while (st == ED_ERR_NOMEM && scratch) {
        cudaStreamSynchronize(s);
        cache_free(h);
        st = build_once(h, bits, max_bytes, scratch, codes, s, scratch);
    }
    if (st != ED_OK) {
        cudaStreamSynchronize(s);  // nothing may still write into what is freed
        cache_free(h);
    }
    return st;
}

ed_status cache_apply(const ed_hamiltonian* h, ed_dtype dt, const void* x, void* y, int nvec, cudaStream_t s,
                      bool diff) {
    const HCache& c = h->cache;
    const ed_basis* b = h->basis;
    CachePass p{};
    p.x = x;
    p.y = y;
    p.ent = (const uint32_t* const*)c.base.p;
    p.chunk_shift = c.chunk_shift;
    p.stab = (const uint16_t*)b->stab.p;
    p.diag = (const double*)c.diag.p;
    p.D = b->dim;
    p.ns = c.ns;
    p.nvec = nvec;
    p.diff = diff;
    p.n_ent = c.n_ent;
    p.n_skip = c.n_skip;
    p.nb = c.nb;
    p.off_bits = (uint32_t)c.off_bits;
    p.n_re = (uint32_t)c.n_re;
    const int K = dt == ED_F64 ? 0 : dt == ED_F32 ? 1 : dt == ED_C128 ? 2 : 3;
    const size_t copy = cache_interleaved_bytes(dt, nvec, b->dim, c.ns, c.sms);
    if (copy) p.xi = h->scratch.get(b->alloc, b->device, copy, s);
    const bool f64 = K == 0 || K == 2;
    // several warps per slice: the general tables
    const bool ax = K >= 2 && !(nvec == 1 && c.lanes > 1) && (f64 ? c.axis_d : c.axis_f);
    const uint8_t* ct = (const uint8_t*)c.ctab.p;
    p.ctab = ct + (ax ? (f64 ? CT_AXD : CT_AXF) : K == 0 ? CT_D1 : K == 2 ? CT_D2 : CT_F2);
    p.isq = b->dt.blob + (f64 ? b->dt.off_sqrt + (size_t)(b->ht.G + 1) * 8 : b->dt.off_sqrtf + (size_t)(b->ht.G + 1) * 4);
    ed_status st = ED_OK;
    for (int k = 0; k < c.nb && st == ED_OK; ++k) {
        p.counts = (const uint8_t*)c.counts.p + (size_t)k * c.ns * NSLICE;
        p.boff = (const uint32_t*)c.boff.p + (size_t)k * c.ns;
        p.xoff = (int64_t)k << c.seg_bits;
        p.mode = c.nb == 1 ? 0 : (k == 0 ? 1 : (k == c.nb - 1 ? 3 : 2));
        p.counters = k == 0 ? (unsigned long long*)h->d_counters.p : nullptr;
        st = launch_cache_pass(p, K, ax, c.lanes, c.sms, s);
    }
    if (p.xi) StreamPool::put(p.xi, s);
    return st;
}

}  // namespace ed

extern "C" ed_status ed_hamiltonian_store(ed_hamiltonian* h, ed_dtype dtype, int32_t seg_log2, size_t max_bytes,
                                          ed_stream stream, size_t* bytes) {
    using namespace ed;
    if (!h) return fail(ED_ERR_ARG, "null argument");
    if ((int)dtype < 0 || (int)dtype > 3) return fail(ED_ERR_ARG, "bad dtype");
    if (seg_log2 != 0 && (seg_log2 < 5 || seg_log2 > 28)) return fail(ED_ERR_ARG, "seg_log2 out of range");
    cudaSetDevice(h->basis->device);
    const ed_status st = cache_build(h, dtype, seg_log2, max_bytes, (cudaStream_t)stream);
    if (bytes) *bytes = st == ED_OK ? h->cache.bytes : 0;
    return st;
}

extern "C" ed_status ed_hamiltonian_store_info(const ed_hamiltonian* h, int64_t* entries, int32_t* segments,
                                               int32_t* codes, size_t* bytes) {
    using namespace ed;
    if (!h) return fail(ED_ERR_ARG, "null argument");
    const HCache& c = h->cache;
    if (entries) *entries = c.valid ? (int64_t)c.n_ent : 0;
    if (segments) *segments = c.valid ? c.nb : 0;
    if (codes) *codes = c.valid ? c.n_code : 0;
    if (bytes) *bytes = c.valid ? c.bytes : 0;
    return ED_OK;
}

extern "C" void ed_hamiltonian_store_free(ed_hamiltonian* h) {
    if (!h) return;
    cudaSetDevice(h->basis->device);
    ed::cache_free(h);
}

// Segment-size autotuner: a segment of x should stay in L2 while its pass
// gathers from it, but every pass also reads each row's count and updates its
// partial sum, and short rows leave more of a warp idle, so fewer, larger segments
// pay where rows are many (the 40-site square sector and the 36-site kagome sector,
// FP64 and FP32, take 2^24 elements).
extern "C" ed_status ed_hamiltonian_store_set_lanes(ed_hamiltonian* h, int32_t lanes_per_row) {
    using namespace ed;
    if (!h) return fail(ED_ERR_ARG, "null argument");
    if (!h->cache.valid) return fail(ED_ERR_ARG, "no stored structure");
    if (lanes_per_row != 1 && lanes_per_row != 2 && lanes_per_row != 4 && lanes_per_row != 8)
        return fail(ED_ERR_ARG, "lanes per row must be 1, 2, 4 or 8");
    h->cache.lanes = lanes_per_row;
    return ED_OK;
}

extern "C" ed_status ed_hamiltonian_store_schedule(const ed_hamiltonian* h, int32_t* seg_log2,
                                                   int32_t* lanes_per_row) {
    using namespace ed;
    if (!h) return fail(ED_ERR_ARG, "null argument");
    const bool v = h->cache.valid;
    if (seg_log2) *seg_log2 = v ? h->cache.seg_bits : 0;
    if (lanes_per_row) *lanes_per_row = v ? h->cache.lanes : 0;
    return ED_OK;
}

extern "C" ed_status ed_hamiltonian_store_autotune(ed_hamiltonian* h, ed_dtype dtype, size_t max_bytes,
                                                   ed_stream stream, int32_t* seg_log2, size_t* bytes) {
    using namespace ed;
    if (!h) return fail(ED_ERR_ARG, "null argument");
    if ((int)dtype < 0 || (int)dtype > 3) return fail(ED_ERR_ARG, "bad dtype");
    if ((dtype == ED_F64 || dtype == ED_F32) && !h->is_real)
        return fail(ED_ERR_ARG, "complex Hamiltonian or characters need a complex dtype");
    cudaSetDevice(h->basis->device);
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t D = h->basis->dim;
    const int b0 = default_seg_bits(dtype);
    std::vector<int> cands;
    for (int b = b0 - 1; b <= b0 + 1; ++b)
        if (b >= 5 && b <= 26 && (((uint64_t)D + ((uint64_t)1 << b) - 1) >> b) <= (uint64_t)CMAXNB) cands.push_back(b);
    if (cands.empty()) cands.push_back(b0);
    const size_t sx = dtype == ED_F32 ? 4 : dtype == ED_C128 ? 16 : 8;
    const Alloc& A = h->basis->alloc;
    BuildScratch sc{&A, s, {}};
    void* x = sc.get((size_t)D * sx);
    void* y = sc.get((size_t)D * sx);
    if (!x || !y) return fail(ED_ERR_NOMEM, "autotune vectors");
    ED_CUDA(cudaMemsetAsync(x, 0, (size_t)D * sx, s));
    cudaEvent_t e0, e1;
    ED_CUDA(cudaEventCreate(&e0));
    ED_CUDA(cudaEventCreate(&e1));
    struct EFree {
        cudaEvent_t a, b;
        ~EFree() {
            cudaEventDestroy(a);
            cudaEventDestroy(b);
        }
    } ef{e0, e1};
    float best = 1e30f;
    int best_b = 0, best_l = 1;
    ed_status last = ED_OK;
    for (int b : cands) {
        last = cache_build(h, dtype, b, max_bytes, s);
        if (last == ED_ERR_NOMEM || last == ED_ERR_TABLE_TOO_LARGE || (last == ED_ERR_ARG && b != b0)) continue;
        if (last != ED_OK) return last;
        for (int l = 1; l <= 8; l *= 2) {
            h->cache.lanes = l;
            ed_status st = cache_apply(h, dtype, x, y, 1, s);  // warm-up
            if (st != ED_OK) return st;
            ED_CUDA(cudaEventRecord(e0, s));
            for (int r = 0; r < 2 && st == ED_OK; ++r) st = cache_apply(h, dtype, x, y, 1, s);
            if (st != ED_OK) return st;
            ED_CUDA(cudaEventRecord(e1, s));
            ED_CUDA(cudaEventSynchronize(e1));
            float ms = 0.f;
            ED_CUDA(cudaEventElapsedTime(&ms, e0, e1));
            if (ms < best) {
                best = ms;
                best_b = b;
                best_l = l;
            }
        }
    }
    if (!best_b) {
        if (bytes) *bytes = 0;
        return last != ED_OK ? last : fail(ED_ERR_NOMEM, "no segment size fits the limit");
    }
    if (!h->cache.valid || h->cache.seg_bits != best_b) {
        const ed_status st = cache_build(h, dtype, best_b, max_bytes, s);
        if (st != ED_OK) return st;
    }
    h->cache.lanes = best_l;
    if (seg_log2) *seg_log2 = best_b;
    if (bytes) *bytes = h->cache.bytes;
    return ED_OK;
}

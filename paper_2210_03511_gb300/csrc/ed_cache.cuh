// Stored-structure H.x: the arguments of one column segment's pass, shared by
// the structure build (ed_cache.cu) and the pass kernels (ed_cache_pass.cu).
#pragma once

#include "ed_apply_impl.cuh"

namespace ed {

constexpr int NCODE = 256;    // coefficient codes at most (one byte)
constexpr int NSLICE = 32;    // rows of a slice (one warp)

// Byte offsets of the tables in HCache::ctab.  A real FP32 coefficient is the real part of
// the complex one; a real FP64 one has its own table (the character enters as its sign,
// as in the matrix-free kernel, whose bits the real sums keep).
constexpr size_t CT_D2 = 0, CT_F2 = (size_t)NCODE * 16, CT_AXD = (size_t)NCODE * 24, CT_AXF = (size_t)NCODE * 40,
                 CT_D1 = (size_t)NCODE * 48, CT_BYTES = (size_t)NCODE * 56;

// Coefficient of code 0 of a kind, and the step from code to code in coefficients of the kind.
template <int K>
constexpr size_t ct_offset = K == 0 ? CT_D1 : (K == 2 ? CT_D2 : CT_F2);
template <int K>
constexpr int ct_step = K == 1 ? 2 : 1;

// Arguments of one segment's pass of the stored-structure H.x.
struct CachePass {
    const uint8_t* counts;      // [32 ns] entries of each row in this segment
    const uint32_t* boff;       // [ns] first entry of each slice, relative to its chunk's entries
    const uint32_t* const* ent; // [chunks] entries of each chunk of slices
    const void* x;              // [nvec][D]
    void* xi;                   // several FP32 vectors: room for their copy interleaved by row (filled at mode 0 and 1), or null
    void* y;                    // [nvec][D]
    const void* ctab;           // coefficients: ct_offset<K>, or an axis-aligned table
    const void* isq;            // [G+1] 1/sqrt(k) of the value kind's real type
    const uint16_t* stab;       // [D] |Stab sigma_i|
    const double* diag;         // [D] Ising part
    int64_t D, ns, xoff;        // xoff: first column of the segment
    bool diff;                  // general complex sums by product differences (RowSum)
    int nvec, mode;             // mode 0: the only segment, 1: first, 2: inner, 3: last
    int chunk_shift;            // slice >> chunk_shift = chunk
    uint32_t off_bits;          // entry = (code << off_bits) | column offset
    uint32_t n_re;              // codes below n_re have real coefficients (complex kinds)
    unsigned long long* counters;  // receives n_ent, n_skip, 0 (ed_apply_counters), or null
    unsigned long long n_ent, n_skip;
    int nb;                     // segments
};

// One segment's pass for p.nvec vectors of kind K, `lanes` warps per slice for
// one vector.  ax: p.ctab is the axis-aligned table.
ed_status launch_cache_pass(const CachePass& p, int K, bool ax, int lanes, int sms, cudaStream_t s);

}  // namespace ed

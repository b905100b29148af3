// Layouts shared by the staged RCR passes on CUDA cores (rcr_staged.cu) and
// their tensor-core rotation passes (rcr_staged_tc.cu).
#pragma once

#include <cstdint>
#include <vector>

#include "common.cuh"

namespace stg {

// one pair (column) of a staged level
struct StgSlot {
    int64_t src_off;   // first coefficient of the source expansion
    int64_t dst_off;   // first coefficient of the target expansion
    int32_t dir;       // translation direction (phase table)
    int32_t pad;
};

// start of degree n in the unfolded rotation factors of one direction
__host__ __device__ __forceinline__ int64_t rot_off(int n) { return (int64_t)n * (2 * n - 1) * (2 * n + 1) / 3; }

// start of degree n in a folded rotation table (blocks (n+1)^2 + n^2)
__host__ __device__ __forceinline__ int64_t fo(int n) {
    return (int64_t)(n - 1) * n * (2 * n - 1) / 3 + (int64_t)n * n;
}

// ---- tensor-core passes ----------------------------------------------------
constexpr int STC_SLOTS = 64;     // slots per item (128 accumulator rows)
constexpr int STC_COLS = 256;     // accumulator columns of an item, at most
constexpr int STC_CROWS = 128;    // coaxial output rows (complex) per item
// Slots of a level whose rotations run on the tensor cores start every
// polar-angle group at a multiple of 16: whole 128-byte lines of u and v.
constexpr int STC_ALIGN = 16;

// One block of a pass applied to up to 64 slots.  R, B: degree n, folded part
// `part`, slots s0 .. s0 + ns of polar-angle group g; C: order n, output
// degrees from n + part on, slots cidx[s0 ..] of one |t| set.
struct StcItem {
    int64_t tab;      // float offset of its table block (R, B: within the group's table)
    int32_t s0, ns;
    int32_t n, part;
    int32_t N, K;     // real columns and summed length
    int32_t g;
    int32_t uni;      // set on the device: groups of slots with one direction,
    int64_t rhs, uoff;   // right-hand side and the offset of its u and v
};

// columns of the folded degree-n block (rows of the table), padded to 16
__host__ __device__ __forceinline__ int stc_pad16(int v) { return (v + 15) & ~15; }

// Float offsets of the pre-split canonical table blocks of one group and
// pass: toff[2 n + part] for degrees n < P (square blocks of
// stc_pad16(n + 1 - part) rows and K values, K chunks of 16 each holding the
// TF32 part then the remainder); returns the floats per group and pass.
int64_t fb_stc_layout(int P, std::vector<int64_t>& toff);

// Appends the items of one polar-angle group (slots [g0, g1)) for degrees
// [0, nmax) of pass 0 (rotation) or 1 (back-rotation; K limited by p_in).
void fb_stc_group_items(int g, int g0, int g1, int nmax, int pass, int p_in, std::vector<StcItem>& out);

// A pre-split coaxial block to build: C^{am}_{am + r0 + i, am + k} of the set
// at coax offset cs_off (row stride pc), i < nr, k < K, at float toff.
struct StcCBlock {
    int64_t cs_off, toff;
    int32_t pc, am, r0, nr, K, pad;
};

// Appends the coaxial items and table blocks of one |t| set (ns slots at
// cidx[c0], coefficients at cs_off, stride pc) of a level; *tfloats grows by
// the floats of the new table blocks.
void fb_stc_coax_set(int c0, int ns, int64_t cs_off, int pc, int p_in, int p_out, std::vector<StcItem>& items,
                     std::vector<StcCBlock>& blocks, int64_t* tfloats);
void fb_stc_sort(std::vector<StcItem>& items);
// Builds the pre-split coaxial blocks (3xTF32 real form of the complex
// blocks) from the FP64 coaxial sets.
fb_status fb_stc_coax_tables(const StcCBlock* blocks, int nblocks, const cd* coax64, float* out, cudaStream_t s);

// Launches the items of a pass: rotation 0 (expansions -> u), back-rotation 1
// (v -> expansions), coaxial 2 (u -> v); ncol_max bounds their columns; ns is
// the level's number of slots, u and v are [coefficient][slot].  For nrhs
// right-hand sides, their expansions rstride and their u and v ustride apart.
fb_status fb_stc_run(int pass, const StcItem* items, int nitems, int ncol_max, const float* tab, int64_t tper,
                     const StgSlot* slots, const int32_t* cidx, const cf* X, cf* out, int64_t ns, const cf* rph,
                     int prot, int* err, cudaStream_t s, int nrhs, int64_t rstride, int64_t ustride);

}  // namespace stg

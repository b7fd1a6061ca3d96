// Bitmaps over the columns of a tableau, 32 columns to a word, as the panel
// kernel (gbs_panel.cu) keeps them: columns that are basic, and columns a panel
// leaves out.  Host and device, so that the CPU tests run the same arithmetic.
#pragma once

#ifdef __CUDACC__
#define GBS_HD __host__ __device__ __forceinline__
#else
#define GBS_HD inline
#endif

namespace gbs {

// The bits of word w (one that holds some of the N columns) past the last
// column.  They are set in every bitmap of columns left out: the vectors listed
// from it then all lie within the N columns.
GBS_HD unsigned past_end(int w, int N) {
    const int here = N - 32 * w;
    return here < 32 ? ~0u << here : 0u;
}

// Whether the u-th vector of VW columns of a word of left-out columns has a
// column that is not left out.
GBS_HD bool vector_kept(unsigned left_out, int u, int VW) {
    const unsigned full = (1u << VW) - 1u;
    return (left_out >> (u * VW) & full) != full;
}

// Overlapped panels go from one tableau buffer to the other: one leaves out the
// columns that did not change in it (`stay`) nor in the panel before (`prev`),
// which are the same in both buffers.  Returns them, and makes prev what the
// next panel needs; a panel that gets all columns leaves none but the padding.
GBS_HD unsigned left_out_of_panel(unsigned &prev, unsigned stay, bool all, unsigned pad) {
    const unsigned out = prev & stay;
    prev = all ? pad : stay;
    return out;
}

// A pivot: column `leaving` is basic no more (nor has it stayed so), column
// `entering` is.  `leaving` may be any bits once the wait for it ran out (the
// solve then ends at its next exchange): outside the N columns it marks nothing.
GBS_HD void change_basis(unsigned *basic, unsigned *stay, int leaving, int entering, int N) {
    if (leaving >= 0 && leaving < N) {
        basic[leaving >> 5] &= ~(1u << (leaving & 31));
        stay[leaving >> 5] &= ~(1u << (leaving & 31));
    }
    basic[entering >> 5] |= 1u << (entering & 31);
}

}  // namespace gbs

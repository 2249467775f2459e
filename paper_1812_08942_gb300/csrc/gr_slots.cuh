// Slots [b, e) of a row, taken U at a time with 32-bit numbers (2 m < 2^32).
// The last row of a graph of 2^31 - 1 edges ends at 2^32 - 2, where `j += U`
// and `j + u < e` may wrap: a kernel either counts what is left down (SlotRun)
// or is launched only where no number past the end wraps (slots_step_fits; the
// row-group sweep, whose four-slot FP32 form takes 75 registers counting down
// and 64 so, a block less per SM).
#pragma once

#ifdef __CUDACC__
#define GR_SLOTS_FN __host__ __device__ __forceinline__
#else
#define GR_SLOTS_FN inline
#endif

namespace gr {

struct SlotRun {
    unsigned at, left;  // the next slot, and how many there are from it on
    GR_SLOTS_FN SlotRun(unsigned b, unsigned e) : at(b), left(e - b) {}
    GR_SLOTS_FN bool has(unsigned u) const { return u < left; }
    GR_SLOTS_FN void next(unsigned step) {
        left = left > step ? left - step : 0u;
        at += step;
    }
};

// j < e <= slots: whether j + u for u < step, and j + step, stay below 2^32
GR_SLOTS_FN bool slots_step_fits(unsigned long long slots, unsigned step) {
    return slots + step <= 0x100000000ull;
}

}  // namespace gr

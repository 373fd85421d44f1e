// The units of work that a CTA takes one after the other.  One loading thread publishes them in two slots of shared memory, every
// other role of the kernel reads them there; the block index of the next unit comes from the hardware's scheduler (tc_common.cuh).
//
// After a wait has run out waits return at once and the roles go through the rest of their unit with whatever is there, so that they
// all come to an end.  What they form addresses from must not change under them: every role arrives on `empty` once a unit, when it
// is done with the slot, and the loading thread stops at its first wait that fails, without another load and without publishing
// anything.  A slot is therefore rewritten only when nobody reads it any more.  A role of whole warps takes a unit with all its
// lanes or with none.
//
// `Io` supplies the barriers and the scheduler (UnitIo in the kernels; a host program can stand in for it).  The first member of
// `Unit` is an int `tile`; -1 says that there is no more work.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define ATTN_UNITS_FN __device__ __forceinline__
#else
#define ATTN_UNITS_FN inline
#endif

namespace attn {
namespace tc {

template <typename Unit, typename Io>
struct UnitQueue {
    volatile Unit *slots;       // two
    uint64_t *full, *empty;     // barriers of each slot: published; read by every role
    uint64_t *answered;         // the scheduler's answer is there
    void *answer;
    Io io;

    // -- the loading thread
    // The slot of the t-th unit, once every role is done with what it held; null: the kernel is giving up.
    ATTN_UNITS_FN volatile Unit *claim(int t) const
    {
        return t < 2 || io.wait(&empty[t & 1], ((t >> 1) - 1) & 1) ? &slots[t & 1] : nullptr;
    }
    ATTN_UNITS_FN void publish(int t) const { io.arrive(&full[t & 1]); }
    // Asks for the unit after the t-th one; once per unit, early enough that the answer is there when the loads get to it.
    ATTN_UNITS_FN void ask() const { io.request(answer, answered); }
    // Its block index, or false: there is none, which the other roles are told, or the kernel is giving up.
    ATTN_UNITS_FN bool next(int t, int &bx, int &by) const
    {
        if (!io.wait(answered, t & 1)) return false;
        const bool late = io.late(), more = io.answer(answer, bx, by);   // both loads in flight
        if (late || more) return !late;
        if (volatile Unit *end = claim(t + 1)) {
            end->tile = -1;
            publish(t + 1);
        }
        return false;
    }

    // -- the other roles: whether there is a t-th unit, for a single thread, a whole warp, and a group of warps that wait for one
    // another without a limit while they work on it: either all of them take it or none (io.all_warps is such a wait itself)
    ATTN_UNITS_FN bool take_alone(int t) const { return io.wait(&full[t & 1], (t >> 1) & 1) && slots[t & 1].tile >= 0; }
    ATTN_UNITS_FN bool take(int t) const { return io.all(io.wait(&full[t & 1], (t >> 1) & 1)) && slots[t & 1].tile >= 0; }
    ATTN_UNITS_FN bool take_together(int t) const { return io.all_warps(io.wait(&full[t & 1], (t >> 1) & 1)) && slots[t & 1].tile >= 0; }
};

}  // namespace tc
}  // namespace attn

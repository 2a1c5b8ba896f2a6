// A loop that a group of threads runs in step, each with waits of its own that may run out.
//
// Every pass holds barriers of the whole group or of parts of it, so no thread may leave before the others know: a thread
// whose wait ran out (ok = false) stays until the next vote, leaves a mark there, and all leave together.  One barrier a
// pass answers both questions, whether anyone has work left and whether everyone's waits succeeded.  After the last
// pass, which no vote follows, the threads agree once more.  (Plain C++, so that it also compiles for the host.)
#pragma once

#ifdef __CUDACC__
#define LLA_VOTED_LOOP_INLINE __device__ __forceinline__
#else
#define LLA_VOTED_LOOP_INLINE inline
#endif

namespace lla {

// At most `most` passes of body(t), which returns false (in all threads alike) to stop.  ok: the same in all threads on
// entry and on return; body may clear it.  marks: two words shared by the group, zero on entry; they are used in turn, so
// that none is set while the last one is still read.  active(): work left for this thread.  any(v): OR of v over the group (a
// barrier).  Returns the passes run.
template <typename Active, typename Body, typename Any>
LLA_VOTED_LOOP_INLINE int voted_loop(int most, bool& ok, volatile int* marks, Active&& active, Body&& body, Any&& any) {
    int t = 0;
    for (; t < most; ++t) {
        const bool mine = active();
        volatile int* mark = marks + (t & 1);
        if (!ok) *mark = 1;
        const bool more = any(mine);
        if (*mark) ok = false;
        if (!more || !ok || !body(t)) break;
    }
    ok = !any(!ok);
    return t;
}

}  // namespace lla

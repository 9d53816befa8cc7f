// What is left of a ring of copies whose steps two producers fill together, once a wait has run
// out: plain bookkeeping, without CUDA, so that it can be checked on the host.
#pragma once

#ifdef __CUDACC__
#define YORO_RING_FN __device__ __forceinline__
#else
#define YORO_RING_FN inline
#endif

namespace yoro {

// Step k's barrier takes one arrival from each producer with its copy.  The producers issued the
// steps below a and below b, the consumer finished those below `used`; all three have stopped.
// For every step that only one of them issued the other's arrival is made up (arrive), so that
// the barrier completes with the copy that is in flight, and every copy is waited for (wait): a
// CTA must not end while a copy into its shared memory is under way.
template <class Arrive, class Wait>
YORO_RING_FN void ring_drain(int used, int a, int b, Arrive arrive, Wait wait)
{
    const int last = a > b ? a : b;
    for (int k = used; k < last; ++k) {
        if (k >= a || k >= b) arrive(k);
        wait(k);
    }
}

}  // namespace yoro

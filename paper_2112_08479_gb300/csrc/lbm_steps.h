// lbm_steps.h -- the host loop of lbm_step over its launches.
#pragma once

namespace lbmgpu {

// Enqueues nsteps time steps, the first of parity `odd`: chain(odd, n, done)
// launches the first `done` of n steps together (0: none), single(odd) one step;
// both return 0 (cudaSuccess) or an error.  `enqueued` counts the steps whose
// launches succeeded, also when a later one fails: the parity of the layout that
// the device will hold, and the caller's step count, follow from it.
template <typename Chain, typename Single>
auto enqueue_steps(bool odd, int nsteps, int& enqueued, Chain&& chain, Single&& single)
    -> decltype(single(odd)) {
    using Error = decltype(single(odd));
    enqueued = 0;
    auto parity = [&] { return odd != ((enqueued & 1) != 0); };
    while (nsteps - enqueued >= 2) {
        int done = 0;
        const Error e = chain(parity(), nsteps - enqueued, done);
        if (e != Error{}) return e;
        if (!done) break;
        enqueued += done;
    }
    while (enqueued < nsteps) {
        const Error e = single(parity());
        if (e != Error{}) return e;
        ++enqueued;
    }
    return Error{};
}

}  // namespace lbmgpu

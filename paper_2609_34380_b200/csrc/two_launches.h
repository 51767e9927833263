// One call that is two launches: plain host control flow, no CUDA, so that its order can be checked.
#pragma once

namespace dps {

// All that can fail in front of the second launch -- set-up, tensor maps -- is done before the first one is enqueued, so that a call that fails there
// has enqueued nothing.  first(): launches; second(prepare_only): prepares, and launches unless told not to.  Errors are non-zero.
template <typename First, typename Second>
auto launch_two(First first, Second second) -> decltype(first()) {
    auto e = second(true);
    if (!e) e = first();
    if (!e) e = second(false);
    return e;
}

}  // namespace dps

// Workspaces that hold a number of parts and serve with fewer (host code without CUDA: any status type).
#pragma once

namespace kh {

// Grows a workspace for `parts` parts by grow(parts); while that reports `no_room` and there are more parts than
// one, for half of them (`parts` is set to what was grown for).  Returns the last status.
template <typename Status, typename Grow>
Status grow_parts(int& parts, Status no_room, Grow grow)
{
    Status e = grow(parts);
    while (e == no_room && parts > 1) {
        parts = (parts + 1) / 2;
        e = grow(parts);
    }
    return e;
}

}  // namespace kh

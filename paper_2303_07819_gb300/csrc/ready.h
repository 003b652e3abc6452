// ready.h -- working memory made and filled by its first user (host only).
#pragma once

namespace msd {

struct WorkArea {
    unsigned char *p = nullptr;
    bool ready = false;      // allocated and filled: p alone does not say so
};

// Allocates w (alloc(p)) and fills it (fill(p)) unless that is done; both
// return 0 or an error, which leaves w to be filled by the next call.
template <class Alloc, class Fill>
auto make_ready(WorkArea &w, Alloc &&alloc, Fill &&fill) -> decltype(fill(w.p))
{
    decltype(fill(w.p)) e{};
    if (w.ready) return e;
    if (!w.p) e = alloc(w.p);
    if (!e && !(e = fill(w.p))) w.ready = true;
    return e;
}

}  // namespace msd

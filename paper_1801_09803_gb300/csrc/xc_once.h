// xc_once.h -- device constants that a handle makes once (host code without CUDA).
#pragma once

#include <stddef.h>

namespace xc {

// Allocates `buf` and has `make` launch what fills it, unless it is made already.  After an error nothing is
// left that the next call would take for made.  The contents are there when the call's stream has run:
// every call waits for it before it returns, also when it fails, so a later one may use any stream.
template <class Buf, class Make>
auto make_once(Buf &buf, size_t bytes, Make make) -> decltype(make()) {
    if (buf.p) return decltype(make())();
    auto e = buf.ensure(bytes);
    if (e == decltype(e)()) e = make();
    if (e != decltype(e)()) buf.release();
    return e;
}

}  // namespace xc

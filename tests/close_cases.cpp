// The serving kernel's agreement to leave (serve_close.h) behind a C interface for ctypes (test
// infrastructure): one party runs while the other is between two of its steps.
#include <functional>

#include "serve_close.h"

namespace {

struct Word {
    int v = 0, step = 0, at = -1;
    std::function<void()> other;
    void turn()
    {
        if (step++ != at) return;
        const auto f = other;
        other = nullptr;
        at = -1;
        if (f) f();
    }
    int add(int d) { turn(); const int o = v; v += d; return o; }
    int cas(int e, int d) { turn(); const int o = v; if (o == e) v = d; return o; }
    int load() { turn(); return v; }
};

}  // namespace

// `first` (0: close, 1: enter) starts with `held` CTAs entered; the other runs before its step `at` (or
// after it). Result: bit 0 the close took effect, bit 1 the CTA entered, bit 2 closed at the end; the
// number entered at the end << 3.
extern "C" int close_case(int first, int held, int at)
{
    using namespace rs;
    Word w;
    for (int i = 0; i < held; ++i) life::enter(w);
    bool did = false, in = false;
    const auto do_close = [&] { did = life::close(w); };
    const auto do_enter = [&] { in = life::enter(w); };
    w.step = 0;
    w.at = at;
    if (first == 0) w.other = do_enter; else w.other = do_close;
    if (first == 0) do_close(); else do_enter();
    w.at = w.step;
    w.turn();                                      // not run in between: now
    return (did ? 1 : 0) | (in ? 2 : 0) | (life::closed(w) ? 4 : 0) | (w.v & ~life::CLOSED) << 3;
}

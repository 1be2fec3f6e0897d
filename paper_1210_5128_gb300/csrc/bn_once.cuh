// bn_once.cuh -- set-up that a kernel needs once per CUDA context, such as its
// shared-memory attribute.  Compiles as plain C++ too.
#pragma once

#include <mutex>

namespace bn {

// One per call site, static.  run() has set_up() done in context `id` of device `dev` before
// it returns, whichever of several threads comes first: a thread that arrives while another
// is at it waits for the end (a launch that went ahead would find the attribute unset).  A
// context destroyed and created again (another id) is set up again; so is one whose set-up
// failed, and one the driver cannot name (id 0).  Returns set_up's code, 0 for success.
struct ContextOnce {
    static constexpr int DEVICES = 64;

    template <class F>
    int run(int dev, unsigned long long id, F set_up)
    {
        std::lock_guard<std::mutex> g(mu);
        const bool named = dev >= 0 && dev < DEVICES && id != 0;
        if (named && done[dev] == id) return 0;
        const int rc = set_up();
        if (named && rc == 0) done[dev] = id;
        return rc;
    }

private:
    std::mutex mu;
    unsigned long long done[DEVICES] = {};
};

}  // namespace bn

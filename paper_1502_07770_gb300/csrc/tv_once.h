// Kernel attributes that are set once: they belong to the kernel in one CUDA context, so a process
// that uses a second device, or has reset one, sets them again.
#pragma once
#include <atomic>

namespace tvh {

class OncePerContext {
    std::atomic<unsigned long long> done_{0};  // id of the context they were last set in, plus 1

public:
    // Calls set() unless it succeeded (returned its type's zero) in the context that id(&ctx)
    // names; always, if there is no id. set() may run in several threads at once.
    template <class ID, class SET>
    auto run(ID id, SET set) -> decltype(set())
    {
        using Status = decltype(set());
        unsigned long long ctx = 0;
        const bool known = id(&ctx);
        if (known && done_.load(std::memory_order_acquire) == ctx + 1) return Status{};
        const Status st = set();
        if (known && st == Status{}) done_.store(ctx + 1, std::memory_order_release);
        return st;
    }
};

}  // namespace tvh

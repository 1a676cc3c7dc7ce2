// Chunked transfers between a host array and the device through a ring of
// slots in page-locked memory: the calling thread enqueues and awaits the
// device's work, chunk by chunk, while worker threads copy between slots and
// array. (Host code only, so that the CPU tests run it.)
#pragma once
#include <algorithm>
#include <atomic>
#include <cstdint>
#include <exception>
#include <thread>

namespace lbm {

constexpr int kStageSlots = 16;

// Io: bool launch(int64_t chunk, int slot)  enqueues the device's part of a chunk;
//     bool wait(int slot)                   returns when the slot's last launch has completed;
//     void copy(int64_t chunk, int slot)    the host's part (any thread).
// to_host: launch, wait, copy; else copy, launch, wait. A slot's next chunk
// begins after its last one has ended. False if a launch or wait failed; on
// every return no launch is outstanding and no copy is running, so slots and
// array may be released. Waits of threads on one another end: chunks advance in
// order, and a failure is seen by all.
template <class Io> bool staged_transfer(Io &io, int64_t chunks, int workers, bool to_host) {
    constexpr int S = kStageSlots;
    std::atomic<bool> stop{false};
    std::atomic<int64_t> given{to_host ? 0 : std::min<int64_t>(S, chunks)};   // chunks whose slot the host may use
    std::atomic<int64_t> taken{0};
    std::atomic<int64_t> copied[S];   // 1 + last chunk copied through the slot
    for (auto &c : copied) c.store(0);
    auto copy_next = [&]() -> bool {   // false: nothing left
        const int64_t c = taken.fetch_add(1);
        if (c >= chunks) return false;
        while (given.load(std::memory_order_acquire) <= c) {
            if (stop.load()) return false;
            std::this_thread::yield();
        }
        io.copy(c, (int)(c % S));
        copied[c % S].store(c + 1, std::memory_order_release);
        return true;
    };
    int64_t launched = 0, awaited = 0;
    auto is_copied = [&](int64_t c) { return copied[c % S].load(std::memory_order_acquire) == c + 1; };
    // As many launches as slots allow: into the slot of a chunk that the host has
    // emptied, or of one that it has filled.
    auto launch_ready = [&]() -> bool {
        while (launched < chunks && launched - awaited < S &&
               (to_host ? launched < S || is_copied(launched - S) : is_copied(launched))) {
            if (!io.launch(launched, (int)(launched % S))) return false;
            ++launched;
        }
        return true;
    };
    bool ok = launch_ready();   // the device works while the threads start
    std::thread th[S];
    workers = ok ? std::min(workers, S) : 0;
    for (int t = 0; t < workers; ++t) {
        try {
            th[t] = std::thread([&] {
                while (!stop.load() && copy_next()) {}
            });
        } catch (const std::exception &) {   // no more threads to be had
            workers = t;
        }
    }
    while (ok && awaited < chunks) {
        if (!(ok = launch_ready())) break;
        // from the host: keep the ring half full, so that copies go on meanwhile
        if (launched > awaited && (to_host || launched == chunks || launched - awaited >= S / 2)) {
            ok = io.wait((int)(awaited % S));
            ++awaited;
            if (ok) given.store(to_host ? awaited : std::min(chunks, awaited + S), std::memory_order_release);
        } else if (workers == 0) {
            copy_next();
        } else {
            std::this_thread::yield();
        }
    }
    for (; awaited < launched; ++awaited) (void)io.wait((int)(awaited % S));
    if (!ok) stop.store(true);
    if (workers == 0 && ok)
        while (copy_next()) {}
    for (auto &x : th)
        if (x.joinable()) x.join();
    return ok;
}

}  // namespace lbm

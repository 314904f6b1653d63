// held.h -- one object per host thread, given back when the thread ends.
#pragma once
#include <mutex>
#include <vector>

namespace hp {

// Held<T, make>::get(): this thread's T (make() where no idle one is left; null
// when that fails, to be tried again).  A thread that ends leaves its T to the next
// one that asks, so there are as many as threads that held one at the same time,
// however many threads come and go.  Nothing is freed: a thread may end while the
// process does, or while another thread captures a stream, where CUDA's calls are
// not allowed.
template <class T, T *(*make)()>
class Held {
    struct Idle {
        std::mutex mu;
        std::vector<T *> all;
    };
    static Idle &idle() {
        static Idle *p = new Idle;  // outlives every thread's holder
        return *p;
    }
    T *p = nullptr;
    ~Held() {
        if (!p) return;
        std::lock_guard<std::mutex> lk(idle().mu);
        idle().all.push_back(p);
    }

  public:
    static T *get() {
        thread_local Held h;
        if (!h.p) {
            std::lock_guard<std::mutex> lk(idle().mu);
            if (!idle().all.empty()) {
                h.p = idle().all.back();
                idle().all.pop_back();
            }
        }
        if (!h.p) h.p = make();
        return h.p;
    }
};

}  // namespace hp

// launch_chain.h -- which launches of one entry point may be late: start before the
// launch ahead of them has completed, and wait for it at their end instead of their
// start (host code, internal).
//
// An on-time launch waits at its start until the launch before it has completed, and
// lets its own successor start only after that wait.  So when a launch starts, all
// that may still be running is the last on-time launch and the late ones since;
// whatever came before the on-time one had completed before that one's wait ended.
// A launch may therefore be late exactly if it reads nothing that those write and
// writes nothing that those read or write -- not only its predecessor: of dX, dW1
// (late), dW2 (late), dX may still run beside dW2.  Buffers are compared by address
// range, so a gradient that the caller stores over the weights which an open launch
// reads (dW1 over W1 while dX runs) makes its launch an on-time one.
#pragma once

#include <stddef.h>
#include <stdint.h>

#include <initializer_list>

namespace vmoe {

struct Span {
    const void *ptr;
    size_t bytes;
};

class LaunchChain {
  public:
    typedef std::initializer_list<Span> Spans;

    // The next launch waits at its start.
    void on_time(Spans reads, Spans writes) {
        n_ = 0;
        anchored_ = true;
        open(reads, false);
        open(writes, true);
    }

    // Whether the next launch is a late one: `wanted`, and it may be; if not, it is an
    // on-time one.  An entry point's first launch never is late: what runs before it
    // is not known here.
    bool late(Spans reads, Spans writes, bool wanted = true) {
        if (!wanted || !anchored_ || n_ + (int)(reads.size() + writes.size()) > MAX || touches(reads, false) ||
            touches(writes, true)) {
            on_time(reads, writes);
            return false;
        }
        open(reads, false);
        open(writes, true);
        return true;
    }

  private:
    static constexpr int MAX = 24;
    struct Use {
        uintptr_t beg, end;
        bool write;
    } use_[MAX];
    int n_ = 0;
    bool anchored_ = false;

    void open(Spans s, bool write) {
        for (const Span &x : s) {
            if (n_ == MAX) {  // more than the chain can hold: nothing is late behind it
                anchored_ = false;
                return;
            }
            use_[n_++] = Use{(uintptr_t)x.ptr, (uintptr_t)x.ptr + x.bytes, write};
        }
    }
    bool touches(Spans s, bool write) const {
        for (const Span &x : s)
            for (int i = 0; i < n_; ++i)
                if ((write || use_[i].write) && (uintptr_t)x.ptr < use_[i].end &&
                    use_[i].beg < (uintptr_t)x.ptr + x.bytes)
                    return true;
        return false;
    }
};

}  // namespace vmoe

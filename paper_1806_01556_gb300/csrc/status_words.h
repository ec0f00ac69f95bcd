// Page-locked words that belong to one host thread, a pair per CUDA context (host code only).
//
// A thread may drive several contexts in turn (one per GPU), so a pair stays with its context and is found
// again by the context's id, which the driver never gives twice. A context that is destroyed takes its
// pair with it: its entry can never match again and is left as it is. The table is bounded: a thread that
// has met kMax contexts gets no words for a further one, and the caller then reads into its own memory.
#pragma once

namespace fdas {

// Memory: `unsigned *allocate()`, a pair for the current context or nullptr; `void release(int device,
// unsigned long long ctx, unsigned *words)`, which frees a pair if that context still lives.
template <class Memory, int kMax = 8>
class StatusWords {
  public:
    ~StatusWords() {
        for (int k = 0; k < count_; ++k) Memory::release(table_[k].device, table_[k].ctx, table_[k].words);
    }
    // The words of context `ctx` (current, on `device`), or nullptr when there are none to be had.
    unsigned *get(int device, unsigned long long ctx) {
        for (int k = 0; k < count_; ++k)
            if (table_[k].ctx == ctx) return table_[k].words;
        if (count_ == kMax) return nullptr;
        unsigned *const words = Memory::allocate();
        if (words) table_[count_++] = Entry{device, ctx, words};
        return words;
    }

  private:
    struct Entry {
        int device;
        unsigned long long ctx;
        unsigned *words;
    };
    Entry table_[kMax];
    int count_ = 0;
};

}  // namespace fdas

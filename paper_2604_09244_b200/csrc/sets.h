// Which scratch set a step takes.
//
// Sets rotate.  A scoring kernel re-arms the hand-over words of its set before it waits for the kernel in front of it, which may still be the tail of the
// step before: that is sound as long as the step before has another set, and the ones before it are complete by then.  Two things break that:
// calls that are captured take sets but run later, or never, and calls that fail have perhaps enqueued nothing.  Five of them in a row, and
// two steps that follow one another on a stream have the same set.  So the first step after either waits for all that its stream has been given.
// (A graph is ordered as a whole against what is launched before and after it; inside it steps follow one another as elsewhere.)
#pragma once

namespace mvla {

constexpr unsigned kSets = 6;         // scratch sets = prune steps that may be in flight at once

class SetRing {
public:
    struct Turn { unsigned set; bool wait; };
    // The next call's set, and whether its first kernel has to wait for all earlier work of the stream.  `capture`: the stream capture it is part of (0: none).
    Turn take(unsigned long long capture)
    {
        const bool wait = open_ || (capture == 0 && capture_ != 0);
        open_ = true;
        capture_ = capture;
        set_ = (set_ + 1) % kSets;
        return {set_, wait};
    }
    // The call has enqueued all that it was to enqueue.
    void done() { open_ = false; }

private:
    unsigned set_ = 0;
    unsigned long long capture_ = 0;
    bool open_ = false;
};

}  // namespace mvla

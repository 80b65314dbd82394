// Test helper: runs the fields warp's order of work (csrc/sk_fields_warp.h) on the host.  A copy stays in
// flight until something waits for it: the release of its stage (its readers have waited for it) or the
// drain.  Arguments: nk nb L stop, where stop is the number of waits that succeed before one gives up
// (negative: none does).  Prints the copies issued and those in flight when the warp leaves.
#include "sk_fields_warp.h"

#include <cstdio>
#include <cstdlib>

struct Host {
    int stop, copies = 0;
    bool flying[sg::kChainStages] = {}, bad = false;
    int filled[sg::kChainStages] = {};
    bool allowed() { return stop != 0 && (stop < 0 || stop-- > 0); }
    bool wait_empty(int s, unsigned phase) {
        if (!allowed()) return false;
        bad |= phase != (unsigned)(filled[s] - 1 & 1);  // the release of the stage's last block
        flying[s] = false;
        return true;
    }
    bool wait_published(int, int) { return allowed(); }
    void copy(int s, int, bool) {
        bad |= flying[s];
        flying[s] = true;
        ++filled[s];
        ++copies;
    }
    void drain(int s, unsigned phase) {
        bad |= phase != (unsigned)(filled[s] - 1 & 1);
        flying[s] = false;
    }
};

int main(int, char** argv) {
    Host h;
    h.stop = std::atoi(argv[4]);
    sg::run_fields_warp(h, std::atoi(argv[1]), std::atoi(argv[2]), std::atoi(argv[3]));
    int left = 0;
    for (bool f : h.flying) left += f;
    std::printf("%d %d %d\n", h.copies, left, (int)h.bad);
}

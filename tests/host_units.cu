// Host-side checks of the call context (no GPU): run by test_host_units_cpu.py, one check per argument.
#include <cstdio>
#include <cstring>
#include <vector>

#include "tk_expand_tf32.cuh"

// host_units_runtime.c: stand-ins for the runtime's calls, which several devices answer
extern "C" int fake_device;      // the current device
extern "C" int fake_set[16];     // devices a kernel's attribute was set on
extern "C" int fake_set_count;

// Stand-ins for the library's error exit and for the stream operations of a fork and of a side branch.
namespace tk {
void fail(tk_status st, const std::string& msg) { throw Error{st, msg}; }
void ctx_fork_begin(Ctx&, int) {}
void ctx_fork_end(Ctx& c, cudaStream_t main, int) { c.stream = main; }
void ctx_side_begin(Ctx& c) { c.stream = c.aux[Ctx::kFork]; }
void ctx_side_end(Ctx& c, cudaStream_t main) { c.stream = main; }
}  // namespace tk

// A branch of a fork or side sees the splits made before it and its own, never another branch's.
static int split_visibility() {
    for (int mode = 0; mode < 3; ++mode) {  // the planning pass, the executing one without and with auxiliary streams
        tk::Ctx c;
        c.exec = mode > 0;
        if (mode == 2)
            for (int i = 0; i < tk::Ctx::kAux; ++i) c.aux[i] = reinterpret_cast<cudaStream_t>(uintptr_t(8 * (i + 1)));
        c.split_cache = true;
        c.splits.push_back({});  // made before
        std::vector<size_t> seen;
        auto branch = [&]() {
            seen.push_back(c.splits.size());
            c.splits.push_back({});
            c.splits.push_back({});
        };
        c.fork(5, [&](int) { branch(); });
        c.fork(1, [&](int) { branch(); });
        c.side(
            [&]() {
                branch();  // the call's own stream: these two stay
                c.fork(2, [&](int) { branch(); });
            },
            branch);
        const std::vector<size_t> want = {1, 1, 1, 1, 1, 1, 1, 1, 3, 3};
        if (seen != want || c.splits.size() != 3) {
            std::printf("mode %d:", mode);
            for (size_t v : seen) std::printf(" %zu", v);
            std::printf(", %zu at the end\n", c.splits.size());
            return 1;
        }
    }
    return 0;
}

// A kernel's shared-memory limit is set once on every device that launches it, and each device has its own SM count.
static int per_device() {
    std::atomic<uint64_t> opted{0};
    for (int dev : {0, 0, 1, 0, 1, 63, 63, 64, 64}) {
        fake_device = dev;
        tk::smem_opt_in(opted, nullptr, 100000);
        if (tk::tc::num_sms() != 100 + dev) return 1;
    }
    const std::vector<int> want = {0, 1, 63, 64, 64};  // (above 63: every time)
    return std::vector<int>(fake_set, fake_set + fake_set_count) == want ? 0 : 1;
}

// An item of an expansion converts its tile of W again: the parts of a tile's blocks are those that end first.
static int expand_parts() {
    struct {
        int64_t ntiles, nblk, nj, want;
    } cases[] = {{7, 156, 39, 21},     // a wave: 8 blocks an item (156 items of one block: two waves)
                 {1, 30, 3, 30},       // few: every block its own item
                 {1024, 16, 39, 1},    // many waves: no part converts the tile again
                 {157, 16, 39, 2},     // three waves of half tiles, not two of whole ones
                 {35, 13, 39, 4},      {1, 1, 1, 1}, {300001, 1, 64, 1}, {1, 1 << 20, 64, 152}};
    for (const auto& c : cases) {
        const int64_t got = tk::tc::expand_parts(c.ntiles, c.nblk, c.nj, 152);
        if (got != c.want) {
            std::printf("%lld tiles, %lld blocks: %lld parts\n", (long long)c.ntiles, (long long)c.nblk, (long long)got);
            return 1;
        }
    }
    return 0;
}

int main(int argc, char** argv) {
    if (argc == 2 && !std::strcmp(argv[1], "split_visibility")) return split_visibility();
    if (argc == 2 && !std::strcmp(argv[1], "per_device")) return per_device();
    if (argc == 2 && !std::strcmp(argv[1], "expand_parts")) return expand_parts();
    return 2;
}

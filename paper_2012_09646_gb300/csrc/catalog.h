// Kernel table shared by the runtime and the built-in kernels.
#pragma once

#include <cstddef>
#include <cstdint>
#include <cstring>
#include <string>

#include "gdag.h"

namespace gdag {

constexpr int kMaxArgs = 16;

// Resolved arguments of one launch: device pointers for arrays, raw scalar
// bits for scalars, plus the array sizes for bounds validation.
struct LaunchArgs {
    void *ptr[kMaxArgs];
    size_t bytes[kMaxArgs];
    uint64_t val[kMaxArgs];
    int nargs = 0;
    bool auto_cfg = true;  // grid chosen by the kernel
    unsigned grid[3] = {0, 0, 0};
    unsigned block[3] = {0, 0, 0};
    size_t smem = 0;

    template <class T> T *p(int i) const { return static_cast<T *>(ptr[i]); }
    int64_t i64(int i) const { return static_cast<int64_t>(val[i]); }
    int32_t i32(int i) const {
        int32_t v;
        std::memcpy(&v, &val[i], 4);
        return v;
    }
    float f32(int i) const {
        float v;
        std::memcpy(&v, &val[i], 4);
        return v;
    }
};

// Validate sizes before anything is issued; return nullptr if fine, else a
// static message.
typedef const char *(*ValidateFn)(const LaunchArgs &);
// Issue the node's kernel launch(es) on `stream` (a cudaStream_t); returns a
// cudaError_t value.
typedef int (*LauncherFn)(const LaunchArgs &, void *stream);
// Issue `count` launches of the kernel (each validated, automatic launch
// shape) as one persistent launch on `stream` (more than one only when
// `count` exceeds the kernel's table capacity); returns a cudaError_t value.
typedef int (*FusedLauncherFn)(const LaunchArgs *members, int count, void *stream);

// Merged launches.  gdag_issue hands a merge rule the run of consecutive
// built-in launches that starts at a launch of the rule's kernel (each with its
// signature's access modes and the automatic launch shape).  The rule may claim
// several of them, the first one among them, to be issued as one unit, whose
// launcher does the work of all members.  The runtime checks that moving the later members up to the first one's place
// passes no conflicting launch, and that no array that a member writes shares
// memory with another array of the unit.
constexpr int kMaxRun = 32;

struct KernelEntry;
struct RunLaunch {
    const KernelEntry *k = nullptr;
    LaunchArgs a;
    int32_t array[kMaxArgs];  // array handles (array arguments only)
};

// A rule is asked at every launch of its kernel, so it looks at kernels and at the
// first launch before it has others resolved: a launch's arguments are resolved
// and validated once a gdag_issue call, when a rule first asks for them.
class Run {
  public:
    // The kernel of the run's launch j; null past the run's end.
    const KernelEntry *kernel(int j) { return j < known_ ? kernel_[j] : look(j); }
    // Launch j, resolved and validated with those before it; null if the run ends
    // before.  Valid for this asking of the rule.
    const RunLaunch *at(int j) { return j < ready_ ? launch_[j] : resolve_to(j); }

  protected:
    ~Run() = default;
    virtual const KernelEntry *look(int j) = 0;
    virtual const RunLaunch *resolve_to(int j) = 0;
    int known_ = 0, ready_ = 0;
    const KernelEntry *kernel_[kMaxRun];
    const RunLaunch *launch_[kMaxRun];
};

// As LauncherFn, over the members' arguments.
typedef int (*MergeLaunchFn)(const LaunchArgs *const *m, int count, void *stream);
struct Merge {
    int count = 0;
    int member[kMaxRun];  // indices into the run, in the order the launcher wants them
    // The first `apart` members need nothing from one another: on streams of their
    // own each would start as soon as its own inputs are there, and the runtime parts
    // them where that differs.  Host writes of up to waits_for bytes do not count, nor
    // kernels that with those before them touch at most waits_for_kernels (each).
    int apart = 0;
    uint32_t waits_for = 0, waits_for_kernels = 0;
    MergeLaunchFn launch = nullptr;
};
typedef bool (*MergeFn)(Run &run, Merge &out);

struct KernelEntry {
    std::string name;
    const void *fn = nullptr;  // user kernels: the __global__ handle
    int nargs = 0;
    gdag_argspec spec[kMaxArgs];
    ValidateFn validate = nullptr;  // built-ins only
    LauncherFn launcher = nullptr;  // built-ins only
    FusedLauncherFn fused = nullptr;  // built-ins with a fused form only
    MergeFn merge = nullptr;          // built-ins that start a merged launch only
};

template <size_t N> inline bool is(const KernelEntry *k, const char (&name)[N])
{
    return k && k->name.size() == N - 1 && std::memcmp(k->name.data(), name, N - 1) == 0;
}

// Built-in kernels (defined by the kernel translation units).
int builtin_count();
const KernelEntry &builtin(int i);

// Helpers for the table.
inline gdag_argspec arr(int mode) { return gdag_argspec{GDAG_ARG_ARRAY, mode, 0, 0}; }
inline gdag_argspec scal(int size) { return gdag_argspec{GDAG_ARG_SCALAR, 0, size, 0}; }

// Scratch sizes of the built-in kernels that need one (0 if none).
size_t scratch_bytes(const char *kernel, int64_t n);

}  // namespace gdag

"""Rules of the kernels' synchronisation that a missed case would break only
now and then on the GPU, checked on the source."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_16843_gb300", "csrc")


def kernels(name):
    """{kernel: body} of one source file, comments removed."""
    with open(os.path.join(CSRC, name)) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    out = {}
    for m in re.finditer(r"__global__ void[^{;]*?\b(k_\w+)\(", text):
        start = text.index("{", m.end())
        depth, end = 0, start
        while True:
            depth += {"{": 1, "}": -1}.get(text[end], 0)
            end += 1
            if depth == 0:
                break
        out[m[1]] = text[start:end]
    return out


def test_cluster_kernels_start_together():
    """A store to another CTA's shared memory is defined only once that CTA has
    started: every kernel that runs on a cluster passes a cluster barrier
    before its first such store and before it enters the step code, whose
    first operation may be a reduction."""
    found = {k: b for k, b in kernels("k_persist.cu").items() if "ClusterX x{" in b}
    assert set(found) == {"k_step_cluster", "k_batch_cluster"}
    for name, body in found.items():
        barrier = body.index("ClusterX::cluster_barrier()") if "ClusterX::cluster_barrier()" in body else len(body)
        first = min(i for i in (body.find("run_steps<"), body.find("st_cluster(")) if i >= 0)
        assert barrier < first, name


# the two waits of the convolution's roles, compiled for the host: 32 threads are the lanes of a warp
WAIT_HARNESS = r"""
#include <atomic>
#include <barrier>
#include <cstdint>
#include <cstdio>
#include <thread>
#include <vector>
#define __device__
#define __forceinline__ inline
static thread_local int lane;
static std::barrier<> meet(32);
static std::atomic<int> votes{0};
static bool __all_sync(unsigned, bool v) {
    votes += v;
    meet.arrive_and_wait();
    const bool all = votes == 32;
    meet.arrive_and_wait();
    if (lane == 0) votes = 0;
    meet.arrive_and_wait();
    return all;
}
// bit l of *bar: lane l finds the phase complete
static bool mbar_try_wait(uint64_t* bar, uint32_t) { return (*bar >> lane) & 1; }
static unsigned long long tc_globaltimer() { return 0; }
static void atomicMax(int* p, int v) { if (*p < v) *p = v; }
%s
int main() {
    const uint64_t done[] = {0xffffffffu, 0u, 1u, 0x55555555u, 0x7fffffffu, 0xffff0000u};
    for (uint64_t mask : done) {
        volatile int abort_flag = 1;
        int err = 0;
        std::vector<int> got(32);
        std::vector<std::thread> warp;
        for (int l = 0; l < 32; ++l)
            warp.emplace_back([&, l] {
                lane = l;
                uint64_t bar = mask;
                got[l] = mbar_wait_warp(&bar, 0u, &abort_flag, &err);
            });
        for (auto& t : warp) t.join();
        for (int l = 0; l < 32; ++l)
            if (got[l] != (mask == 0xffffffffu)) {
                std::printf("lanes %%llx: lane %%d went its own way\n", (unsigned long long)mask, l);
                return 1;
            }
    }
    return 0;
}
"""


def test_read_out_warps_of_the_convolution_give_up_together(tmp_path):
    """A read-out warp's lanes wait for an accumulator and then read it
    together; when another role gives up while the accumulator completes, some
    lanes see the one and some the other.  The warp goes on only if all lanes
    may, for every split of the lanes, and every read-out wait is of that
    kind."""
    import subprocess

    with open(os.path.join(CSRC, "unet.cu")) as f:
        src = f.read()
    funcs = []
    for name in ("mbar_wait_role", "mbar_wait_warp"):
        m = re.search(r"__device__ __forceinline__ bool %s\(.*?\n}\n" % name, src, re.S)
        assert m, name
        funcs.append(m[0])
    read_out = kernels("unet.cu")["k_conv_zb"]
    read_out = read_out[read_out.index("lane_base"):]
    assert "mbar_wait_warp(" in read_out and "mbar_wait_role(" not in read_out
    cpp = tmp_path / "wait.cpp"
    cpp.write_text(WAIT_HARNESS % "".join(funcs))
    exe = tmp_path / "wait"
    subprocess.run(["g++", "-std=c++20", "-O1", "-pthread", str(cpp), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout


def test_convolution_waits_for_every_bulk_copy():
    """The thread that issues the weights' bulk copies waits for the last of
    each buffer whatever became of the other roles (one of them may give up
    after this thread is through), so no copy lands in shared memory that
    another CTA already owns."""
    body = kernels("unet.cu")["k_conv_zb"]
    staging = body[:body.index("mbar_drain(&b_wfull")]
    tail = staging[staging.rindex("cp_async_wait_all();"):]
    assert "s_abort" not in tail and "if (pt == 0)" in tail


def test_weight_gradient_ctas_give_up_together():
    """After a chunk's barrier every thread of a CTA reads whether a wait gave up;
    a fast thread may by then be in its next wait.  So consecutive chunks, and
    the waits after the last, write other words than the one being read:
    threads that disagree would wait at different barriers."""
    body = kernels("unet.cu")["k_wgrad_tc"]
    assert re.search(r"__shared__ int s_abort\[3\]", body) and "s_abort[flag] = 1" in body
    loop = body[body.index("for (int c = 0; c < nch; ++c)"):]
    assert re.search(r"const int b = c & 1;\s+wait_mma\(b, b\);", loop)
    assert re.search(r"__syncthreads\(\);\s+if \(s_abort\[b\]\) break;", loop)
    assert re.search(r"wait_mma\(b, 2\);\s+__syncthreads\(\);", loop)

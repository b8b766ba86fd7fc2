"""Host-side rules of the kernels' headers, compiled and run without a device."""
import re
import subprocess
from pathlib import Path

CSRC = Path(__file__).resolve().parent.parent / "paper_2607_01844_b200" / "csrc"


def run_host_program(tmp_path, source):
    src, exe = tmp_path / "check.cu", tmp_path / "check"
    src.write_text(source)
    subprocess.run(["nvcc", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-diag-suppress", "550", "-I", str(CSRC),
                    "-o", str(exe), str(src)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0, out.stdout
    return out.stdout


def test_every_box_that_a_token_tile_can_pick_has_a_tensor_map(tmp_path):
    """An expert may hold all T k rows (a caller's indices may name it more than once for a token): whatever the size of its
    tiles, the box that the kernel picks is among the maps that the host encodes, and covers the CTA's half of the tile."""
    run_host_program(tmp_path, r"""
#include "gemm_tn.cuh"
#include <cstdio>
#include <vector>
using namespace mop;
static std::vector<unsigned> rows_of_box;
static CUresult fake_encode(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                            const cuuint32_t* box, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                            CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
    rows_of_box.push_back(box[1]);
    return CUDA_SUCCESS;
}
int main() {
    int bad = 0;
    for (int T = 1; T <= 300; ++T)
        for (int k = 1; k <= 32; ++k) {
            TcPlan p{};
            p.s.T = T; p.s.k = k; p.encode = reinterpret_cast<void*>(fake_encode);
            TnMaps m{};
            rows_of_box.clear();
            if (!tn_token_maps(&p, m.b, nullptr, (uint64_t)T * k, 64) || rows_of_box.size() > TN_BOXES) ++bad;
            for (int rows = 1; rows <= 256 && rows <= T * k; ++rows) {
                const int box = tn_box(rows);
                if (box >= (int)rows_of_box.size() || (int)rows_of_box[box] < ((rows + 15) & ~15) / 2) {
                    if (!bad++) std::printf("T %d, k %d, a tile of %d rows: %d maps\n", T, k, rows, (int)rows_of_box.size());
                }
            }
        }
    return bad != 0;
}
""")


def test_the_two_warps_of_an_epilogue_pair_leave_together(tmp_path):
    """The walk over the work items with every pair of points at which the two warps may see the CTA give up (or not at all):
    neither is ever left waiting at the vote, and both drain the same items."""
    run_host_program(tmp_path, r"""
#include "gemm_tn.cuh"
#include <chrono>
#include <condition_variable>
#include <cstdio>
#include <mutex>
#include <thread>
#include <vector>
using namespace mop;
struct Vote {                         // a barrier of two that ANDs their outcomes
    std::mutex m;
    std::condition_variable cv;
    int here = 0, round = 0;
    bool all = true, result[64], hung = false;
    bool operator()(bool ok) {
        std::unique_lock<std::mutex> l(m);
        all = all && ok;
        const int r = round;
        if (++here == 2) { here = 0; result[r % 64] = all; all = true; ++round; cv.notify_all(); return result[r % 64]; }
        if (!cv.wait_for(l, std::chrono::seconds(2), [&] { return round != r || hung; }) || hung) { hung = true; cv.notify_all(); return false; }
        return result[r % 64];
    }
};
int main() {
    const int items = 5;              // 0 .. 4, then none left
    for (int group = 0; group < 2; ++group)
        for (int a = 0; a <= 9; ++a)
            for (int b = 0; b <= 9; ++b) {        // the step (waits for items and for accumulators) from which a warp gives up
                Vote vote;
                std::vector<int> drained[2];
                auto warp = [&](int who, int give_up) {
                    int step = 0;
                    tn_walk_items<true>(group, [&](int n) { return step++ < give_up && n < items; },
                                        [&](int) { return step++ < give_up; }, [&](bool ok) { return vote(ok); },
                                        [&](int n) { drained[who].push_back(n); });
                };
                std::thread gate(warp, 0, a), up(warp, 1, b);
                gate.join();
                up.join();
                if (vote.hung || vote.here || drained[0] != drained[1]) {
                    std::printf("group %d: give-up at steps %d and %d leaves a warp behind\n", group, a, b);
                    return 1;
                }
                if (a == 9 && b == 9 && (int)drained[0].size() != (items + 1 - group) / 2) { std::printf("not drained\n"); return 1; }
            }
    return 0;
}
""")


def test_warps_that_wait_with_all_lanes_go_on_together():
    """Rings and parities count warps: a wait that every lane of a warp takes ends in a vote (mbar_wait_all, or an __all_sync of
    its outcome).  Single lanes wait for themselves in mbar_wait_warp, in the self-test and where one lane hands out the work items."""
    alone = ("if (lane == 0) ok = mbar_wait(", "limit_cycles);", "if (r >= 0 && !mbar_wait(signal_bar(")
    for path in sorted(CSRC.glob("*.cuh")):
        text = path.read_text()
        for call in re.finditer(r"\b(mbar_wait|mbar_wait_cluster|next_item)\(", text):
            start, end = text.rfind("\n", 0, call.start()) + 1, text.find("\n", call.end())
            line, before = text[start:end], text[start:call.start()]
            if "__forceinline__ bool mbar_wait" in line or "if (!mbar_wait_cluster(item_bar(n)" in line or any(a in line for a in alone):
                continue                                          # definitions (next_item itself included), single lanes
            # voted on in place, or in the next statements
            assert "__all_sync(0xffffffffu, " in before or "if (!__all_sync(0xffffffffu, ok))" in text[end:end + 250], \
                f"{path.name}: {line.strip()}"


def test_kernels_launched_beside_their_predecessor_wait_or_acquire_what_they_read():
    """Every kernel that pdl_launch starts begins with one of the forms of pdl_begin.  They are all there is of griddepcontrol, and
    the one that does not wait for its predecessor acquires a word that the predecessor releases after its own wait, waits all
    the same where it does not find it, puts a proxy fence before what TMA reads, and waits at its end."""
    texts = {p.name: p.read_text() for p in sorted(CSRC.glob("*.cu*"))}
    for name, text in texts.items():
        assert name == "common.cuh" or "griddepcontrol" not in text, name
    every = "\n".join(texts.values())
    started = set(re.findall(r"\bpdl_launch(?:_clusters)?\((\w+_kernel)\b", every)) | set(re.findall(r"\bgo\((\w+_kernel)<", every))
    assert len(started) > 20
    for kernel in sorted(started):
        body = re.search(r"__global__[^;{]*?\b" + kernel + r"\((?:[^{;]*)\{(.*?)\n\}", every, re.S).group(1)
        assert re.search(r"\bpdl_begin(_gemm|_beside)?\(", body), kernel

    def function(name):
        return re.search(r"void " + name + r"\(.*?\{\n(.*?)\n\}|void " + name + r"\(\) \{(.*?)\}\n", texts["common.cuh"], re.S).group(0)
    order = lambda text, *parts: [text.index(p) for p in parts] == sorted(text.index(p) for p in parts)
    assert order(function("pdl_begin"), "griddepcontrol.wait", "griddepcontrol.launch_dependents")
    assert order(function("pdl_begin_gemm"), "griddepcontrol.wait", "st.release.gpu", "__syncthreads()", "griddepcontrol.launch_dependents")
    assert order(function("pdl_begin_beside"), "ld.acquire.gpu", "__syncthreads_and", "griddepcontrol.wait", "fence.proxy.async.global")
    assert "griddepcontrol.wait" in function("pdl_end_beside")
    # a GEMM lets only a GEMM start early: smaller blocks would pile up on the SMs that empty first
    for name in ("pdl_begin_gemm", "pdl_begin_beside"):
        assert function(name).count("griddepcontrol.launch_dependents") == function(name).count('if (gemm_follows) asm volatile("griddepcontrol.launch_dependents') == 1
    for name, text in texts.items():
        assert text.count("pdl_begin_beside(") == text.count("pdl_end_beside("), name


def test_what_is_written_to_a_buffer_that_tma_copies_is_fenced_in_every_case():
    """SwiGLU backward: a step's results lie in a buffer that TMA then reads, or, where the rows leave one by one, writes over.
    Both are another proxy's accesses, so the fence between them and the lanes' stores hangs on no condition."""
    text = (CSRC / "gemm_tn.cuh").read_text()
    start = text.index("stmatrix4_trans(st + a * TN_STASH_BYTES")
    step = text[start:text.index("bar_vote_all(pair_bar", start)]
    assert re.search(r'\n +asm volatile\("fence\.proxy\.async\.shared::cta;"', step)
    assert step.index("fence.proxy.async") < step.index("if (")

"""Host-side rules of the kernels' headers, compiled and run without a device."""
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

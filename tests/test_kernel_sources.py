"""Orders inside the CUDA kernels that no run can show: a kernel that breaks one of them works almost always and is undefined,
or hangs, when the scheduler does something unusual.  Read from the sources, without a GPU."""
import os
import re
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_06172_b200", "csrc")


def kernels():
    """(file, kernel name, body without comments) of every __global__ function."""
    out = []
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith((".cu", ".cuh")):
            continue
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
        text = re.sub(r"__launch_bounds__\([^()]*\)", "", text)
        for m in re.finditer(r"__global__\s+void\s+(\w+)\s*\([^{;]*\)\s*\{", text):
            depth, at = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[at], 0)
                at += 1
            out.append((f, m.group(1), text[m.end():at]))
    return out


KERNELS = kernels()


def test_every_kernel_is_found():
    names = {k for _, k, _ in KERNELS}
    assert {"tgp_argmax_kernel", "tgp_wstream_tc_kernel", "tgp_matmul_tc_pair_kernel", "tgp_attn_prefill_tc_kernel", "tgp_expert_mma_kernel"} <= names


REMOTE = r"mapa\.shared::cluster|ld_remote_|sum_slices<|mbar_arrive_remote|tma_load_2d_pair|umma_pair|umma_commit_pair"
CLUSTER_WAIT = r"cluster_sync_all\(\)|barrier\.cluster\.wait"


@pytest.mark.parametrize("f,name,body", [k for k in KERNELS if re.search(REMOTE, k[2])], ids=lambda v: v if isinstance(v, str) and len(v) < 60 else "")
def test_shared_memory_of_another_cta_is_touched_only_after_a_cluster_barrier(f, name, body):
    """Another CTA's shared memory may be accessed only when that CTA is known to run, and it may leave only when nobody will touch its
    memory any more: one cluster barrier before the first access, one after the last."""
    waits = [m.start() for m in re.finditer(CLUSTER_WAIT, body)]
    uses = [m.start() for m in re.finditer(REMOTE, body)]
    assert waits and waits[0] < uses[0] and waits[-1] > uses[-1], (f, name)


@pytest.mark.parametrize("f,name,body", [k for k in KERNELS if "tcgen05.alloc" in k[2] and "launch_dependents" in k[2]], ids=lambda v: v if isinstance(v, str) and len(v) < 60 else "")
def test_a_kernel_holds_its_tensor_memory_before_it_releases_its_dependents(f, name, body):
    """A CTA that releases the next kernel before it has allocated tensor memory may find a CTA of that kernel on its SM with the columns
    it needs, which gives them back only after this kernel has ended.  The first thread that asks releases for the whole CTA, so
    the one place that asks stands behind the allocation, in the warp that made it."""
    assert body.count("launch_dependents") == 1, (f, name)
    assert re.search(r"tcgen05\.alloc[^;]*;[^}]*tcgen05\.relinquish_alloc_permit[^;]*;[^}]*griddepcontrol\.launch_dependents", body), (f, name)


def test_a_launch_hint_is_given_on_every_device_and_fails_no_product():
    """Function attributes are a device's own, so a flag of the process alone would leave a second device without them; and the
    error of a hint that was refused must not be found by the check behind the launch."""
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "tgp_kernels.cu")).read())
    body = re.search(r"static void launch_weights\(.*?\n\}\n", text, re.S).group(0)
    assert not re.search(r"static\s+(const\s+)?(cudaError_t|bool|auto)\b", body) and "cudaGetDevice" in body
    assert re.search(r"cudaFuncSetAttribute\([^;]*!= cudaSuccess\) cudaGetLastError\(\);", body)


def test_what_is_a_devices_own_is_kept_by_device():
    """A process may use several devices: an attribute that a flag of the process says is set, or a number of SMs asked for once, would be the first one's."""
    sources = {f: re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read()) for f in sorted(os.listdir(CSRC)) if f.endswith((".cu", ".cuh", ".h", ".cpp"))}
    for f, text in sources.items():
        assert not re.search(r"static\s+(bool|int|uint32_t)\s+(\w+\s*=\s*0\s*,\s*)?(attr_\w+|sms)\b", text), f
    held = {f: len(re.findall(r"cudaFuncSetAttribute\(", text)) for f, text in sources.items()}
    # tgpk_allow_smem() and launch_weights(), a bit per device each
    assert {f: n for f, n in held.items() if n} == {"tgp_kernels.h": 2, "tgp_kernels.cu": 1}
    assert sum(len(re.findall(r"cudaDevAttrMultiProcessorCount", text)) for text in sources.values()) == 1
    for f, name in (("tgp_kernels.h", "tgpk_allow_smem"), ("tgp_kernels.cu", "tgpk_sms")):
        body = re.search(r"\b%s\([^;{]*\) \{\n.*?\n\}\n" % name, sources[f], re.S).group(0)
        assert "tgpk_device()" in body, name
    assert "cudaGetDevice" in re.search(r"inline int tgpk_device\(\).*", sources["tgp_kernels.h"]).group(0)


# (activation rows, weight tiles, K): activation rows per tile that were within 3 % of the fastest, on 148 SMs (us; K = 64 and M = 288: 144 rows 9.8, 96 10.2, 64 11.1, 32 14.1)
FASTEST = {(288, 57, 64): {144}, (288, 57, 256): {144}, (212, 59, 128): {224, 256}, (417, 40, 128): {144}, (1264, 42, 256): {256}, (1758, 30, 256): {256}, (509, 56, 512): {256},
           (300, 118, 64): {160}, (300, 118, 1024): {112, 160}, (603, 8, 64): {80, 96}, (603, 8, 2048): {80, 96}, (1024, 16, 128): {256}, (1024, 16, 2048): {256}, (2000, 8, 512): {224},
           (400, 12, 64): {80}, (400, 12, 2048): {80},
           (501, 51, 4584): {256}, (501, 51, 5832): {256}, (2493, 33, 4584): {240}, (2493, 33, 7000): {240}, (539, 59, 232): {192}}


def test_tiles_of_the_paired_products_are_the_fastest_measured(tmp_path):
    """The estimate that chooses the tiles, compiled by itself: it knows the cost of a tile's end, which is most of a short K, and of rows that begin inside a line."""
    text = open(os.path.join(CSRC, "tgp_gemm_sm100.cu")).read()
    body = "".join(re.search(r"static \w+ %s\(uint32_t M, uint32_t wt.*?\n\}\n" % f, text, re.S).group(0) for f in ("pair_cost", "pair_rows"))
    calls = "".join('printf("%%u\\n", pair_rows(%du, %du, %du, 74, 256));' % case for case in FASTEST)
    src = tmp_path / "rows.cpp"
    src.write_text("#include <algorithm>\n#include <cstdint>\n#include <cstdio>\nconstexpr uint32_t BK = 64;\nstatic int g_tc_variant = 0;\n" + body + "int main() {" + calls + "}\n")
    subprocess.run(["g++", "-std=c++17", "-o", str(tmp_path / "rows"), str(src)], check=True)
    rows = [int(r) for r in subprocess.run([str(tmp_path / "rows")], capture_output=True, text=True, check=True).stdout.split()]
    assert len(rows) == len(FASTEST) and all(r in best for r, best in zip(rows, FASTEST.values())), dict(zip(FASTEST, rows))

"""Rules of the device code that no run can show broken, checked in its text:
the hardware leaves open what would go wrong, so a kernel that breaks one may
still give the right values on the chip at hand."""
import os
import re
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1310_3422_gb300", "csrc")


def code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"/\*.*?\*/|//[^\n]*", "", text, flags=re.S)


def functions(text):
    """(name, body) of every __global__ function."""
    for m in re.finditer(r"__global__\s+void[^;{]*?(\w+)\s*\((?:[^()]|\([^()]*\))*\)\s*\{", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        yield m.group(1), text[m.end():i]


@pytest.mark.parametrize("kernel", ["prop_tile_kernel", "prop_duo_kernel"])
def test_a_commit_comes_from_the_lane_that_issued_the_products(kernel):
    """tcgen05.commit tracks the MMAs of its own thread, and which lane
    elect.sync picks is not specified: a commit of a fixed lane may track none."""
    body = dict(functions(code("ge_prop.cu")))[kernel]
    assert re.search(r"bool leader = elect_one\(\)", body)
    assert re.findall(r"\btc_commit\w*\(\w+", body) == ["tc_commit_if(leader"]


def test_a_tile_buffer_is_fenced_before_tma_writes_it_again():
    """The rounds of a launch use the same two buffers, which threads wrote and
    read before: a proxy fence between those accesses and the copy, at every load."""
    loads = [m.start() for m in re.finditer(r"\btma_load_rows\(", code("ge_tb.cu"))]
    assert len(loads) == 2
    for at in loads:
        before = code("ge_tb.cu")[:at]
        assert re.search(r"fence_proxy_async_smem\(\);\s*mbar_arrive_expect_tx\([^;]*\);\s*$", before)


def test_two_teams_fit_shared_memory(tmp_path):
    """duo_rows for every halo and table size: the planes of both teams, and
    the 128 rows the MMA reads from any row of the last one's halo, end
    within the block's shared memory."""
    header = re.findall(r"constexpr int kProp[^;]*;", code("ge_prop.h"))
    text = code("ge_prop.cu")
    consts = re.findall(r"constexpr int kDuo[^;]*;", text)
    rows = re.search(r"__host__ __device__ __forceinline__ int duo_rows.*?\n\}", text, re.S).group(0)
    src = tmp_path / "duo.cpp"
    src.write_text("#include <cstdio>\n#define __host__\n#define __device__\n#define __forceinline__ inline\n"
                   + "\n".join(header + consts) + "\n" + rows + """
int main()
{
    int bad = 0;
    for (int hb = 1; hb <= kDuoHb; ++hb)
        for (int tab = 0; tab <= kPropTab32; tab += 16) {
            const int C = duo_rows(tab, hb);
            if (C <= 2 * hb)
                continue;  // the kernel leaves such a table to dot products
            const int left = kDuoSmem - 1024 - (tab + 1023) / 1024 * 1024;
            const int used = ((2 * kPropNv32 - 1) * C + 128 + 2 * hb) * 128;
            if ((C % 8 || used > left) && !bad++)
                std::printf("halo %d, %d bytes of tables: %d rows, %d of %d bytes\\n", hb, tab, C, used, left);
        }
    return bad ? 1 : 0;
}
""")
    exe = tmp_path / "duo"
    subprocess.run(["g++", "-std=c++17", "-O1", str(src), "-o", str(exe)], check=True)
    res = subprocess.run([str(exe)], capture_output=True, text=True)
    assert res.returncode == 0, res.stdout


def test_kernel_attributes_are_set_for_every_model():
    """The attributes a launch needs belong to a device: set once a process,
    a model on the next device would fail at its first launch."""
    text = code("ge_sno_tc.cu")
    assert not re.search(r"\bstatic\s+(bool|int)\b", text)
    assert len(re.findall(r"cudaFuncAttributeMaxDynamicSharedMemorySize", text)) == 1
    kernels = {name for name, _ in functions(text)}
    prepared = re.search(r"cudaError_t sno_tc_prepare.*?\n\}", text, re.S).group(0)
    assert kernels and kernels == set(re.findall(r"prepare_kernel\((\w+)", prepared))
    assert "sno_tc_prepare(&s->grid" in code("ge_sno.cpp")


def test_weights_of_any_number_are_prepared():
    """Models of 2^31 parameters and more (100 GB: no test makes one) take
    64-bit indices instead of an error."""
    body = re.search(r"cudaError_t sno_prepare\(.*?\n\}", code("ge_sno_kernels.cu"), re.S).group(0)
    assert "cudaErrorInvalidValue" not in body and "prepare_kernel<unsigned long long>" in body

"""What the sources of chained kernels (launched while their predecessor still writes) have to keep to, read from the files."""
import os
import re
import subprocess

from paper_2608_00916_b200 import build

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_00916_b200", "csrc")
FILES = ("route.cu", "combine.cu", "gemm.cu", "gemm2.cu", "gemm_common.cuh")
# what the caller hands in, complete before the first kernel of the call: x / dy (src), the router's weight, bias and logits
INPUTS = {"x", "src", "w", "W_r", "b_r", "logits_in"}


def sources():
    for name in FILES:
        with open(os.path.join(CSRC, name)) as f:
            yield name, f.read()


def chained_kernels(text):
    """(name, parameter list, start, body) of every kernel whose body starts with the chain's wait, or with chain_enter."""
    for m in re.finditer(r"__global__ [^;{(]*(?:__launch_bounds__\([^)]*\)\s+[^;{(]*)?\b(\w+)\(([^{;]*?)\) \{\s+(chain_wait\(\)|chain_enter\(\w+\));", text):
        yield m.group(1), m.group(2), m.group(3), text[m.end() : text.index("\n}\n", m.end()) + 1]


def test_predecessor_outputs_are_not_declared_read_only():
    kernels = set()
    for name, text in sources():
        for kernel, params, _, _ in chained_kernels(text):
            kernels.add(kernel)
            for param in params.split(","):
                if "const" in param and "__restrict__" in param:
                    assert param.split()[-1] in INPUTS, f"{name}: {kernel}: {param.strip()}"
        for helper, what in (("build_masks", "idx"), ("psum_columns", "psum_part"), ("scan_kernel", "tile_counts")):
            assert not re.search(helper + r"\([^{;]*__restrict__ " + what + r"\b", text), f"{name}: {helper}: {what}"
    # those that may run beside their predecessor among them
    assert {"router_bwd_kernel", "unpermute_sum_kernel", "dwr_partial_kernel", "unpermute_bwd_kernel"} <= kernels
    assert len(kernels) == 15


def test_a_kernel_beside_its_predecessor_ends_after_it():
    beside = set()
    for name, text in sources():
        for kernel, _, start, body in chained_kernels(text):
            if start.startswith("chain_enter"):
                beside.add(kernel)
                flag = start[len("chain_enter") :]
                assert body.endswith(f"  chain_leave{flag};\n"), f"{name}: {kernel}"
            else:
                assert "chain_leave" not in body, f"{name}: {kernel}"
    # all small kernels of the backward pass that need nothing of the weight gradient in front of them, with the router on tensor
    # cores and without
    assert beside == {"router_bwd_kernel", "unpermute_sum_kernel", "dwr_partial_kernel", "unpermute_bwd_kernel"}


def test_a_gemm_lets_its_successor_in_only_after_waiting():
    """Small kernels beside a GEMM read what its predecessor has written without a wait of their own: the first trigger of a block
    counts, so that each of its threads that triggers has waited.  (The other threads wait in front of the rows unless `ready`.)"""
    for name in ("gemm.cu", "gemm2.cu", "gemm_tokens.cu"):
        with open(os.path.join(CSRC, name)) as f:
            lines = [line.split("//")[0].strip() for line in f]
        triggers = [i for i, line in enumerate(lines) if "chain_next()" in line]
        assert triggers, name
        for i in triggers:
            assert lines[i - 1 : i + 1] == ["if (p.ready) chain_wait();", "chain_next();"], f"{name}:{i + 1}"
        assert any(line == "chain_warp(p.next_early);" for line in lines), name
    with open(os.path.join(CSRC, "gemm_common.cuh")) as f:
        text = f.read()
    assert text.count("chain_next()") == 1
    assert re.search(r"void chain_warp\(int next_early\) \{\s+chain_wait\(\);\s+if \(next_early\) chain_next\(\);\s+\}", text)


def test_non_coherent_loads_are_of_inputs_only():
    loads = [(name, arg) for name, text in sources() for arg in re.findall(r"__ldg\(([^;]*)\);", text)]
    assert loads
    for name, arg in loads:
        # W_r, the rows of src (s4), and hg / hu (qh, qu), which the forward call has left in the workspace
        assert re.search(r"\b(W_r|s4|qh|qu)\b", arg), f"{name}: __ldg({arg})"


def test_barriers_after_the_one_thread_roles_do_not_need_whole_warps():
    """elect_one() sends one lane through a role's loop and the others past it: the barrier that follows takes threads one by
    one, and the warp that frees tensor memory, an instruction for whole warps, comes together first."""
    for name, text in sources():
        if name in ("gemm.cu", "gemm2.cu"):
            after = text[text.rindex("elect_one()"):]
            end = re.search(r"\n  tc_fence_before\(\);\n  (\w+)\(\);[^\n]*\n  if \(warp == 1\) \{\n    __syncwarp\(\);[^\n]*\n"
                            r"    tc_fence_after\(\);\n    tmem_dealloc", after)
            assert end and end.group(1) in ("block_sync_diverged", "cluster_sync_diverged"), name


def test_a_failed_launch_of_a_gemm_is_reported_once():
    """The runtime's last error is taken by the call that failed; left in place, the next call would return it again."""
    for name, text in sources():
        if name in ("gemm.cu", "gemm2.cu"):
            assert re.search(r"  launch_kernel\([^;]*;\n  return cudaGetLastError\(\) == cudaSuccess \? MOE_OK : MOE_ERR_CUDA;", text), name


def test_the_ring_of_a_gemm_starts_its_shared_memory():
    """The operand tiles' swizzle needs stages at multiples of 1024 bytes: the ring is the dynamic memory itself, declared aligned, and
    nothing static lies in front of it."""
    for name, text in sources():
        if name in ("gemm.cu", "gemm2.cu", "gemm_common.cuh"):
            declared = re.findall(r"[^\n]*__shared__[^\n]*", text)
            assert all(re.match(r"\s*extern __shared__ __align__\(1024\) unsigned char \w+\[\];", line) for line in declared), name
            assert len(declared) == (name != "gemm_common.cuh"), name


def test_pairs_that_run_freely_ask_nothing_per_k_block():
    """What the copy thread does per K block sets the pace of short tiles: only the kernels that keep step ask where a tile's end is."""
    with open(os.path.join(CSRC, "gemm2.cu")) as f:
        text = f.read()
    loop = text[text.index("for (; kb < tl.nkb; ++kb, ++it) {") : text.index("issue_loads2<KIND>(p, tl, kb, rank, sA")]
    asks = [line for line in loop.splitlines() if "pace" in line]
    assert asks and all("if (PACED &&" in line for line in asks)


def test_no_gemm_keeps_registers_in_memory(tmp_path):
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    runs = [subprocess.Popen([nvcc, *build.NVCC_FLAGS, "-Xptxas", "-v", "-c", os.path.join(CSRC, name), "-o", str(tmp_path / (name + ".o"))],
                             stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True) for name in ("gemm.cu", "gemm2.cu", "gemm_tokens.cu")]
    kernels = 0
    for run in runs:
        out, _ = run.communicate()
        assert run.returncode == 0, out
        for kernel, spilt in re.findall(r"Compiling entry function '(\w+)'.*?(\d+) bytes spill stores", out, flags=re.DOTALL):
            kernels += 1
            assert spilt == "0", kernel
    assert kernels >= 20


def compiles(tmp_path, argument):
    src = tmp_path / "launch.cu"
    src.write_text('#include "common.cuh"\n'
                   "__global__ void kernel(const float* in, long n) {}\n"
                   "void go(float* f, const unsigned short* u, cudaStream_t st) {\n"
                   f"  moe::launch_kernel(kernel, 1, 32, 0, st, {argument}, 7);\n"
                   "}\n")
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    return subprocess.run([nvcc, *build.NVCC_FLAGS, "-I", CSRC, "-c", str(src), "-o", str(tmp_path / "launch.o")],
                          stdout=subprocess.DEVNULL, stderr=subprocess.DEVNULL).returncode == 0


def test_launch_arguments_convert_as_in_a_plain_launch(tmp_path):
    assert compiles(tmp_path, "f") and compiles(tmp_path, "nullptr")
    assert not compiles(tmp_path, "u")  # another pointer type
    assert not compiles(tmp_path, "7")  # a number

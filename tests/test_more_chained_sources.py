"""The properties of test_chained_sources.py, read from the kernels in files of their own."""
import pytest

import test_chained_sources as rules


@pytest.fixture(autouse=True)
def files(monkeypatch):
    monkeypatch.setattr(rules, "FILES", ("router.cu", "gemm_tokens.cu"))


def test_predecessor_outputs_are_read_by_ordinary_loads():
    for name, text in rules.sources():
        assert "__restrict__" not in text, name
        assert "chain_wait();" in text and "chain_next();" in text, name
    rules.test_non_coherent_loads_are_of_inputs_only()  # hg and hu, which the forward call has left


def test_barriers_after_the_one_thread_roles_do_not_need_whole_warps():
    """One lane of a warp is in its role's loop while the others wait: the barriers of whole blocks and clusters that follow take
    threads one by one, and the warp that frees tensor memory comes together first."""
    for name, text in rules.sources():
        after = text[text.index("elect_one()"):]
        assert "__syncthreads()" not in after and "cluster_sync_all()" not in after, name
        assert "if (warp == 1) {\n    __syncwarp();" in after, name


def test_a_failed_launch_is_reported_once():
    for name, text in rules.sources():
        assert text.count("launch_kernel(") == text.count("return cudaGetLastError() == cudaSuccess ? MOE_OK : MOE_ERR_CUDA;"), name


def test_every_row_gemm_walks_its_tiles_in_groups_by_one_rule():
    text = dict(rules.sources())["gemm_tokens.cu"]
    assert "p.row_group = row_group_for(" in text


def test_the_issuer_looks_a_tile_up_before_its_loop():
    """Producer and issuer are one thread each, and what they do per K block sets the pace: nothing there but barriers, copies and MMAs."""
    text = dict(rules.sources())["gemm_tokens.cu"]
    loop = text[text.index("for (int kb = 0; kb < nkb; ++kb) {") : text.index("umma_commit_pair_both(done);")]
    assert "idesc =" not in loop and not any(name in loop for name in ("__shared__", "get_token_tile", "stage_n"))
    assert text.count("__shared__") == 3  # dynamic memory, the barriers, the base of the accumulators

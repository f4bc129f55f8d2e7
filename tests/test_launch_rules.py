"""Source rules of kernels that start before their predecessor has finished (programmatic dependent launches).

They are properties of the source that no run shows reliably: breaking one gives a hang or a stale read only when a
launch happens to overlap its neighbours in the wrong way.
"""
import os
import re
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_19664_b200", "csrc")
TEXT = {f: re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read()) for f in sorted(os.listdir(CSRC))}
ALL = "\n".join(TEXT.values())


def _span(start, opening, closing):
    depth, i = 1, start
    while depth:
        depth += {opening: 1, closing: -1}.get(ALL[i], 0)
        i += 1
    return i


# name -> (arguments, body) of every kernel; a device function that holds the two calls of an early start is written out
HELPERS = {}
for m in re.finditer(r"__device__ __forceinline__ void (\w+)\(\) \{", ALL):
    body = ALL[m.end():_span(m.end(), "{", "}") - 1]
    if "grid_dependency_wait" in body or "grid_launch_dependents" in body:
        HELPERS[m.group(1)] = body
KERNELS = {}
for m in re.finditer(r"__global__ void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\s*\(", ALL):
    args_end = _span(m.end(), "(", ")")
    body = ALL.index("{", args_end) + 1
    text = ALL[body:_span(body, "{", "}")]
    for name, helper in HELPERS.items():
        text = text.replace(name + "();", helper)
    KERNELS[m.group(1)] = (ALL[m.end():args_end], text)


@pytest.mark.parametrize("name", sorted(k for k, (_, b) in KERNELS.items() if "tmem_alloc" in b and "grid_launch_dependents" in b))
def test_dependents_start_only_after_tensor_memory_is_allocated(name):
    """tcgen05.alloc waits without a limit.  A dependent that is let in first can take the columns its predecessor waits
    for, and then waits for that predecessor's end."""
    body = KERNELS[name][1]
    alloc, start = body.index("tmem_alloc"), body.index("grid_launch_dependents")
    assert alloc < start and re.search(r"__syncthreads\(\)|cluster_sync_all\(\)", body[alloc:start])


PREFILL = ["kvd_prefill_attn_tc_kernel", "kvd_prefill_attn_dual_kernel", "kvd_prefill_attn_split_kernel"]


def test_every_kernel_with_tensor_memory_is_covered():
    early = {k for k, (_, b) in KERNELS.items() if "tmem_alloc" in b}
    assert early == {"kvd_rows_kernel", "kvd_recompute_kernel", *PREFILL}
    assert all("grid_launch_dependents" in KERNELS[k][1] and "grid_dependency_wait" in KERNELS[k][1] for k in early)


@pytest.mark.parametrize("name", PREFILL + ["kvd_attn_split_kernel", "kvd_attn_split_mma_kernel", "kvd_attn_merge_kernel"])
def test_attention_reads_nothing_of_its_predecessor_before_the_wait(name):
    args, body = KERNELS[name]
    assert "__restrict__" not in args and "__ldg" not in body
    before = body[:body.index("grid_dependency_wait();")]
    assert not re.search(r"P\.(q|q_pos|k|v|out|part_o|part_ml|status)\b", before)


def test_few_row_producer_waits_for_its_last_copies_on_every_path():
    """A CTA that ends with a bulk copy in flight lets it land in the next CTA's shared memory."""
    body = KERNELS["kvd_rows_kernel"][1]
    drain = body[body.index("int issued"):body.index("umma_kblock")]
    drain = drain[:drain.index("else if (warp == 1)")]
    last = drain[drain.rindex("for (int b = 0; b < stages && b < issued"):]
    assert "mbar_try_wait(bar_full(b), par)" in last and "tmo +" in last
    between = drain[drain.rindex("ph ^= 1u;"):drain.rindex("for (int b = 0")]
    assert "if (" not in between  # the wait hangs on no condition


def test_a_few_row_cta_outlives_the_columns_it_is_sent():
    """What another CTA of the head sends must not land in the shared memory of whatever runs there next.  Each CTA waits
    for it; one that gave up leaves behind the cluster barrier (all have sent) and a second wait (it has landed)."""
    body = KERNELS["kvd_rows_kernel"][1]
    tail = body[body.index("cluster_arrive_relaxed();"):]
    assert re.search(r"mbar_try_wait_cluster\(bar_head, 0\)", tail[:tail.index("const bool got = !exchange || columns_within(tmo);")])
    assert "return;" not in tail
    assert re.fullmatch(r"\s*if \(!got\) columns_within\(\d+ull\);\s*\}\s*\}\s*", tail[tail.index("cluster_wait();") + 15:])


SMALL = sorted(set(re.findall(r"launch_dependent\((?:ctx, )?(kvd_\w+)", ALL)))


def test_the_small_dependent_kernels_are_found():
    assert len(SMALL) == 10 and all(k in KERNELS for k in SMALL), SMALL


@pytest.mark.parametrize("name", SMALL)
def test_inputs_of_a_small_dependent_kernel_are_plain_loads_behind_the_wait(name):
    args, body = KERNELS[name]
    assert "__restrict__" not in args and "__ldg" not in body
    assert "grid_dependency_wait();" in body


def test_row_statistics_are_plain_loads():
    text = TEXT["kvd_ptx.cuh"]
    assert "__ldg" not in text[text.index("void warp_rows_sumsq("):]
    for f in ("kvd_recompute.cu", "kvd_rows.cu"):
        assert not re.search(r"__ldg\([^)]*(sumsq|J\.scale|positions)", TEXT[f]), f


def test_keys_values_and_queries_are_coherent_loads():
    """Attention is resident while the projection writes the new tokens' keys and values, the recompute kernel while
    something writes the queries; the non-coherent load is for memory that nobody writes during the kernel."""
    assert ".nc" not in ALL
    assert "__ldg" not in TEXT["kvd_attention.cu"]
    assert not re.search(r"__ldg\(\s*q", TEXT["kvd_recompute.cu"])
    tables = re.compile(r"__ldg\(\s*(?:src \+ i|p\.w_scale|t_lo \+|t_hi \+|p\.gamma_k \+)")  # rotation tables, prepared weights
    for f in ("kvd_recompute.cu", "kvd_rows.cu", "kvd_prefill_attention_tc.cu", "kvd_scaffold.cu", "kvd_fp4.cu"):
        assert len(re.findall(r"__ldg\(", TEXT[f])) == len(tables.findall(TEXT[f])), f


def test_the_early_start_threshold_follows_the_device():
    """Which grids leave half of the SMs free is a question to the device, not a literal."""
    text = TEXT["kvd_internal.h"]
    fn = text[text.index("inline cudaError_t launch_dependent("):]
    fn = fn[:fn.index("\n}")]
    assert "ctx->num_sms" in fn and not re.search(r"grid\.x\s*[<>]=?\s*\d", fn)


def test_attention_launches_ask_the_device_for_its_sms():
    text = TEXT["kvd_attention.cu"]
    launch = text[text.index("static cudaError_t attn_launch_pair("):]
    launch = launch[:launch.index("\n}")]
    assert not re.search(r"\b148\b", launch) and len(re.findall(r"<= num_sms \*", launch)) == 4


def test_kernels_that_derive_store_slots_or_tiles_test_them_in_the_checking_build():
    body = KERNELS["kvd_rows_kernel"][1]
    for index in ("append_slot[r]", "col0"):
        assert re.search(r"KVD_BOUNDS_OK\([^;]*" + re.escape(index), body), index


def test_waits_on_what_the_other_cta_completes_acquire_at_cluster_scope():
    """st.async and bulk copies between the CTAs of a cluster release at cluster scope; a CTA-scope acquire does not
    synchronise with them, and no run shows that."""
    body = KERNELS["kvd_prefill_attn_split_kernel"][1]
    waits = re.findall(r"(\w*wait\w*(?:<\w+>)?)\(\s*(?:bar_(m|chain|sum|pv_done|p_ready)\(|(chain|m)_bar)", body)
    assert {a or b for _, a, b in waits} == {"m", "chain", "sum", "pv_done", "p_ready"} and len(waits) >= 12
    assert {f for f, _, _ in waits} <= {"peer_wait", "polite_wait<true>", "mbar_try_wait_cluster"}, waits
    assert "polite_warp_wait<true>" in body[body.index("auto peer_wait"):].split(";")[0]
    helper = TEXT["kvd_prefill_attention_tc.cu"]
    helper = helper[helper.index("bool polite_warp_wait("):]
    helper = helper[:helper.index("\n}")]
    assert "CLUSTER ? mbar_try_wait_cluster" in helper and "polite_wait<CLUSTER>" in helper


MARK = r"""
#include "kvd_launch_mark.h"
using kvd::LaunchMark;
int main() {
  LaunchMark m;
  int s1, s2;
  if (m.directly_before(0, &s1)) return 1;            // nothing launched yet
  m.set(7, &s1);
  if (!m.directly_before(7, &s1)) return 2;
  if (m.directly_before(7, &s2)) return 3;            // another stream
  if (m.directly_before(8, &s1) || m.directly_before(9, &s1)) return 4;  // another launch in between, or used up
  m.set(9, &s2);
  return m.directly_before(9, &s2) ? 0 : 5;
}
"""


def test_attention_starts_early_only_straight_behind_the_projection(tmp_path):
    """Grids of several waves start early behind the few-row projection; behind anything else their waiting CTAs take the
    SMs that a longer kernel needs.  What counts is the context's last launch, on this stream, not the last projection."""
    (tmp_path / "mark.cpp").write_text(MARK)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-o", str(tmp_path / "mark"), str(tmp_path / "mark.cpp")], check=True)
    assert subprocess.run([str(tmp_path / "mark")]).returncode == 0
    text = TEXT["kvd_attention.cu"]
    assert "S.early = ctx->few_rows.directly_before(ctx->launches, stream);" in text
    assert len(re.findall(r"small \|\| S\.early\)", text)) == 2  # both kernels, whatever the rows and the head size
    assert len(re.findall(r"few_rows\.set\(", ALL)) == 1
    rows = TEXT["kvd_rows.cu"]
    assert rows.index("ctx->launches += 1") < rows.index("few_rows.set(ctx->launches, stream")


def test_the_comparison_switch_reaches_whole_tiles_in_calls_of_any_length():
    """KVD_PREFILL_PAIR chooses single CTAs or pairs with whole tiles, so a shared tile is taken only where it is not set."""
    text = TEXT["kvd_prefill_attention_tc.cu"]
    choice = text[text.index('getenv("KVD_PREFILL_PAIR")'):]
    assert re.search(r"if \(!env && prefill_split_pays\(", choice)

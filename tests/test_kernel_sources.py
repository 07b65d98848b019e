"""Orders that a kernel has to keep and that no run shows reliably, read from the sources."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2406_13868_b200", "csrc")


def kernels():
    """(file, name, body without comments) of every __global__ function"""
    out = []
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith(".cu"):
            continue
        src = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(os.path.join(CSRC, f)).read(), flags=re.S)
        for m in re.finditer(r"__global__", src):
            open_brace = src.index("{", m.end())
            name = re.findall(r"(\w+)\s*\((?=[^()]*\)\s*$)", src[m.end():open_brace])[-1]
            depth, at = 1, open_brace + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(src[at], 0)
                at += 1
            out.append((f, name, src[open_brace:at]))
    return out


# what reaches another CTA's shared memory, and what says that every CTA of the cluster has started
REMOTE = re.compile(r"(?:st|ld)\.shared::cluster|ptx::(?:st_async|ld_cluster|mbar_arrive_remote|tc2_commit_both|tc2_commit_remote)\w*")
STARTED = re.compile(r"ptx::cluster_sync\(\)|barrier\.cluster\.wait")


def test_the_sources_are_read():
    names = [n for _, n, _ in kernels()]
    assert {"pack_kernel", "quant_act_fused_kernel", "channel_norm_kernel", "sdq_linear_kernel", "sdq_linear_pair_kernel", "sdq_linear_group_kernel"} <= set(names)
    assert sum(bool(REMOTE.search(b)) for _, _, b in kernels()) == 6


@pytest.mark.parametrize("name", [n for _, n, b in kernels() if REMOTE.search(b)])
def test_no_remote_shared_memory_before_the_cluster_has_started(name):
    """distributed shared memory may be touched only when all CTAs of the cluster are known to have started"""
    for _, n, body in kernels():
        if n == name:
            first, started = REMOTE.search(body).start(), STARTED.search(body)
            assert started and started.start() < first


@pytest.mark.parametrize("name", ["pack_kernel", "quant_act_fused_kernel"])
def test_a_thread_block_whose_wait_gives_up_stays_for_its_peers(name):
    """peers may still store into the shared memory of a thread block that gave up: it waits for them before it can leave"""
    body = {n: b for _, n, b in kernels()}[name]
    gave_up = re.search(r"if \(__any_sync\(0xffffffffu, !ptx::mbar_wait_cluster\(&s_bar, 0[^()]*\)\)\) \{([^{}]*)\}", body)
    assert gave_up and re.search(r"= 1u;|atomicOr\(&flags\[FLAG_TIMEOUT\], 1u\);", gave_up.group(1))
    assert re.search(r"ptx::cluster_wait_for_others\(\);\s*\(void\)ptx::mbar_wait_cluster\(&s_bar, 0\);", gave_up.group(1))


def test_a_packing_call_whose_wait_gave_up_returns_the_timeout():
    """it reads its kernel's report back anyway"""
    body = {n: b for _, n, b in kernels()}["pack_kernel"]
    assert re.search(r"if \(__any_sync\(0xffffffffu, !ptx::mbar_wait_cluster\(&s_bar, 0[^()]*\)\)\) \{[^{}]*\(p.gave_up\) = 1u;", body)
    src = open(os.path.join(CSRC, "sdq_pack.cu")).read()
    host = src[src.index("static sdq_status_t decompose("):]
    assert re.search(r"give_back\(report\);[^{}]*gave_up \? SDQ_ERR_TIMEOUT", host[:host.index("\n}\n")])


def test_packing_does_not_depend_on_the_device_s_status_word():
    """a packing call reports through words of its own; the plain layout's has no wait at all"""
    for f in ("sdq_pack.cu", "sdq_plain.cu"):
        assert "device_flags" not in open(os.path.join(CSRC, f)).read()


def test_packed_weights_are_ordered_behind_the_kernels_in_front():
    """a quantizer lets the next launch in (which may read packed weights at once) only behind its own wait for the previous
    one, and the grouped kernel copies nothing before its wait -- but in the calls that want the weights complete"""
    body = {n: b for _, n, b in kernels()}
    q = body["quant_act_fused_kernel"]
    wait = q.index("griddepcontrol.wait")
    lets_in = [(m.start() < wait, m.group(1)) for m in re.finditer(r"if \(([^()]*)\) asm volatile\(\"griddepcontrol\.launch_dependents", q)]
    assert lets_in == [(True, "early_next && tid == 0"), (False, "!early_next && tid == 0")]
    g = body["sdq_linear_group_kernel"]
    assert re.search(r"if \(p\.w_early && inl && c == 0\) \{\s*for [^{}]*seek\(\)", g)
    assert "if (!(p.w_early && wc)) ptx::griddep_wait();" in g
    src = open(os.path.join(CSRC, "sdq_linear.cu")).read()
    assert src.count("stream, true)") - src.count("stream, true); }") == src.count("w_early = 1") == 1
    assert 0 < src.index("w_early = 1") - src.index("&xq, stream, true)") < 100
    assert "out, stream, false); }" in open(os.path.join(CSRC, "sdq_quant_act.cu")).read()


def test_the_device_table_is_safe_to_share():
    """what host threads share per device is atomic, or filled in under a lock before an atomic word says so"""
    src = open(os.path.join(CSRC, "sdq_internal.h")).read()
    members = re.findall(r"^  ([\w:<>]+) (\w+)(?:\[\d\])?;", src[src.index("struct DeviceInfo {"):src.index("constexpr int MAX_DEVICES")], flags=re.M)
    assert {n for t, n in members if not t.startswith("std::atomic")} == {"sm_count", "pair_clusters"}
    pair = open(os.path.join(CSRC, "sdq_linear_pair.cu")).read()
    body = pair[pair.index("const int* pair_max_clusters(DeviceInfo* d)\n{"):]
    assert body.index("lock_guard") < body.index("&d->pair_clusters[k]") < body.index("d->clusters_known = 1")

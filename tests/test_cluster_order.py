"""A CTA's shared memory may be addressed by another CTA of its cluster only once both are known to run, which a cluster barrier
guarantees.  A missing wait shows on no run that happens to be slow enough, so the kernels' source is checked: in each kernel a
cluster wait stands before the first access to another CTA's shared memory."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_00608_b200", "csrc")
WAIT = re.compile(r"cluster_wait\(\)|cluster_sync_all\(\)|barrier\.cluster\.wait")
REMOTE = re.compile(r"st\.shared::cluster|copy_to_peer\(|mbar_arrive(?:_expect_tx)?_cluster\w*\(|commit2?_to_cluster\(|umma2_commit\w*\(")


def source():
    return {os.path.basename(p): re.sub(r"//[^\n]*", "", open(p).read()) for p in sorted(glob.glob(os.path.join(CSRC, "*.cu*")))}


def body_at(text, start):
    """The braces' content from the first one after `start`."""
    open_at = text.index("{", start)
    depth, i = 1, open_at + 1
    while depth:
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        i += 1
    return open_at, text[open_at:i]


def kernels():
    """(name, body) of every __global__ function."""
    for file, text in source().items():
        for m in re.finditer(r"__global__", text):
            open_at, body = body_at(text, m.end())
            name = re.search(r"(\w+)\s*\((?!\()[^()]*\)\s*$|(\w+)\s*\(const", text[m.end():open_at])
            yield file, name.group(1) or name.group(2), body


WITH_REMOTE = [(f, n, b) for f, n, b in kernels() if REMOTE.search(b)]


def test_the_cluster_kernels_are_found():
    names = {n for _, n, _ in WITH_REMOTE}
    assert {"gn_cluster_kernel", "conv_split_kernel", "conv_pair_kernel", "conv_f32_kernel", "conv_tc_kernel"} <= names, names


@pytest.mark.parametrize("file,name,body", WITH_REMOTE, ids=[n for _, n, _ in WITH_REMOTE])
def test_a_cluster_wait_precedes_remote_shared_memory(file, name, body):
    wait, remote = WAIT.search(body), REMOTE.search(body)
    assert wait and wait.start() < remote.start(), f"{file}: {name} reaches another CTA before it is known to run"


def test_what_other_ctas_send_is_waited_for_after_a_wait_gave_up():
    """The other CTAs of the cluster send their partial sums in any case: only the limit may end the wait for them."""
    text = source()["conv_cluster.cuh"]
    body = body_at(text, text.index("bool wait_cluster("))[1]
    assert "WAIT_LIMIT_CYCLES" in body
    assert not re.search(r"if\s*\(\s*\*abort_flag", body)


def test_loads_on_their_way_land_after_a_wait_gave_up():
    """A CTA whose wait ran into its limit must not end, or reuse the stages, while bulk loads are on their way into them."""
    for name in ("conv_split_kernel", "conv_pair_kernel", "conv_f32_kernel"):
        body = next(b for _, n, b in kernels() if n == name)
        landed = re.search(r"abort_flag\)\s*\{?\s*land_loads\(", body)
        assert landed, name
        if name == "conv_f32_kernel":                        # and nothing new is loaded
            assert re.search(r"!\*abort_flag\) \{\s*bars->issued = u \+ n_w;\s*load_weights\(", body)
        else:                                                # whatever wait it was: once the accumulators are complete, before the last arrival
            wait = body.rindex("mbar_wait(smem_u32(&bars->acc_full)", 0, landed.start())
            assert landed.start() - wait < 200 and landed.start() < body.rindex("cluster_arrive()")


BARRIER = re.compile(r"named_barrier_sync\(")


def enclosing(body, at):
    """What stands before each brace that is open at `at`: conditions, loops, lambdas, from the outermost in."""
    open_braces = []
    for i in range(at):
        if body[i] == "{":
            open_braces.append(i)
        elif body[i] == "}":
            open_braces.pop()
    return [re.split(r"[{}]|;(?![^()]*\))", body[:i])[-1].strip() for i in open_braces], open_braces


WITH_BARRIERS = [(f, n, b) for f, n, b in kernels() if BARRIER.search(b)]


@pytest.mark.parametrize("file,name,body", WITH_BARRIERS, ids=[n for _, n, _ in WITH_BARRIERS])
def test_every_warp_reaches_its_named_barriers_after_a_wait_gave_up(file, name, body):
    """Warps learn of a wait that gave up one by one.  If one of them left for the end of the kernel, the others would stand in their
    named barrier for good: whether a warp comes to a barrier must not depend on its waits, once it has waited at all."""
    for m in BARRIER.finditer(body):
        headers, braces = enclosing(body, m.start())
        if any(re.search(r"\bu == 0\b", h) for h in headers):        # the first pass of a loop: before any wait
            continue
        for h, at in zip(headers, braces):
            assert not re.search(r"\bok\b|abort_flag", h), f"{file}: {name}: a barrier under `{h}`"
            if re.match(r"(for|while)\b", h):
                loop = body_at(body, at)[1]
                assert not re.search(r"\b(break|return)\b", loop), f"{file}: {name}: a barrier in a loop that a warp may leave"


ONE_LANE = re.compile(r"\b(lane|tid|ptid) == |\bif \(lead\)|elected")
# (not conv_tc_kernel: its operand warps end where they leave; a vote per chunk cost 0.5 to 0.8 % of the large decodes)
WITH_ALIGNED = [(f, n, b) for f, n, b in kernels() if re.search(r"tmem_ld\d*\(|__syncwarp\(", b) and "mbar_wait" in b and n != "conv_tc_kernel"]


@pytest.mark.parametrize("file,name,body", WITH_ALIGNED, ids=[n for _, n, _ in WITH_ALIGNED])
def test_a_warp_decides_as_one_whether_a_wait_gave_up(file, name, body):
    """Where whole warps wait, the answer that they act on is voted on: lanes that part would meet the warp's barriers and tensor
    memory instructions at different places."""
    for m in re.finditer(r"\bmbar_wait(?:<[^>]*>)?\(", body):
        before = re.split(r"[;{}]", body[:m.start()])[-1]
        if "(void)" in before or "__all_sync(" in before or any(ONE_LANE.search(h) for h in enclosing(body, m.start())[0]):
            continue
        raise AssertionError(f"{file}: {name}: {before.strip()} mbar_wait(...) is not voted on")


@pytest.mark.parametrize("kernel", ["attn_tc_kernel", "gn_batch_kernel"])
def test_the_landing_starts_from_the_last_load(kernel):
    """The wait for everything to be consumed may itself give up half-way, and has moved on then: where the copies on their way are,
    the number of the loads says."""
    body = next(b for _, n, b in kernels() if n == kernel)
    assert re.search(r"land_loads\((?:bars->)?full, \w+, issued\)", body) and "--st" not in body


@pytest.mark.parametrize("kernel,bar,last", [("attn_tc_kernel", "drained", "tmem_dealloc2("), ("attn_small_kernel", "o_full", "tmem_dealloc("),
                                             ("conv_f32_tc_kernel", "acc_full", "tmem_dealloc(")])
def test_products_under_way_complete_before_tensor_memory_goes(kernel, bar, last):
    """After a wait gave up the issuing warp goes on or leaves, and nobody else waits for the products that it has in flight: it
    does so itself, and a flag that is already up does not end that wait."""
    body = next(b for _, n, b in kernels() if n == kernel)
    wait = re.search(r"if \(\*abort_flag\)[^;]*(?:;[^;]*){0,2}wait_cluster\(smem_u32\(&bars->" + bar, body)
    assert wait and wait.start() < body.rindex(last)

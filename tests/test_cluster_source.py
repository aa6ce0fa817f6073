"""Rules of thread-block clusters, checked in the text of the kernels (no GPU).

Shared memory of another CTA of a cluster may be accessed only once that CTA is known to run, which a
cluster barrier gives and co-scheduling alone does not.
"""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1504_06443_gb300", "csrc")
REMOTE = re.compile(r"map_shared_rank|\bmapa\.")
BARRIER = re.compile(r"\bcl\.sync\(\)|barrier\.cluster\.wait")


def functions(text):
    """[(name, body, is_kernel)] of the device functions and kernels of a source, comments taken out."""
    text = re.sub(r"//[^\n]*", "", text)
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    out = []
    for m in re.finditer(r"__(global|device)__[^;{]*?(\w+)\s*\([^{;]*\)\s*\{", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        name = m.group(2)
        if m.group(1) == "global":  # the name before the parameter list (attributes come before it)
            name = re.findall(r"(\w+)\s*\(", m.group(0))[-1]
        out.append((name, text[m.end():i], m.group(1) == "global"))
    return out


def first_events(body, helpers, depth=0):
    """The remote accesses and cluster barriers of a body in program order, helpers expanded in place."""
    pats = [REMOTE.pattern, BARRIER.pattern] + ([r"\b(?:%s)\s*\(" % "|".join(helpers)] if helpers else [])
    for m in re.finditer("|".join(pats), body):
        if REMOTE.fullmatch(m.group(0)):
            yield "remote"
        elif BARRIER.fullmatch(m.group(0)):
            yield "barrier"
        elif depth < 4:
            yield from first_events(helpers[m.group(0).rstrip("( \t")], helpers, depth + 1)


def cluster_kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        fns = functions(open(path).read())
        helpers = {n: b for n, b, k in fns if not k}
        for name, body, kernel in fns:
            if kernel and "remote" in list(first_events(body, helpers)):
                yield pytest.param(body, helpers, id=f"{os.path.basename(path)}:{name}")


def test_cluster_kernels_are_found():
    assert {p.id for p in cluster_kernels()} >= {"tri.cu:k_potrf_diag", "gemm_res.cu:k_res_gemm",
                                                 "tridiag_cluster.cu:k_trd_cluster",
                                                 "panel_cluster.cu:k_panel_qr_cluster"}


@pytest.mark.parametrize("body,helpers", list(cluster_kernels()))
def test_no_remote_access_before_a_cluster_barrier(body, helpers):
    assert next(first_events(body, helpers)) == "barrier"


def test_a_failed_wait_ends_the_panel_at_one_column():
    """The warp that accumulates T meets the row warps at one barrier a column only, so it may read the flag of a
    failed wait when warp 0 already stores the next column's.  The flag therefore names its column: were it a
    mere truth value, the warps would leave at different columns and wait at different barriers for good."""
    text = open(os.path.join(CSRC, "panel_cluster.cu")).read()
    body = {n: b for n, b, _ in functions(text)}["k_panel_qr_cluster"]
    stores = re.findall(r"sh\.fail\s*=(?!=)\s*([^;]+);", body)
    tests = re.findall(r"if\s*\(([^()]*sh\.fail[^()]*)\)", body)
    assert stores and tests
    assert set(stores) == {"0", "c + 1"} and set(tests) == {"sh.fail == c + 1"}


def test_the_copies_of_a_pair_are_waited_for():
    """The CTAs of a pair may give up at different steps.  Between the barrier after which both step counts
    stand and the one after which the CTAs retire, the first CTA waits for the copies of both."""
    text = open(os.path.join(CSRC, "gemm_res.cu")).read()
    body = {n: b for n, b, _ in functions(text)}["k_res_gemm"]
    tail = body[body.index("issued = g;"):]
    order = ["cluster_sync_all()", "pair_addr(smem_u32(&issued), rank ^ 1)", "mbar_expect_tx(bar_full", "mbar_wait_bounded(bar_full",
             "cluster_sync_all()", "tcgen05.dealloc"]
    at = 0
    for token in order:
        at = tail.index(token, at) + 1


@pytest.mark.parametrize("first,second", [(f, f + a) for f in (0, 1, 5, 6, 7, 12, 40) for a in range(-6, 7) if f + a >= 0])
def test_model_of_the_pairs_last_copies(first, second):
    """A model of those barriers (one arrival and an expected byte count a phase): with the first CTA at `first` steps and the
    second up to a ring ahead or behind, the closing steps leave no copy unexpected and no wait unmet."""
    R = 6
    done = max(min(first, second), max(first, second) - R)  # steps consumed: every older phase is complete
    phase, arrived, tx = [0] * R, [False] * R, [0] * R

    def settle(s):
        if arrived[s] and tx[s] == 0:
            phase[s], arrived[s] = phase[s] + 1, False

    def expect(s, n):
        assert not arrived[s]
        arrived[s], tx[s] = True, tx[s] + n
        settle(s)

    def land(s):
        tx[s] -= 1
        settle(s)

    for s in range(done):
        expect(s % R, 2), land(s % R), land(s % R)
    for s in range(done, first):
        expect(s % R, 2), land(s % R)
    for s in range(done, second):
        land(s % R)
    for s in range(second, first):  # the second CTA's missing copies
        land(s % R)
    for s in range(max(first - R, 0), max(first, second)):
        if s >= first:
            expect(s % R, 1)
        assert phase[s % R] % 2 != (s // R) % 2, "a wait that would not end"
    assert tx == [0] * R and not any(arrived)


@pytest.mark.parametrize("source,kernel", [("tri.cu", "k_potrf_diag"), ("tridiag_cluster.cu", "k_trd_cluster"),
                                           ("panel_cluster.cu", "k_panel_qr_cluster")])
def test_pushes_have_landed_before_a_cta_leaves(source, kernel):
    """A push (st.async) is complete only when the barrier it reports to says so.  Also after a timeout, when the main loop
    was left early, the CTAs wait for the pushes under way between two cluster barriers, and return behind the second."""
    text = open(os.path.join(CSRC, source)).read()
    bodies = {n: b for n, b, _ in functions(text)}
    body = bodies[kernel]
    if "st.async" not in body:  # the columns are a function of their own, called last
        body = body.rstrip("} \n") + bodies["trc_columns"]
    assert "st.async" in body
    barriers = [m.start() for m in re.finditer(r"cl\.sync\(\)", body)]
    drain = body.index("cluster_wait<true>")
    assert barriers[-2] < drain < barriers[-1]
    assert not re.search(r"\breturn\s*;", body[:barriers[-1]])
    assert "DRAIN" in open(os.path.join(CSRC, "cluster.cuh")).read()


def test_merges_order_numbers_only():
    """The orders that divide and conquer forms are used as indices, which comparisons with a NaN would leave unset: a
    merge looks for numbers that are not finite before it forms any."""
    text = open(os.path.join(CSRC, "dc.cu")).read()
    body = {n: b for n, b, _ in functions(text)}["k_prep"]
    check = body.index("__syncthreads_or(bad)")
    assert "0x7FF" in body[:check] and "atomicCAS(st" in body[check:check + 120]
    assert check < body.index("w.perm[")

"""The unit queue of the SM-pair weight gradients, by reading (CPU only): the leader CTA
asks for units ahead into a ring of slots, the answers land in both CTAs, and a slot is
asked into again once the leader's `empty` barrier has counted its readers.

A small model of that protocol (one role a CTA, a ring of two, every interleaving) shows
which readers have to be among them, and the arrivals are counted in the kernels' source."""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_16188_gb300", "csrc")
DEPTH, LAST = 2, 4  # ring slots; the answer that ends the loops


def explore(peer_scheduler_frees: bool):
    """Every reachable wrong read or dead end, as a set of texts.

    State: leader scheduler's index; peer scheduler's index and whether it stands between its
    wait and its read; each CTA's role index; the peer's armed answers; what each CTA's slots
    hold; the leader slots' arrivals.  A scheduler waits for the answer that it asked for, so
    the leader is one step an answer; the answer lands in both CTAs in that step."""
    bad, seen = set(), set()
    need = 3 if peer_scheduler_frees else 2  # leader's role, peer's role (+ peer's scheduler)
    # (leader sched, peer sched, peer between wait and read, leader role, peer role, peer slots, arrivals a slot)
    start = (0, 0, False, 0, 0, (-1,) * DEPTH, (need,) * DEPTH)
    todo = [start]
    while todo:
        st = todo.pop()
        if st in seen:
            continue
        seen.add(st)
        ls, ps, mid, lr, pr, slots, arr = st
        nxt = []

        def free(arr, s):
            return arr[:s] + (arr[s] + 1,) + arr[s + 1:]

        s = ls % DEPTH
        if ls <= LAST and arr[s] >= need:  # the leader asks and the answer lands in both CTAs
            nxt.append((ls + 1, ps, mid, lr, pr, slots[:s] + (ls,) + slots[s + 1:], arr[:s] + (0,) + arr[s + 1:]))
        # the peer's scheduler: arms once its own roles are done with the slot and waits for the answer ...
        if ps <= LAST and not mid and ls > ps and pr > ps - DEPTH:
            nxt.append((ls, ps, True, lr, pr, slots, arr))
        if mid:  # ... then reads it
            got = slots[ps % DEPTH]
            if got != ps:
                bad.add("the peer's scheduler reads answer %d in the place of %d" % (got, ps))
            else:
                nxt.append((ls, ps + 1, False, lr, pr, slots, free(arr, ps % DEPTH) if peer_scheduler_frees else arr))
        if lr <= LAST and ls > lr:
            nxt.append((ls, ps, mid, lr + 1, pr, slots, free(arr, lr % DEPTH)))
        armed = ps + 1 if mid else ps  # the peer's role needs its own barrier armed by its scheduler
        if pr <= LAST and ls > pr and armed > pr:
            if slots[pr % DEPTH] != pr:
                bad.add("a peer's role reads answer %d in the place of %d" % (slots[pr % DEPTH], pr))
            nxt.append((ls, ps, mid, lr, pr + 1, slots, free(arr, pr % DEPTH)))
        if not nxt and min(ls, ps, lr, pr) <= LAST and not mid:
            bad.add("dead end")
        todo += nxt
    return bad


def test_the_peers_scheduler_is_a_reader():
    assert any("peer's scheduler" in b for b in explore(False))
    assert explore(True) == set()


@pytest.mark.parametrize("kernel", ["wgrad_pair_kernel", "wgrad_pair_stream_kernel"])
def test_the_kernels_count_every_reader(kernel):
    queue = open(os.path.join(CSRC, "gemm_tc.cuh")).read()
    pair = open(os.path.join(CSRC, "gemm_tc2.cuh")).read()
    roles = int(re.search(r"constexpr int PAIR_ROLES = (\d+);", pair).group(1))
    body = pair[pair.index("\n%s(" % kernel):]
    count = re.search(r"clc_init\(clc, leader \? ([^:]+) : ([^)]+)\)", body)
    leader, peer = (eval(e, {"PAIR_ROLES": roles}) for e in count.groups())
    assert peer == roles
    assert leader == 2 * roles + 1  # both CTAs' roles and the peer's scheduler
    # the scheduler frees the leader's slot after its read of it, and before it goes on
    sched = queue[queue.index("void clc_scheduler("):]
    sched = sched[:sched.index("pdl_launch_dependents();")]
    read = sched.index("more = clc_query(")
    assert "mbar_arrive_remote(leader_empty" in sched[read:]
    assert re.search(r"clc_scheduler[^;(]*\(clc, leader_empty,", body)


# clc_scheduler as host code, its primitives played by a script: answer i holds a CTA while i < hold,
# the wait for answer `fail` gives up, and that answer lands late or never.
HARNESS = r"""
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#define __device__
#define __forceinline__ inline
struct ClcQueue { int resp[%(depth)d + 1]; uint64_t full[%(depth)d], empty[%(depth)d], drain; };
constexpr int CLC_DEPTH = %(depth)d;
static ClcQueue q;
static int hold, fail, lands, asked, waits, wrong;
static bool unread, none;
static unsigned long long now;
static uint32_t smem_u32(const void *p) { return (uint32_t)((const char *)p - (const char *)&q); }
static unsigned long long global_ns() { return now += 10000000ull; }
static bool is(uint32_t bar, const uint64_t *b) { return bar >= smem_u32(b) && bar < smem_u32(b + CLC_DEPTH); }
static bool wait_phase(uint32_t bar, uint32_t, volatile int *, int *) { return !(is(bar, q.full) && waits++ == fail); }
static bool mbar_try_wait(uint32_t bar, uint32_t) { return bar == smem_u32(&q.drain) || lands; }
static void mbar_expect_tx(uint32_t, uint32_t) {}
static void mbar_arrive_remote(uint32_t) {}
static void fence_proxy_async() {}
static void pdl_launch_dependents() {}
template <bool> void clc_try(uint32_t, uint32_t) {
    if (unread || none) ++wrong;  // asked before the last answer was read, or after "none left"
    unread = true;
    ++asked;
}
static bool clc_query(uint32_t, uint32_t &x) {
    unread = false;
    x = 0;
    none = asked > hold;
    return !none;
}
%(code)s
int main(int, char **v) {
    hold = atoi(v[1]), fail = atoi(v[2]), lands = atoi(v[3]);
    int flag = 0;
    clc_scheduler%(args)s;
    printf("%%d %%d\n", wrong, asked);
}
"""


@pytest.fixture(scope="module")
def scheduler(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no host compiler")
    src = open(os.path.join(CSRC, "gemm_tc.cuh")).read()
    at = src.index("clc_scheduler(ClcQueue &q")
    begin = src.rindex("\n//", 0, at)  # behind the comment above it
    code = src[src.index("\n", begin + 1):src.index("\n}\n", at) + 3].strip()
    depth = int(re.search(r"constexpr int CLC_DEPTH = (\d+);", src).group(1))
    args = "<true>" if code.startswith("template") else ""
    args += "(q, %s, &flag, nullptr)" % ("true" if "bool issue," in code else "0u")
    d = tmp_path_factory.mktemp("sched")
    (d / "s.cpp").write_text(HARNESS % {"depth": depth, "code": code, "args": args})
    subprocess.run(["g++", "-std=c++17", "-O1", "-o", str(d / "s"), str(d / "s.cpp")], check=True)
    return lambda *a: [int(w) for w in subprocess.run([str(d / "s"), *map(str, a)], check=True, capture_output=True,
                                                      text=True).stdout.split()]


@pytest.mark.parametrize("hold", [0, 1, 7])
@pytest.mark.parametrize("fail", [-1, 0, 1, 7])
@pytest.mark.parametrize("lands", [0, 1])
def test_the_scheduler_never_asks_past_the_last_answer(scheduler, hold, fail, lands):
    wrong, asked = scheduler(hold, fail, lands)
    assert wrong == 0
    if fail < 0 or lands:  # every CTA that was left has been taken, and "none left" read once
        assert asked == hold + 1

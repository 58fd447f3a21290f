"""The barriers of the tcgen05 attention kernels, every interleaving of their roles: no wait is passed before its event, and none
is missed.  The steps' barriers and parities, the rings and the producers' rule are the kernels' own (csrc/attn_ring.h, compiled
here); the roles' order of waits and arrivals is restated from csrc/attn_tcgen05.cuh: `explore` for attn_tcgen05_kernel (128-token
blocks), `explore_b64` for attn_tcgen05_b64_kernel (64-token blocks)."""
import ctypes
import os
import re
import subprocess

import pytest

from paper_2609_32420_b200 import build


@pytest.fixture(scope="module")
def ring(tmp_path_factory):
    d = tmp_path_factory.mktemp("ring")
    src, lib = os.path.join(d, "ring.cpp"), os.path.join(d, "ring.so")
    with open(src, "w") as f:
        f.write('#include "attn_ring.h"\nusing namespace carnator::tc;\nextern "C" int bar(int i) { return step_bar(i); }\n'
                'extern "C" int parity(int i) { return int(step_parity(i)); }\nextern "C" int stages() { return kStages; }\n'
                '// c0, c1: phases that the two barriers have completed\n'
                'extern "C" int slot_free(int u, int c0, int c1) { return slot_is_free(u, [=](int b, uint32_t p) { return ((b ? c1 : c0) & 1) != int(p); }); }\n'
                'template <int N> static int at(int i) { Ring<N> r; while (i--) r.next(); return 2 * r.slot + int(r.phase); }\n'
                '// slot and phase of step i in a ring of n slots\n'
                'extern "C" int ring_at(int n, int i) { return n == 2 ? at<2>(i) : n == 3 ? at<3>(i) : at<4>(i); }\n')
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", build.CSRC, "-o", lib, src], check=True)
    return ctypes.CDLL(lib)


class Stuck(Exception):
    pass


class Early(Exception):
    pass


def explore(T, stages, bar, parity, slot_free, form, warps=1):
    """Walks all reachable states of one block of T steps.  `bar`, `parity`: barrier of a step for "scores there" and "P V
    done"; `slot_free`: the producers' rule.  `form`, the attn_tcgen05_kernel's own: "late" gives the scores' buffer back once the reference
    is published, "rescaling" like "late" with P V of the step before awaited in front of the reference, in every step.  Two orders that
    the same barriers allow and that no kernel has: "early" gives the buffer back on reading the scores, "low" with P V of the step
    itself (the scores' columns hold a part of P until then).

    Counters of a state: K tiles asked for / landed, V tiles asked for / landed, Q K^T issued / completed, P V issued /
    completed, then per softmax warp (group-major) its operations done.  Each role's next operation follows from its counter."""
    kslot, kpar = lambda i: i % stages, lambda i: (i // stages) & 1          # tiles: one barrier per ring slot
    half, hpar = lambda i: i & 1, lambda i: (i >> 1) & 1                     # one barrier per softmax group
    n_ops = 3                                                                # operations of a softmax warp per step (below)

    def passed(at, par, done, i, event):
        """A wait for event i of a kind whose events 0 .. done - 1 have happened, event j on barrier at(j)."""
        c = sum(1 for j in range(done) if at(j) == at(i))                  # phases this barrier has completed
        ok = (c & 1) != par(i)
        if ok and i >= done:
            raise Early(f"{event} {i} taken for done at {done}")
        return ok

    def free(done, u):
        """A producer's wait for step u of a kind whose steps 0 .. done - 1 have completed."""
        ok = slot_free(u, (done + 1) // 2, done // 2)
        if ok and u >= done:
            raise Early(f"slot of step {u} taken for free at {done}")
        return ok

    def group_done(st, g, op):
        """Steps of group g whose operation `op` all its warps have done, as a step number: first one not done."""
        n = min((o - op + n_ops - 1) // n_ops if o > op else 0 for o in st[8 + g * warps: 8 + (g + 1) * warps])
        return g + 2 * n

    def count(st, op):
        """How many of steps 0, 1, 2, .. have done operation `op`, per group as separate barriers: steps below are done."""
        return [group_done(st, g, op) for g in (0, 1)]

    def group_wait(st, op, i, event):                                        # barriers indexed by the group
        g = i & 1
        done = (count(st, op)[g] - g) // 2                                   # phases of the group's barrier
        ok = (done & 1) != hpar(i)
        if ok and i // 2 >= done:
            raise Early(f"{event} {i} taken for done")
        return ok

    def moves(st):
        ka, kl, va, vl, qi, qd, pi, pd = st[:8]

        def step(k, v=1):
            n = list(st)
            n[k] += v
            return tuple(n)
        if ka < T and (ka < stages or free(qd, ka - stages)):
            yield step(0)
        if kl < ka:
            yield step(1)
        if va < T and (va < stages or free(pd, va - stages)):
            yield step(2)
        if vl < va:
            yield step(3)
        sfree_op = 0 if form == "early" else 1
        if qi < T and passed(kslot, kpar, kl, qi, "K tile") and \
                (qi < 2 or (passed(bar, parity, pd, qi - 2, "P V") if form == "low" else group_wait(st, sfree_op, qi - 2, "scores read"))):
            yield step(4)
        if qd < qi:
            yield step(5)
        if pi < T and passed(kslot, kpar, vl, pi, "V tile") and group_wait(st, 2, pi, "P"):
            yield step(6)
        if pd < pi:
            yield step(7)
        for g in (0, 1):
            for w in range(warps):
                k = 8 + g * warps + w
                i, op = g + 2 * (st[k] // n_ops), st[k] % n_ops
                if i >= T:
                    continue
                if op == 0:          # scores of step i are there; "early": S given back
                    ok = passed(bar, parity, qd, i, "Q K^T")
                elif op == 1:        # reference of step i - 1 (from the same warp of the other group), own one published; "late": S given back
                    o = st[8 + (g ^ 1) * warps + w]
                    refs = (o + 1) // n_ops                                  # steps of the other group with the reference published
                    ok = i == 0 or (refs > 0 and (g ^ 1) + 2 * (refs - 1) >= i - 1)
                    ok = ok and (form != "rescaling" or i == 0 or passed(bar, parity, pd, i - 1, "P V"))
                else:                # P V of step i - 1 has read P; P of step i handed over
                    ok = i == 0 or passed(bar, parity, pd, i - 1, "P V")
                if ok:
                    yield step(k)

    start = (0,) * (8 + 2 * warps)
    end = (T,) * 8 + tuple(n_ops * len(range(g, T, 2)) for g in (0, 1) for _ in range(warps))
    seen, todo = {start}, [start]
    while todo:
        st = todo.pop()
        nxt = list(moves(st))
        if not nxt and st != end:
            raise Stuck(st)
        for n in nxt:
            if n not in seen:
                seen.add(n)
                todo.append(n)
    assert end in seen
    return len(seen)


def explore_b64(T, at, v_stages, rescaling, warps=1, k_stages=3, qk_waits=True):
    """The same for the kernel of three softmax groups: a group leaves P in the columns of its scores, so that "P V of step i has
    completed" (a barrier per group) frees the score buffer and the V slot, and Q K^T of step i + 3 waits for it.  Producers watch
    the one barrier of the step that last used the slot.  `at`: slot and phase of a step in a ring of n slots, as 2 * slot + phase;
    `rescaling`: P V of the step before is awaited behind the reference, in every step.

    State: K tiles asked for, bits of those landed (in any order), the same for V, Q K^T issued / completed, P V issued / completed,
    then per softmax warp (group-major) its operations done (three per step: scores there; reference taken over and published; P
    handed over)."""
    G, n_ops = 3, 3
    slot, phase = lambda n, i: at(n, i) >> 1, lambda n, i: at(n, i) & 1

    def passed(n, par, step, done, what):
        """A wait with parity `par` for event `step` on a ring of n barriers; done(j): has event j happened?"""
        c = sum(1 for j in range(step % n, T, n) if done(j))               # phases that this barrier has completed
        ok = (c & 1) != par
        if ok and not done(step):
            raise Early(f"{what} {step}")
        return ok

    def moves(st):
        ka, kl, va, vl, qi, qd, pi, pd = st[:8]
        ops = lambda g, w: st[8 + g * warps + w]
        below = lambda n: (lambda j: j < n)
        landed = lambda bits: (lambda j: bool(bits >> j & 1))

        def step(k, v=None):
            n = list(st)
            n[k] = st[k] + 1 if v is None else v
            return tuple(n)
        # producers: step u = i - stages, counted by Ring<3> from the first step that waits
        if ka < T and (ka < k_stages or passed(G, phase(G, ka - k_stages), ka - k_stages, below(qd), "K slot of step")):
            yield step(0)
        if va < T and (va < v_stages or passed(G, phase(G, va - v_stages), va - v_stages, below(pd), "V slot of step")):
            yield step(2)
        for j in range(T):
            if j < ka and not kl >> j & 1:
                yield step(1, kl | 1 << j)
            if j < va and not vl >> j & 1:
                yield step(3, vl | 1 << j)
        if qi < T and passed(k_stages, phase(k_stages, qi), qi, landed(kl), "K tile") and \
                (qi < G or not qk_waits or passed(G, phase(G, qi) ^ 1, qi - G, below(pd), "P V")):
            yield step(4)
        if qd < qi:
            yield step(5)
        handed = lambda j: all(ops(j % G, w) >= n_ops * (j // G) + 3 for w in range(warps))
        if pi < T and passed(v_stages, phase(v_stages, pi), pi, landed(vl), "V tile") and passed(G, phase(G, pi), pi, handed, "P"):
            yield step(6)
        if pd < pi:
            yield step(7)
        for g in range(G):
            for w in range(warps):
                o = ops(g, w)
                i, op, ph = g + G * (o // n_ops), o % n_ops, o // n_ops & 1
                if i >= T:
                    continue
                ph_prev = ph ^ 1 if g == 0 else ph                         # phase of step i - 1 on the barriers of its group
                published = lambda j: ops(j % G, w) >= n_ops * (j // G) + 2
                if op == 0:
                    ok = passed(G, ph, i, below(qd), "Q K^T")
                elif op == 1:
                    ok = i == 0 or passed(G, ph_prev, i - 1, published, "reference")
                else:
                    ok = i == 0 or not rescaling or passed(G, ph_prev, i - 1, below(pd), "P V")
                if ok:
                    yield step(8 + g * warps + w)

    start, full = (0,) * (8 + G * warps), (1 << T) - 1
    end = (T, full, T, full, T, T, T, T) + tuple(n_ops * len(range(g, T, G)) for g in range(G) for _ in range(warps))
    seen, todo = {start}, [start]
    while todo:
        st = todo.pop()
        nxt = list(moves(st))
        if not nxt and st != end:
            raise Stuck(st)
        for n in nxt:
            if n not in seen:
                seen.add(n)
                todo.append(n)
    assert end in seen
    return len(seen)


@pytest.mark.parametrize("form,T,warps", [("early", 9, 1), ("late", 9, 1), ("rescaling", 9, 1), ("low", 9, 1), ("early", 6, 2), ("late", 6, 2), ("low", 6, 2), ("rescaling", 6, 2)])
def test_every_interleaving_ends_and_no_wait_is_passed_early(ring, form, T, warps):
    assert explore(T, ring.stages(), ring.bar, ring.parity, ring.slot_free, form, warps) > 1000


@pytest.mark.parametrize("form", ["early", "late", "rescaling", "low"])
def test_a_producer_that_watches_one_barrier_can_miss_its_phase(ring, form):
    """The search finds the fault it is there for: a step and the one two steps on share a barrier."""
    one = lambda u, c0, c1: ((c1 if u & 1 else c0) & 1) != ((u >> 1) & 1)
    with pytest.raises(Stuck):
        explore(6, ring.stages(), ring.bar, ring.parity, one, form)


@pytest.mark.parametrize("T,v_stages,rescaling,warps", [(8, 2, False, 1), (8, 2, True, 1), (8, 3, False, 1), (8, 3, True, 1), (5, 2, True, 2), (5, 3, False, 2)])
def test_three_groups_every_interleaving_ends(ring, T, v_stages, rescaling, warps):
    """V rings of the head dimensions 128 (two slots) and 64 (three)."""
    assert explore_b64(T, ring.ring_at, v_stages, rescaling, warps) > 1000


@pytest.mark.parametrize("change", [dict(v_stages=4), dict(k_stages=4), dict(qk_waits=False)])
def test_three_groups_the_search_finds_faults(ring, change):
    """A fourth slot lets the step that shares the awaited barrier run ahead of the producer (the kernel asserts that there are at
    most as many slots as groups); without the wait for P V, Q K^T overtakes the group that reads its scores."""
    with pytest.raises((Stuck, Early)):
        explore_b64(8, ring.ring_at, **dict(dict(v_stages=3, rescaling=False), **change))


def test_every_wait_that_orders_tensor_memory_is_followed_by_a_fence():
    """What another role's products or loads did to tensor memory is ordered before this role's accesses by the barrier and by
    tcgen05.fence::after_thread_sync behind the wait: in the source, a fence between each such wait and the next access."""
    with open(os.path.join(build.CSRC, "attn_tcgen05.cuh")) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    text = text[text.index("attn_tcgen05_kernel("):text.index("wait_timeout_selftest_kernel")]
    waits = [m.end() for m in re.finditer(r"mbar_wait_warp\((?:kLowInS \? )?bar_(?:sfull|sfree|pvdone|pfull|q\b|o\b)", text)]
    assert len(waits) >= 8
    for at in waits:
        access = re.compile(r"\b(?:tmem_ld|tmem_st|mma_ts_el|mma_ss_el)").search(text, at)
        fence = text.find("tc_fence_after()", at)
        assert access is None or at < fence < access.start(), text[at - 60:access.end() + 20]


def test_every_load_from_tensor_memory_is_handed_on_by_its_wait():
    """Arithmetic on loaded registers is ordered behind the wait only if the wait names them; one without names leaves that to the
    compiler's schedule (a row maximum of registers that are still being filled, without an error)."""
    for name in sorted(os.listdir(build.CSRC)):
        with open(os.path.join(build.CSRC, name)) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        loads = re.findall(r"(?:tmem_ld(?:16|32)\([^;]*, |float )(\w+(?:\[\w+\])?)(?:\)| = tmem_ld1\([^;]*\));", text)
        calls = [m.group(1) for m in re.finditer(r"(?<!void )tmem_wait_ld\(([^;]*)\);", text)]
        named = {v.strip() for c in calls for v in c.split(",")}
        named |= {"s[c]"} if {"s[0]", "s[1]", "s[2]", "s[3]"} <= named else set()
        assert "" not in named and set(loads) <= named, (name, loads, calls)
        assert text.count("tcgen05.wait::ld") == (2 if name == "attn_tcgen05.cuh" else 0), name


def test_the_abort_flag_is_raised_behind_its_report():
    """The first report stands, and a role that sees the flag while it waits reports a time-out: whoever raises the flag for another
    reason has to have reported it."""
    with open(os.path.join(build.CSRC, "attn_tcgen05.cuh")) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    text = text[text.index("attn_tcgen05_kernel("):text.index("wait_timeout_selftest_kernel")]
    raised = [m.start() for m in re.finditer(r"\*abortp = 1", text)]
    assert raised
    for at in raised:
        assert re.search(r"set_status\([^;]*\);\s*$", text[:at]), text[at - 80:at + 20]

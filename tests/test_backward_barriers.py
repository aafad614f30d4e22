"""The backward kernel's barriers, on the CPU: no wait may miss its phase.

A wait names a phase by its parity, so it is only sound if the phase after it
cannot complete before the waiting warp has looked: the warp would then wait
for a parity that has flipped back, until its budget runs out.  The model runs
every role of a CTA with one role held at one of its waits for good and the
others as far as they get (an arrival never hinders another role, so this is
the furthest the barrier can be driven); the held barrier must not get past
the phase that the wait names.  The roles' operations are taken from the
kernel's source in their order, and checked against the list written here.
"""
import os
import re

import pytest

SOURCE = os.path.join(os.path.dirname(__file__), "..", "paper_2608_01127_gb300", "csrc", "mw_bwd.cu")
OP = re.compile(r"(warp_wait|mbar_wait|umma_commit|mbar_arrive_expect_tx|mbar_arrive)\(&?(\w+)(\[[^\]]*\])?")


def source():
    with open(SOURCE) as f:
        text = f.read()
    return text[text.index("bca_bwd_kernel"):text.index("bwd_pre_kernel")]


def ops(text):
    return [("wait" if "wait" in m[1] else "arrive", m[2]) for m in OP.finditer(text)]


def between(text, first, last):
    start = text.index(first)
    return text[start:text.index(last, start)]


def constant(text, name, d64):
    m = re.search(rf"{name} = \(D == 64\) \? (\d+) : (\d+)", text)
    return int(m[1] if d64 else m[2])


@pytest.fixture(scope="module")
def layout():
    with open(SOURCE) as f:
        return f.read()


def buffers(kernel, bar, dims):
    """Barriers behind a name, from how it is initialised."""
    m = re.search(rf"for \(int (\w) = 0; \1 < ([\w:]+); \+\+\1\) (?:\{{[^}}]*?)?mbar_init\(&{bar}\[\1\]", kernel)
    return dims[m[2].replace("L::", "")] if m else 1


def roles(kernel, layout, d64, n):
    """Per role (copies, operations); an operation is (kind, barrier, index, phase)."""
    nq, nd, nb = (constant(layout, c, d64) for c in ("QSTAGES", "DOSTAGES", "DS_BUFS"))
    dims = {"NQ": nq, "ND": nd, "DS_BUFS": nb}
    count = {b: buffers(kernel, b, dims) for b in
             ("q_full", "q_empty", "do_full", "do_empty", "p_ready", "ds_free")}

    def at(kind, bar, j, lag=0):  # the j-th use of a barrier (lag: buffers' uses before it)
        c = count.get(bar, 1)
        return (kind, bar, j % c, j // c - lag)

    def keep(op):
        return op[0] != "wait" or op[3] >= 0

    tma, a, b, pds, drain = [("arrive", "kv_full", 0, 0)], [at("wait", "kv_full", 0)], [at("wait", "kv_full", 0)], [], []
    for j in range(n):
        more = j + 1 < n
        tma += [at("wait", "q_empty", j, 1), at("arrive", "q_full", j),
                at("wait", "do_empty", j, 1), at("arrive", "do_full", j)]
        if d64:
            if j == 0:
                a += [at("wait", "q_full", 0), at("arrive", "s_full", 0),
                      at("wait", "do_full", 0), at("arrive", "dp_full", 0)]
            if more:
                a += [at("wait", "s_free", j), at("wait", "q_full", j + 1), at("arrive", "s_full", j + 1)]
            a += [at("wait", "pt_ready", j), at("arrive", "do_empty", j)]
            if more:
                a += [at("wait", "dp_free", j), at("wait", "do_full", j + 1), at("arrive", "dp_full", j + 1)]
            b += [at("wait", "p_ready", j)] + ([at("wait", "dq_free", j - 1)] if j else [])
            pds += [at("wait", "s_full", j), at("arrive", "s_free", j), at("wait", "dp_full", j),
                    at("arrive", "pt_ready", j), at("wait", "ds_free", j, 1), at("arrive", "dp_free", j),
                    at("arrive", "p_ready", j)]
        else:
            if j == 0:
                a += [at("wait", "q_full", 0), at("arrive", "s_full", 0)]
            a += [at("wait", "do_full", j)] + ([at("wait", "dq_free", j - 1)] if j else [])
            a += [at("arrive", "dp_full", j), at("wait", "pt_ready", j), at("arrive", "do_empty", j)]
            if more:
                a += [at("wait", "q_full", j + 1), at("arrive", "s_full", j + 1)]
            b += [at("wait", "p_ready", j)]
            pds += [at("wait", "s_full", j), at("arrive", "pt_ready", j), at("wait", "dp_full", j),
                    at("wait", "ds_free", j, 1), at("arrive", "p_ready", j)]
        b += [at("arrive", "dq_full", j), at("arrive", "q_empty", j), at("arrive", "ds_free", j)]
        drain += [at("wait", "dq_full", j), at("arrive", "dq_free", j)]
    a.append(("arrive", "dkv_full", 0, 0))
    b.append(("arrive", "dkv_full", 0, 0))
    pds.append(("wait", "dkv_full", 0, 0))
    return [(k, list(filter(keep, o))) for k, o in ((1, tma), (1, a), (1, b), (8, pds), (4, drain))]


def expected_arrivals(kernel):
    return {m[1]: int(m[2]) for m in re.finditer(r"mbar_init\(&?(\w+)(?:\[\w\])?, (\d+)\)", kernel)}


def run(warps, arrivals, held=None, at_op=None):
    """Completed phases per barrier once no warp gets further, warp `held`
    kept at its operation `at_op`; and whether all others finished."""
    got, pos = {}, [0] * len(warps)
    moved = True
    while moved:
        moved = False
        for w, seq in enumerate(warps):
            while pos[w] < len(seq) and not (w == held and pos[w] == at_op):
                kind, bar, idx, phase = seq[pos[w]]
                n = got.get((bar, idx), 0)
                if kind == "wait" and n // arrivals[bar] <= phase:
                    break
                if kind == "arrive":
                    got[bar, idx] = n + 1
                pos[w] += 1
                moved = True
    return {k: v // arrivals[k[0]] for k, v in got.items()}, all(p == len(s) for p, s in zip(pos, warps))


VARIANTS = pytest.mark.parametrize("d64", [True, False], ids=["d64", "d128"])


@VARIANTS
@pytest.mark.parametrize("n", [1, 2, 3, 4, 7])
def test_no_wait_can_miss_its_phase(layout, d64, n):
    kernel = source()
    arrivals = expected_arrivals(kernel)
    warps, held = [], []
    for copies, seq in roles(kernel, layout, d64, n):
        held.append(len(warps))  # one warp of each role (the others are like it)
        warps += [seq] * copies
    _, finished = run(warps, arrivals)
    assert finished
    for w in held:
        for i, (kind, bar, idx, phase) in enumerate(warps[w]):
            if kind == "wait":
                done, _ = run(warps, arrivals, w, i)
                assert done.get((bar, idx), 0) <= phase + 1, \
                    f"{bar}[{idx}] gets past phase {phase} before a warp that waits for it has looked"


@VARIANTS
def test_the_model_is_the_kernel(layout, d64):
    """The roles' operations in the order of the source, one step each."""
    kernel = source()
    issuers = between(kernel, "bool ok = warp_wait(kv_full", "one arrival per issuing warp")
    paired, separate = issuers.split("} else {\n        if (ok && role_a)")
    if d64:
        assert ops("if (ok && role_a)" + separate) == [
            ("wait", "q_full"), ("arrive", "s_full"), ("wait", "do_full"), ("arrive", "dp_full"),
            ("wait", "s_free"), ("wait", "q_full"), ("arrive", "s_full"),
            ("wait", "pt_ready"), ("arrive", "do_empty"),
            ("wait", "dp_free"), ("wait", "do_full"), ("arrive", "dp_full"),
            ("wait", "p_ready"), ("wait", "dq_free"), ("arrive", "dq_full"), ("arrive", "q_empty"),
            ("arrive", "ds_free"), ("arrive", "dkv_full")]
    else:
        assert ops(paired) == [
            ("wait", "kv_full"), ("wait", "q_full"), ("arrive", "s_full"), ("wait", "do_full"),
            ("wait", "dq_free"), ("arrive", "dp_full"), ("wait", "pt_ready"), ("arrive", "do_empty"),
            ("wait", "q_full"), ("arrive", "s_full"),
            ("wait", "p_ready"), ("arrive", "dq_full"), ("arrive", "q_empty"), ("arrive", "ds_free")]
    pds = ops(between(kernel, "regs_inc<L::REGS_PDS>", "regs_inc<L::REGS_DRAIN>"))
    # (s_free, the first dp_full and dp_free: d = 64; the second dp_full: d = 128)
    assert pds == [("wait", "s_full"), ("arrive", "s_free"), ("wait", "dp_full"), ("arrive", "pt_ready"),
                   ("wait", "dp_full"), ("wait", "ds_free"), ("arrive", "dp_free"), ("arrive", "p_ready"),
                   ("wait", "dkv_full")]
    assert ops(between(kernel, "regs_dec<L::REGS_DRAIN>", "tmem_dealloc")) == [
        ("wait", "dq_full"), ("arrive", "dq_free"), ("arrive", "dq_free")]
    assert ops(between(kernel, "TMA producer", "MMA issuers")) == [
        ("arrive", "kv_full"), ("wait", "q_empty"), ("arrive", "q_full"), ("wait", "do_empty"),
        ("arrive", "do_full")]
    # every wait on a barrier with buffers takes the buffer of its step
    for bar in ("p_ready", "ds_free"):
        uses = set(m[1] for m in re.finditer(rf"(?:umma_commit|warp_wait|mbar_arrive)\(&?{bar}(\[[^\]]*\])?", kernel))
        assert uses in ({"[j % L::DS_BUFS]"}, {"[j % L::DS_BUFS]", "[buf]"})

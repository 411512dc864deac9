"""The order of the cluster exchanges of the resident BCCG solve (k_resident.cu), played on the CPU:
no CTA may send into a buffer of another before that one has read what the buffer held, however late
a CTA or a message is, with the CTAs without mode columns (which wait for no modes) of every size.
The slots of the sums are those of the kernel's source."""
import os
import random
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2203_16467_gb300", "csrc",
                   "k_resident.cu")
SIZES = [(nx, ny) for nx in (16, 32, 64, 128, 256) for ny in (16, 32, 64, 128, 256) if nx * ny <= 1 << 14]


def slots():
    """Slots of the sums of one iteration: p.Jp, the iterate's eight, the explicit residual's seven."""
    body = open(SRC).read().split("k_res_bccg(")[1].split("k_res_lap(")[0]
    one = re.findall(r"one_sum<W, CS>\(s, sh, (\d)", body)
    sent = re.findall(r"many_sums<(\d), W, CS>\(s, sh, (\d)", body)
    taken = re.findall(r"take_many<(\d), CS>\(s, (\d)", body)
    assert len(one) == 1 and sent == taken and [n for n, _ in sent] == ["8", "7"]
    return "sum" + one[0], "sum" + sent[0][1], "sum" + sent[1][1]


def program(own, explicit):
    """What one CTA does: ("send", buffer), ("wait", buffer), ("read", buffer)."""
    p_jp, eight, seven = slots()
    operate = [("send", "modes"), ("wait", "modes"), ("read", "modes"), ("send", "rows")]
    rows = [("wait", "rows"), ("read", "rows")]
    prog = []
    for full in explicit:
        prog += operate + [("send", p_jp)] + rows + [("wait", p_jp), ("read", p_jp)]
        prog += [("send", eight), ("wait", eight), ("read", eight)]
        if full:
            prog += operate + rows + [("send", seven), ("wait", seven), ("read", seven)]
    if not own:   # no modes to wait for, no rows to send
        prog = [op for op in prog if op not in (("wait", "modes"), ("read", "modes"), ("send", "rows"))]
    return prog


def play(nx, ny, seed):
    cs = 16 if nx * ny >= 1024 else 8
    nm = nx // 2 + 1
    per = (nm + cs - 1) // cs
    own = [min(per, nm - c * per) > 0 for c in range(cs)]
    rng = random.Random(seed)
    explicit = [rng.random() < 0.5 for _ in range(6)]
    progs = [program(o, explicit) for o in own]
    owners = [c for c in range(cs) if own[c]]
    late = rng.randrange(cs)                 # a CTA that runs when no other can
    pc = [0] * cs
    sent = [dict() for _ in range(cs)]       # exchanges of a buffer sent by a CTA
    read = [dict() for _ in range(cs)]       # exchanges of a buffer of this CTA that it has read
    arrived = [dict() for _ in range(cs)]    # (buffer, exchange) -> messages
    flying = []
    while any(pc[c] < len(progs[c]) for c in range(cs)):
        def can(c):
            if pc[c] == len(progs[c]):
                return False
            what, buf = progs[c][pc[c]]
            if what != "wait":
                return True
            need = len(owners) if buf == "rows" else cs
            return arrived[c].get((buf, read[c].get(buf, 0)), 0) == need
        ready = [c for c in range(cs) if c != late and can(c)]
        fast = [m for m in flying if m[1] != late and m[0] != late]
        if fast and (not ready or rng.random() < 0.5):
            m = rng.choice(fast)
        elif ready:
            m = None
            c = rng.choice(ready)
        elif can(late) and (not flying or rng.random() < 0.2):
            m = None
            c = late
        else:
            m = rng.choice(flying)           # (an empty list here would be a deadlock)
        if m is not None:
            flying.remove(m)
            _, to, buf, k = m
            assert read[to].get(buf, 0) == k, f"{buf} of CTA {to}: exchange {k} arrives before {k - 1} is read"
            arrived[to][(buf, k)] = arrived[to].get((buf, k), 0) + 1
            continue
        what, buf = progs[c][pc[c]]
        pc[c] += 1
        if what == "send":
            k = sent[c].get(buf, 0)
            sent[c][buf] = k + 1
            flying += [(c, to, buf, k) for to in (owners if buf == "modes" else range(cs))]
        elif what == "read":
            read[c][buf] = read[c].get(buf, 0) + 1


@pytest.mark.parametrize("nx,ny", SIZES)
def test_no_exchange_arrives_before_the_previous_one_is_read(nx, ny):
    for seed in range(6):
        play(nx, ny, seed)

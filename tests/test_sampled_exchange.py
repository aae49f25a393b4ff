"""Order of the peers' writes in the sampled acceptance (csrc/sampled.cu).  A CTA writes partial sums, maxima and the
children's (P, Q) into its peers' shared memory, and every exchange has one cluster barrier: behind it the peers read.
A peer that is ahead writes the next exchange's values before the next barrier, so that nothing it writes may be what
the others still read.  A race on shared memory is not a thing to provoke on a GPU: the rule is followed here over all
walks, and the kernel's text is held to the rule."""
import itertools
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2601_12212_b200", "csrc", "sampled.cu")


def walks(nodes, children):
    """Outcomes per visited node: number of rejections, and whether a child is accepted behind them."""
    one = [(r, True) for r in range(children)]
    for n in range(nodes):
        for head in itertools.product(one, repeat=n):
            for r in range(children + 1):
                yield list(head) + [(r, False)]


def exchanges(walk):
    """(kind, arrays written, rejections so far at the node) in order."""
    for rejections, _ in walk:
        yield "start", ("sum", "top", "tab"), 0
        for j in range(rejections):
            yield "reject", ("sum", "tab"), j + 1
    yield "draw", ("sum",), 0


def overlaps(place):
    """Exchange i + 1 writes before its barrier what exchange i's readers read until they arrive at that barrier."""
    for walk in walks(3, 3):
        seq = list(exchanges(walk))
        for i in range(len(seq) - 1):
            read = {place(name, i, seq[i][0], seq[i][2]) for name in seq[i][1]}
            if any(place(name, i + 1, seq[i + 1][0], seq[i + 1][2]) in read for name in seq[i + 1][1]):
                return True
    return False


def test_a_set_per_exchange_in_turn_never_overlaps():
    assert not overlaps(lambda name, i, kind, j: (name, i & 1))
    # one copy of the maxima, or a table chosen by the number of rejections, does overlap
    assert overlaps(lambda name, i, kind, j: (name, 0 if name == "top" else i & 1))
    assert overlaps(lambda name, i, kind, j: (name, j & 1 if name == "tab" else i & 1))


def test_the_kernel_keeps_the_rule():
    text = re.sub(r"//[^\n]*", "", open(SRC).read())
    kernel = text[text.index("accept_sampled_kernel"):]
    stores = re.findall(r"store_pair_to_peer\(\s*([^,]+),", kernel)
    assert len(stores) == 4
    assert all(s.startswith("sh.ex[set].") for s in stores), stores
    # the only other write to a peer is the drawn token, behind the last exchange
    assert re.findall(r"peer_address\(([^,]+),", kernel) == ["&sh.pick"]
    assert re.findall(r"\bset\b\s*(?:\^=|=)\s*[^;]+;", kernel) == ["set = 0;", "set ^= 1;"]
    assert "Exchange ex[2];" in text

"""The pre-pass is a chain of kernels whose neighbours overlap (programmatic
dependent launch), so a kernel of the chain may not read what the chain writes
through the read-only path (__ldg, and find_owner, which uses it): such a load is
undefined while another kernel writes the data.  Checked in the source, since
the fault is a race: every pointer that RunArgs and SortArgs declare as writable
is off limits to those reads in the pre-pass."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_01897_gb300", "csrc")


def _source(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


def _writable_fields():
    txt, out = _source("vista_internal.h"), set()
    for struct in ("SortArgs", "RunArgs"):
        body = re.search(r"struct %s \{(.*?)\n\};" % struct, txt, re.S).group(1)
        for decl in body.split(";"):
            if "*" in decl and "const" not in decl:
                out |= set(re.findall(r"\*\s*(\w+)", decl))
    return out


def _arguments(txt, call):
    """The argument text of every call of `call` (parentheses balanced)."""
    for m in re.finditer(r"(?<![\w])%s\(" % call, txt):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(txt[i], 0)
            i += 1
        yield txt[m.end():i - 1]


def test_chain_reads_what_it_writes_by_ordinary_loads():
    fields = _writable_fields()
    assert {"ioff", "hist", "qstart", "slot", "key", "perm", "tmp", "segcnt", "items", "ctr", "recs", "ccells"} <= fields
    txt = _source("vista_order.cu")
    reads = list(_arguments(txt, "__ldg")) + list(_arguments(txt, "find_owner"))
    assert len(reads) >= 3
    for args in reads:
        hit = fields & set(re.findall(r"\b(?:so|a)\.(?:so\.)?(\w+)", args))
        assert not hit, "read-only load of %s, which the pre-pass writes: %s" % (sorted(hit), args)


def test_read_only_search_is_the_one_with_ldg():
    txt = _source("vista_device.cuh")
    body = txt[txt.index("find_owner_chained("):]
    body = body[:body.index("\n}")]
    assert "__ldg" not in body and "__restrict__" not in body

"""Where the kernels wait: a warp whose lanes poll a barrier leaves the loop lane by lane, and the tensor-memory accesses and
products that follow are warp-wide.  Checked in the sources (no GPU): code that a whole warp runs uses the waits that leave
the warp converged; the plain one is for code that a single lane runs."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_07524_b200", "csrc")


def enclosing_headers(text, pos):
    """What stands before each brace that is open at `pos`, innermost first, and the guard of the statement itself."""
    out, depth = [], 0
    line = text[:pos].rfind("\n") + 1
    out.append(text[line:pos])
    for i in range(pos - 1, -1, -1):
        if text[i] == "}":
            depth += 1
        elif text[i] == "{":
            if depth:
                depth -= 1
            else:
                start = max(text.rfind(c, 0, i) for c in ";}\n")
                out.append(text[start + 1:i])
    return out


def single_lane(text, pos):
    headers = enclosing_headers(text, pos)
    if any(re.search(r"if \((lane|threadIdx\.x) == 0\b[^|]*\)", h) for h in headers):
        return True
    for h in headers:                                # a lambda: all of its calls
        m = re.search(r"auto (\w+) = \[", h)
        if m:
            calls = [c.start() for c in re.finditer(rf"\b{m.group(1)}\(", text)]
            return bool(calls) and all(single_lane(text, c) for c in calls)
    return False


def test_plain_waits_are_single_lane_code():
    n = 0
    for fn in sorted(os.listdir(CSRC)):
        if not fn.startswith("attn_") or not fn.endswith(".cu"):
            continue
        with open(os.path.join(CSRC, fn)) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        for m in re.finditer(r"\bmbar_wait\(", text):
            n += 1
            assert single_lane(text, m.start()), f"{fn}: line {text[:m.start()].count(chr(10)) + 1} waits lane by lane"
    assert n >= 10


def test_loads_after_a_rows_own_stores_follow_a_barrier():
    """A store that only some rows (lanes) take, inside a loop that loads tensor memory again."""
    n = 0
    for fn in ("attn_fwd.cu", "attn_bwd.cu"):
        with open(os.path.join(CSRC, fn)) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        for m in re.finditer(r"\n( *)if \((key_)?valid\) \{\n", text):
            close = text.index("\n" + m.group(1) + "}\n", m.end())
            if "uint4" not in text[m.end():close]:
                continue
            n += 1
            loop = text[text.rfind("#pragma unroll", 0, text.rfind("tmem_ld_x32", 0, m.start())):close + 200]
            before_load, after_stores = loop[:loop.index("tmem_ld_x32")], text[close:].split("\n")[2]
            assert "__syncwarp();" in before_load + after_stores, f"{fn}: line {text[:m.start()].count(chr(10)) + 2}"
    assert n == 3


def test_a_product_of_another_shape_waits_for_the_one_that_reads_what_it_overwrites():
    """The pair backward up to 96 columns: S (256 x 128) overwrites the P^T that dV (256 x 96) reads, dP the dS^T that dK reads,
    and only products of one shape are known to be ordered among themselves."""
    with open(os.path.join(CSRC, "attn_bwd_pair.cu")) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    loop = text[text.index("while (cur) {"):]
    for overwrites, reader in (("kS", "dv_done"), ("kDp", "dk_done")):
        end = loop.index(f"issue_abt(tmem + Cols::{overwrites},")
        before = loop[loop.rindex("commit(", 0, end):end]
        assert re.search(rf"kOwnDq\) wait\(2, .*&sh\.{reader}, k,|wait\(Cols::kOwnDq \? 2 : 1, .*&sh\.{reader}, k,", before), overwrites


def test_a_vote_is_followed_by_a_barrier():
    """Waits whose lanes poll different barriers: a vote does not order memory, so what one lane acquired is the others' (the one
    that issues the product among them) only behind a warp barrier."""
    with open(os.path.join(CSRC, "sm100_ptx.cuh")) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    for name in ("mbar_wait_warp", "mbar_wait_all", "mbar_wait_cluster"):
        start = text.index(f"bool {name}(")
        body = text[start:text.index("\n}\n", start)]
        assert re.search(r"__syncwarp\(\);\s*return got;\s*$", body), name
        assert body.count("return") == 1, name

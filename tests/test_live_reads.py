"""The non-coherent load (__ldg) is defined for data that nothing writes while the kernel
runs.  The steps of the short rounds run in one launch and read what the steps before
wrote, so parse.cu reads through ld_in, whose form the launch chooses."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2411_12439_gb300", "csrc")


def _functions(text):
    """(head, body) of the functions of a file, by its column-0 braces."""
    return re.findall(r"\n((?:template|__device__|__global__|static|constexpr)[^;{}]*)\{\n(.*?)\n\}", text, flags=re.S)


def test_parse_reads_its_own_writes_with_plain_loads():
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "parse.cu")).read())
    # the caller's bytes (parse_queued, byte rounds) and the first round's string offsets
    # (body_tile_strings) are the launch's input
    allowed = {"ld_in": 1, "parse_queued": 3, "body_tile_strings": 1}
    found = {}
    for head, body in _functions(text):
        n = body.count("__ldg(")
        if n:
            found[re.search(r"(\w+)\([^()]*(?:\([^()]*\)[^()]*)*\)\s*$", head.strip()).group(1)] = n
    assert found == allowed
    assert text.count("__ldg(") == sum(allowed.values())


def test_short_rounds_choose_the_plain_loads():
    text = open(os.path.join(CSRC, "parse.cu")).read()
    for kernel in ("k_parse_small", "k_naming_small"):
        body = text[text.index(f") {kernel}("):]
        body = body[:body.index("\n}\n")]
        calls = re.findall(r"(body_breaks|body_parse|rules_range)<([^>]*)>", body)
        assert calls and all(args.split(",")[-1].strip() == "true" for _, args in calls), calls

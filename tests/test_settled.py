"""When a product may read its weights before the kernel in front of it has finished (csrc/settled.h): the rule by itself, on the CPU."""
import os
import subprocess

import pytest

from paper_2311_14272_b200 import build as build_mod

# Each case: what happens in turn, and whether the product at its end may read early.  `at` is the moment a product takes before it is launched.
CASES = {
    "first": ("", False),
    "second": ("product(a);", True),
    "other_stream": ("product(a);", "b", False),
    "encoded_since": ("product(a); encode();", False),
    "after_the_one_behind_an_encode": ("product(a); encode(); product(a);", True),
    "encode_that_is_still_being_launched": ("product(a); count.begin();", False),
    "product_during_an_encode": ("product(a); count.begin(); product(a); count.end();", False),
    "two_encodes_at_once": ("product(a); count.begin(); count.begin(); count.end(); product(a);", False),
    "encode_while_a_product_is_launched": ("uint64_t at = count.now(); encode(); handle.note(a, at, true);", False),
    "captured_product": ("handle.note(a, count.now(), false);", False),
    "captured_product_on_a_settled_stream": ("product(a); if (!handle.holds(a, count.now())) handle.note(a, count.now(), false);", True),
    # An encode in a graph: replays are not counted, so nothing is early while there is such a graph, on this handle or another one over its buffers.
    "captured_encode": ("count.graph_made(); encode(); product(a);", False),
    "captured_encode_after_the_product": ("product(a); count.graph_made(); encode(); product(a); product(a);", False),
    "captured_encode_long_ago": ("count.graph_made(); encode(); encode(); product(a); encode(); product(a);", False),
    "product_before_the_graph_was_gone": ("product(a); count.graph_made(); encode(); product(a); count.graph_gone();", False),
    "product_after_the_graph_was_gone": ("count.graph_made(); encode(); product(a); count.graph_gone(); product(a);", True),
    "one_of_two_graphs_gone": ("count.graph_made(); encode(); count.graph_made(); encode(); count.graph_gone(); product(a);", False),
}


# (whether it decided to read early, what happens while it is launched, error and number of launches)
LAUNCHES = {
    "alone": (1, "", "0 1"),
    "encoded_meanwhile": (1, "count.begin(); count.end();", "0 2"),
    "being_encoded": (1, "count.begin();", "0 2"),
    "captured_meanwhile": (1, "count.graph_made();", "0 2"),
    "encoded_meanwhile_but_not_early": (0, "count.begin(); count.end();", "0 1"),
    "failed": (1, "count.begin(); return 3;", "3 1"),
}


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("settled")
    bodies = "".join(
        'if (!strcmp(name, "%s")) { EncodeCount count; Settled handle; int s[2]; const void *a = s, *b = s + 1; (void)b;\n'
        '  auto encode = [&] { count.begin(); count.end(); }; auto product = [&](const void *st) { handle.note(st, count.now(), true); };\n'
        '  (void)encode; (void)product; %s\n  puts(handle.holds(%s, count.now()) ? "early" : "waits"); return 0; }\n'
        % (name, case[0], case[1] if len(case) == 3 else "a") for name, case in CASES.items())
    # launches of a product that decided at a moment whether it reads early: what happens during the first one, and how often it is launched
    for name, (early, during, launches) in LAUNCHES.items():
        bodies += ('if (!strcmp(name, "%s")) { EncodeCount count; struct { int early; } p = {%d}; int n = 0; const uint64_t at = count.now();\n'
                   '  int e = launch_product(count, p, at, [&] { if (!n++) { %s } else if (p.early) return 7; return 0; });\n'
                   '  printf("%%d %%d\\n", e, n); return 0; }\n' % (name, early, during))
    src = d / "settled.cpp"
    src.write_text('#include <cstdio>\n#include <cstring>\n#include "settled.h"\nusing namespace crisp;\n'
                   "int main(int, char **argv) {\nconst char *name = argv[1];\n" + bodies + "return 1; }\n")
    subprocess.check_call([os.environ.get("CXX", "g++"), "-std=c++17", "-I", build_mod.CSRC, "-o", str(d / "settled"), str(src)])
    return str(d / "settled")


@pytest.mark.parametrize("name", sorted(CASES))
def test_rule(program, name):
    out = subprocess.run([program, name], capture_output=True, text=True, check=True).stdout.strip()
    assert out == ("early" if CASES[name][-1] else "waits")


@pytest.mark.parametrize("name", sorted(LAUNCHES))
def test_an_encode_that_comes_between(program, name):
    """The decision and the launch are not one step: behind an encode of another thread the product is made once more, and not early."""
    assert subprocess.run([program, name], capture_output=True, text=True, check=True).stdout.strip() == LAUNCHES[name][-1]

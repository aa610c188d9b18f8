"""The stored DRAM traffic counts as long as the kernel's code is the captured
one: every header that the kernel includes belongs to the hash."""
import os
import re

import bench

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_every_included_header_is_hashed():
    seen, todo = set(), ["paper_1410_1629_gb300/csrc/rt_forward.cu"]
    while todo:
        name = todo.pop()
        if name in seen:
            continue
        seen.add(name)
        text = open(os.path.join(ROOT, name), encoding="utf-8").read()
        for inc in re.findall(r'^\s*#\s*include\s+"([^"]+)"', text, re.M):
            near = os.path.normpath(os.path.join(os.path.dirname(name), inc))
            todo.append(near if os.path.exists(os.path.join(ROOT, near)) else os.path.join("include", os.path.basename(inc)))
    assert len(seen) >= 5 and seen <= set(bench.KERNEL_SOURCES)


def test_a_change_of_any_of_them_changes_the_hash():
    def read(changed, extra):
        def f(name):
            text = open(os.path.join(ROOT, name), encoding="utf-8").read()
            return text + extra if name == changed else text
        return f

    plain = bench.kernel_sources_hash()
    for name in bench.KERNEL_SOURCES:
        assert bench.kernel_sources_hash(read(name, "\nint another_line;\n")) != plain
        if not name.endswith(".py"):
            assert bench.kernel_sources_hash(read(name, "\n/* a\n comment */ // and another\n")) == plain

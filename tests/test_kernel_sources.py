"""Rules of the CUDA sources that keep a warp together, checked on the text.

A bounded wait may run out in one lane (or see the abort there) while its
neighbours' succeed.  Where a warp goes on to warp-collective instructions, its
lanes must not part over that: such a wait is taken by ``mbar_wait_warp`` /
``mbar_wait_spin_warp``, and the per-thread forms are left to single threads.
Lanes that took a branch apart meet again before the next such instruction:
inside its wrapper, or before a run of warp-level products.  And no bulk copy may
still be landing in a CTA's shared memory when the CTA leaves.
"""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_02438_gb300", "csrc")
ONE_THREAD = re.compile(r"\b(lane|threadIdx\.x) == 0\b")


def _sources():
    """name -> text without comments and string literals (newlines kept)."""
    out = {}
    for f in sorted(os.listdir(CSRC)):
        if f.endswith((".cu", ".cuh")):
            with open(os.path.join(CSRC, f)) as fh:
                text = fh.read()
            out[f] = re.sub(r'//[^\n]*|/\*.*?\*/|"(?:\\.|[^"\\])*"', lambda m: "\n" * m.group(0).count("\n"), text,
                            flags=re.S)
    return out


def _context(text, at):
    """The headers of the blocks around position `at`, outermost first, and the
    start of its own statement."""
    stack, start, depth = [], 0, 0
    for i in range(at):
        c = text[i]
        if c == "(":
            depth += 1
        elif c == ")":
            depth -= 1
        elif c == "{":
            stack.append((text[start:i], depth))
            start, depth = i + 1, 0
        elif c == "}":
            _, depth = stack.pop()
            start = i + 1
        elif c == ";" and depth == 0:
            start = i + 1
    return [h for h, _ in stack], text[start:at]


def _function(headers):
    """The name of the innermost named function among block headers."""
    for h in reversed(headers):
        m = re.search(r"__device__ __forceinline__ [\w ]+?\b(\w+)\([^{]*$", h, flags=re.S)
        if m:
            return m.group(1)
    return None


def _single_thread(sources, name, at, seen=()):
    headers, stmt = _context(sources[name], at)
    if any(ONE_THREAD.search(h) for h in headers) or ONE_THREAD.search(stmt):
        return True
    fn = _function(headers)
    if fn is None or fn in seen:
        return False
    calls = [(f, m.start()) for f, t in sources.items() for m in re.finditer(r"\b%s(<\w+>)?\(" % fn, t)
             if not re.search(r"__forceinline__ [\w ]+$", t[max(0, m.start() - 80):m.start()])]
    return bool(calls) and all(_single_thread(sources, f, p, (*seen, fn)) for f, p in calls)


def test_waits_of_a_whole_warp_are_taken_together():
    sources = _sources()
    found = 0
    for name, text in sources.items():
        for m in re.finditer(r"\bmbar_wait(_spin)?\(", text):
            headers, _ = _context(text, m.start())
            if not headers[1:] or _function(headers) in ("mbar_wait_warp", "mbar_wait_spin_warp"):
                continue                                 # the definitions
            found += 1
            line = text.count("\n", 0, m.start()) + 1
            assert _single_thread(sources, name, m.start()), f"{name}:{line}: a per-thread wait outside a single thread"
    assert found > 30


def test_warp_collective_instructions_rejoin_the_warp_first():
    found = 0
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith((".cu", ".cuh")):
            continue
        with open(os.path.join(CSRC, f)) as fh:
            text = fh.read()
        for m in re.finditer(r"tcgen05\.(?:ld|st|alloc|dealloc|relinquish_alloc_permit)\.[\w.:]*sync\.aligned|\bbar\.(?:sync|red)\b",
                             text):
            found += 1
            body = text[text.rindex("__device__ __forceinline__", 0, m.start()):m.start()]
            line = text.count("\n", 0, m.start()) + 1
            assert "__syncwarp();" in body, f"{f}:{line}: {m.group(0)} does not rejoin the warp"
    assert found >= 8


def test_warp_level_products_start_from_a_joined_warp():
    found = 0
    for name, text in _sources().items():
        for m in re.finditer(r"\bmma_bf16_16816\(", text):
            before = text[:m.start()]
            if before.endswith("void "):
                continue                                 # the definition
            found += 1
            line = before.count("\n") + 1
            at = before.rfind("__syncwarp();")
            assert at >= 0 and not re.search(r"\bif \(|\?", before[at:]), f"{name}:{line}: a branch since the warp met"
    assert found >= 8


def test_every_copy_is_drained_when_a_kernel_gives_up():
    kernels = 0
    for name, text in _sources().items():
        copies = set(re.findall(r"mbar_expect_tx\(&sh\.(\w+)", text))
        drained = set(re.findall(r"mbar_wait(?:_spin)?\(&sh\.(\w+)[^;]*&dummy", text))
        kernels += bool(copies)
        assert copies <= drained, f"{name}: {sorted(copies - drained)} may still be landing"
    assert kernels >= 9

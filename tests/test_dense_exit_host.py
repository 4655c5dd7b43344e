"""The dense block kernel's way out of a wait that ran out, read in its source:
whatever the lanes of a warp see, they leave together, and nothing that writes
shared memory asynchronously outlives the CTA.  (The kernel's waits run out on
the GPU in test_gpu_errors.py.)"""
import re
from pathlib import Path

SOURCE = Path(__file__).parents[1] / "paper_2512_20927_gb300" / "csrc" / "dense.cu"


def _roles():
    """The kernel's text by role, without comments."""
    text = SOURCE.read_text()
    text = text[text.index("dense_block_kernel(const float4"):text.index("cudaError_t run_block")]
    cut = [text.index("- " + r) for r in ("consumers", "producers", "loader")] + [len(text)]
    parts = [re.sub(r"//[^\n]*", "", text[a:b]) for a, b in zip(cut, cut[1:])]
    return dict(zip(("consumers", "producers", "loader"), parts))


def _calls(text, name):
    """(start, whole call) of every call of name, its brackets matched."""
    for m in re.finditer(rf"\b{name}\(", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        yield m.start(), text[m.start():i]


def test_every_wait_is_voted_by_its_warp():
    """A wait is the argument of a vote, or sets the `ok` that is voted on before
    the lanes part: in the consumers in place of the barrier that ends a slot,
    in the producers after lane 0's branch."""
    for role, text in _roles().items():
        voted = [c for _, c in _calls(text, "__all_sync")]
        waits = list(_calls(text, "dense_wait"))
        assert waits, role
        for at, call in waits:
            if any(call in v for v in voted):
                continue
            assert re.search(r"ok = (ok && )?$", text[:at]), (role, call)
            assert "__all_sync(FULL, ok)" in text[at:], (role, call)
    consumers = _roles()["consumers"]
    wait, vote = consumers.index("dense_wait("), consumers.index("if (!__all_sync(FULL, ok)) break;")
    assert not re.search(r"\b(break|continue|return|__syncwarp)\b", consumers[wait:vote])


def test_nothing_in_flight_outlives_the_cta():
    """A work request is waited for, with the full limit, by the lane that
    issued it when its wait gave up; the loader waits for its last row copies
    on every way out, as another role may give up after it has finished."""
    roles = _roles()
    ask = roles["producers"].index("try_cancel(")
    after = roles["producers"][ask:roles["producers"].index("mail_empty", ask)]
    assert re.search(r"else\s+tma_mbar_wait\(&sh\.clc, i & 1u, kDenseSpin\);", after)
    loader = roles["loader"]
    drain = re.search(r"(\S+)\s+for \(uint32_t i = rc > kRows [^\n]*\n\s*"
                      r"tma_mbar_wait\(&sh\.r_full\[i % kRows\], \(i / kRows\) & 1u, kDenseSpin\);",
                      loader)
    assert drain and drain[1] == "}", "the loader's drain depends on a condition"
    assert drain.start() > loader.rindex("bulk_row(")

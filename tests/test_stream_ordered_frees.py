"""Phase 1's arrays are freed in the order of the stream that writes them: the
device pool is shared by every context, so a free on the null stream, which a
non-blocking stream does not wait for, would give arrays that a kernel is still
writing to another request.  Read off the sources (the race itself is not run):
only the public cat_factor_free, whose callers have waited, names no stream."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2601_11621_gb300", "csrc")


def calls(name):
    for f in sorted(os.listdir(CSRC)):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
        for m in re.finditer(r"\b" + name + r"\(([^;{]*)\)\s*;", text):
            yield f, m.group(1)


def test_frees_name_their_stream():
    frees = [(f, args) for name in ("factor_free", "dev_free") for f, args in calls(name)
             if "Ctx &" not in args and "cat_ctx *" not in args]
    assert len(frees) >= 10
    unordered = [(f, args) for f, args in frees
                 if not re.search(r"(^|[\s,.>])(s|stream)$", args.strip())]
    assert unordered == [("capi.cu", "ctx->c, f, nullptr")]

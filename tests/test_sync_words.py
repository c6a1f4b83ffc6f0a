"""Layout of the persistent kernel's synchronisation words (mxp_internal.h): every
tile's epoch word lies in a 128-byte line of its own, apart from the barrier and error
words, and the buffer holds the last tile's word."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_03617_gb300", "csrc")


def test_epoch_words_do_not_share_lines():
    with open(os.path.join(CSRC, "mxp_internal.h")) as fh:
        head = fh.read()
    with open(os.path.join(CSRC, "persist2d.cu")) as fh:
        kern = fh.read()
    env = {}
    for name in ("kPersistMaxTiles", "kPersistFlagStride", "kPersistBarWords"):
        expr = re.search(rf"constexpr \w+ {name} = (.*?);", head).group(1).replace("(size_t)", "")
        env[name] = eval(expr, {}, env)                      # arithmetic of the constants above
    bases = {eval(m, {}, env) for m in re.findall(r"bar \+ (\w+)(?: \+ \(by|,|;)", kern) if m not in ("1", "2")}
    assert len(bases) == 1, bases                            # posts, polls and the reset agree
    base = bases.pop()
    word = [4 * (base + t * env["kPersistFlagStride"]) for t in range(env["kPersistMaxTiles"])]
    lines = [w // 128 for w in word]
    assert len(set(lines)) == len(lines) and 0 not in lines  # line 0: barrier and error words
    assert word[-1] + 4 <= 4 * env["kPersistBarWords"]

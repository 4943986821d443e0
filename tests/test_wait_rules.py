"""Static check of the CUDA sources (CPU): every way to wait on an mbarrier, whatever it is called, is the one bounded
helper with a status pointer."""
import re

from test_source_rules import call_args, sources, top_level_commas


def test_one_bounded_wait():
    src = sources()
    names = {n for text in src.values() for n in re.findall(r"\bmbar\w*wait\w*", text)}
    assert names == {"mbar_wait", "mbar_try_wait"}
    helper = src["tc_ptx.cuh"]
    start = helper.index("bool mbar_wait(")
    body = helper[start:helper.index("\n}\n", start)]
    # inline waits only inside mbar_try_wait, its calls only inside mbar_wait, which gives up
    inline = 0
    for name, text in src.items():
        for m in re.finditer(r"mbarrier\.(try_wait|test_wait)", text):
            owner = text.rfind("__device__", 0, m.start())
            assert text[owner:].startswith("__device__ __forceinline__ bool mbar_try_wait("), name
            inline += 1
    definitions = len(re.findall(r"bool mbar_try_wait\(", helper))
    assert inline == definitions
    calls = sum(len(re.findall(r"\bmbar_try_wait\(", t)) for t in src.values()) - definitions
    assert calls == len(re.findall(r"\bmbar_try_wait\(", body)) == 2
    assert "clock64() - t0 > WAIT_LIMIT" in body and "atomicOr(status, ST_TIMEOUT)" in body
    for name, text in src.items():
        assert not re.search(r"\bmbar_wait\s*<", text), name
        for args in call_args(text, "mbar_wait"):
            assert top_level_commas(args) == 2 and args.split(",")[-1].strip().endswith("status"), (name, args)

"""The binding's default schedule settings are the library's: set_tuning with one of them named leaves the
others where a new context has them."""
import inspect
import os
import re

from paper_2309_00651_gb300 import hfx

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_defaults_agree():
    with open(os.path.join(ROOT, "include", "hfx.h")) as f:
        header = int(re.search(r"batch of packed transforms \(default (\d+) GiB\)", f.read()).group(1)) << 30
    with open(os.path.join(ROOT, "paper_2309_00651_gb300", "csrc", "hfx_api.cu")) as f:
        text = f.read()
    lib = int(re.search(r"size_t transform_budget = size_t\((\d+)\) << 30;", text).group(1)) << 30
    block = int(re.search(r"int bsize = (\d+);", text).group(1))
    assert "bool pipeline = true;" in text
    for f in (hfx.hfx_set_tuning, hfx.Exchange.set_tuning):
        p = inspect.signature(f).parameters
        assert p["batch_bytes"].default == header == lib and p["block"].default == block and p["pipeline"].default is True

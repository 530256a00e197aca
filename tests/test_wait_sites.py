"""The site that a timed-out wait records names its kernel: no two kernels
share one. (In a kernel several waits may, e.g. those of a loop's halves.)"""
import glob
import os
import re

from conftest import ROOT

CALL = re.compile(r"\b(\w*wait\w*|mma_done|record_timeout|load)\s*\(")
SITE = re.compile(r"(?:^|,)\s*(\d{2,3})\s*$")


def _arguments(text, start):
    depth, i = 1, start
    while depth:
        depth += {"(": 1, ")": -1}.get(text[i], 0)
        i += 1
    return text[start:i - 1]


def _sites():
    """{(file, kernel): sites} of every kernel in the sources."""
    out = {}
    for path in glob.glob(os.path.join(ROOT, "paper_2607_20214_gb300", "csrc",
                                       "*.cu")):
        with open(path) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        for part in text.split("__global__")[1:]:
            kernel = re.search(r"\b(k_\w+)\s*\(", part).group(1)
            for m in CALL.finditer(part):
                site = SITE.search(_arguments(part, m.end()))
                if site:
                    key = (os.path.basename(path), kernel)
                    out.setdefault(key, set()).add(int(site.group(1)))
    return out


def test_sites_name_their_kernel():
    sites = _sites()
    kernels = {k for _, k in sites}
    assert {"k_block_attn_ws", "k_block_attn_pair", "k_race_keys_ws",
            "k_race_keys_t", "k_causal_base", "k_topk_select_tc",
            "k_bwd_block_tc", "k_bwd_keys_tc"} <= kernels
    owner = {}
    for kernel, numbers in sites.items():
        for n in numbers:
            assert owner.setdefault(n, kernel) == kernel, (
                "site %d is in %s and %s" % (n, owner[n], kernel))

"""The rule on which reads before a kernel's grid wait rest (see common.cuh): a kernel launched as one that triggers its
successor late does so directly behind its own wait, in every place.  A trigger moved, or a launcher changed, breaks no result
on most days; so the source is read."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_18183_b200", "csrc")


def _sources():
    for f in sorted(os.listdir(CSRC)):
        if f.endswith(".cu"):
            text = re.sub(r"/\*.*?\*/", "", open(os.path.join(CSRC, f)).read(), flags=re.S)
            yield f, re.sub(r"//[^\n]*", "", text)


def test_kernels_trigger_as_they_are_launched():
    early, late, launched_early, launched = set(), set(), set(), set()
    for f, text in _sources():
        for part in text.split("__global__")[1:]:
            name = re.search(r"\b(k_[a-z0-9_]+)\s*\(", part).group(1)
            body = part[part.index("{"):]
            triggers = re.findall(r"(pdl_wait\(\);\s*)?(if \((!?)a\.few\) )?pdl_trigger\(\);", body)
            assert triggers and "pdl_wait();" in body, (f, name)
            # attention does either, by one flag, which its launch passes on
            one_flag = name == "k_attention_tma" and [(bool(w), n) for w, _, n in triggers] == [(False, ""), (True, "!")]
            (late if one_flag or all(w and not cond for w, cond, _ in triggers) else early).add(name)
        launched_early |= set(re.findall(r"launch_early\(\s*(k_[a-z0-9_]+)", text))
        launched |= set(re.findall(r"launch_k\(\s*(k_[a-z0-9_]+)", text))
        launched |= set(re.findall(r"launch_kc\(\s*(?:true|!a\.few),\s*(k_[a-z0-9_]+)", text))
    assert early == launched_early == {"k_commit", "k_gemm_simt_small"}
    assert late == launched and not launched & launched_early

"""Every kernel that may start beside the launch before it waits for it."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2510_03932_gb300", "csrc")


def test_every_overlapping_kernel_waits():
    waits, ordinary = set(), set()
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        ordinary |= set(re.findall(r"\b(k_\w+)(?:<[^;<>]*>)?<<<", text))
        for k in re.finditer(r"__global__[^;{]*?\b(k_\w+)\(", text):
            body = text[k.end():text.index("\n}", k.end())]
            called = re.findall(r"\b(\w+_kernel_body)<", body)
            for c in called:
                at = re.search(r"\b%s\(" % c, text).end()
                body += text[at:text.index("\n}", at)]
            if "start_follow_on();" in body:
                waits.add(k.group(1))
            else:
                ordinary.add(k.group(1))
    assert waits == {"k_node_eval", "k_node_eval_split", "k_node_jprod", "k_node_jtprod", "k_node_hprod", "k_euler", "k_god", "k_extra",
                     "k_heat_eval", "k_heat_jh", "k_heat_hprod", "k_heat_prod_unit", "k_kkt_values", "k_obj_grad",
                     "k_obj_hvp", "k_jtprod_coo", "k_jtprod_coo_long", "k_batch_eval"}
    assert not waits & ordinary
    # an ordinary kernel is never handed to launch(), which lets it overlap
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        for call in re.findall(r"\blaunch(?:_args)?\([^;]*;", open(path).read()):
            assert not any(re.search(r"\b%s\b" % k, call) for k in ordinary), call

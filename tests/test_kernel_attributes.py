"""A kernel's shared-memory limit belongs to a device, so the sources keep no process-wide "already
raised" flag: limits go through set_smem_once, which remembers them per device under a
lock, or are raised at every launch."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1710_10769_gb300", "csrc")


def test_no_process_wide_attribute_flag():
    for name in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, name)) as f:
            text = f.read()
        if name != "tensor_map.cu":
            assert not re.search(r"\bstatic bool \w+\s*=", text), name


def test_every_slot_is_used_once():
    """A slot shared by two kernels would leave the second one's limit as it was."""
    text = "".join(open(os.path.join(CSRC, n)).read() for n in sorted(os.listdir(CSRC)) if n.endswith(".cu"))
    with open(os.path.join(CSRC, "internal.cuh")) as f:
        slots = re.findall(r"\b(kSmemSlot\w+)\b", f.read())
    names = [s for s in dict.fromkeys(slots) if s != "kSmemSlots"]
    assert len(names) >= 8
    for s in names:
        assert len(re.findall(rf"\b{s}\b", text)) == 1, s

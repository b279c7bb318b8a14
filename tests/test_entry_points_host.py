"""CPU test: an entry point of lbm.cu that queues, allocates or copies selects its handle's device first
(the caller's current device may be another one).  Checked in the source, since it takes two devices to
see it fail."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1409_5929_gb300", "csrc")
WORK = r"<<<|\bcuda(Malloc|Memcpy|Memset|Free|Stream|Event)\w*\(|\b(batch_rebuild|batch_reshape|batch_launch_\w+|launch_\w+)\("


def test_entry_points_select_their_device():
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "lbm.cu")).read())
    seen, bad = 0, []
    for m in re.finditer(r"^int (lbm_\w+)\((lbm_handle|lbm_batch)\* (\w+)[^{;]*\) \{\n(.*?)^\}", src, flags=re.M | re.S):
        name, arg, body = m.group(1), m.group(3), m.group(4)
        work = re.search(WORK, body)
        if not work:
            continue
        seen += 1
        device = body.find(f"cudaSetDevice({arg}->device)")
        if device < 0 or device > work.start():
            bad.append(name)
    assert seen > 25 and not bad, (seen, bad)

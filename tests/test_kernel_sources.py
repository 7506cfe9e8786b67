"""Orders inside the kernels that a run cannot show safely, read from the sources: no GPU."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_00422_b200", "csrc")


def kernels():
    """(file, kernel, body without comments)"""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)
        for part in re.split(r"\b__global__\b", text)[1:]:
            name = re.search(r"(\w+)\s*\(const|(\w+)\s*\(", part.split(")", 1)[-1] if part.lstrip().startswith("void __launch_bounds__") else part)
            yield os.path.basename(path), name.group(0).strip("( "), part.split("\n}\n")[0]


def test_dependents_start_behind_the_allocation_of_tensor_memory():
    """A dependent block that fits beside a block still waiting in tcgen05.alloc could take the columns that this one waits for and keep
    them until this grid has ended.  So between the allocation (one warp's) and the trigger stands a barrier of the block."""
    seen = 0
    for path, name, body in kernels():
        alloc = re.search(r"\btmem_alloc(_pair)?\(", body)
        triggers = [m.start() for m in re.finditer(r"\bgriddep_launch_dependents\(", body)]
        if not alloc or not triggers:
            continue
        seen += 1
        assert all("__syncthreads();" in body[alloc.end():t] for t in triggers), f"{path}: {name}"
        # ... that every path to the trigger has passed: it is no statement of a branch
        sync = body.index("__syncthreads();", alloc.end())
        line = body[body.rfind("\n", 0, sync) + 1:sync]
        assert line.strip() == "" and len(line) == 4, f"{path}: {name}: a barrier under a condition"
    assert seen >= 7, seen


def test_an_edit_of_any_included_file_recompiles():
    """Objects of two states of a header in one library would disagree on sizes and layouts."""
    from paper_2605_00422_b200 import build
    known = {os.path.basename(h) for h in build._headers()}
    for path in glob.glob(os.path.join(CSRC, "*.cu*")) + glob.glob(os.path.join(CSRC, "*.h")):
        included = set(re.findall(r'#include "([^"]+)"', open(path).read()))
        assert included <= known, f"{os.path.basename(path)}: {included - known}"

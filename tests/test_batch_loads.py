"""The persistent batch kernel writes the particle arrays and reads them after grid barriers of the
same launch, where the read-only load path is undefined: every item it runs takes plain loads.
Read from the sources, as a stale line would show only now and then on a GPU."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_15908_gb300", "csrc")


def _definitions(name):
    """The functions and structs at file scope, by name, comments taken out."""
    with open(os.path.join(CSRC, name)) as f:
        lines = re.sub(r"//[^\n]*", "", f.read()).split("\n")
    out, chunk = {}, []
    for line in lines:
        if not chunk and not re.match(r"(template|struct|__device__|__global__|__host__)", line):
            continue
        chunk.append(line)
        if line.startswith("}") or (line.endswith("}") and line[0] not in " \t"):
            text = "\n".join(chunk)
            head = re.sub(r"__launch_bounds__\([^)]*\)|template <[^\n]*>\n", "", text.split("{")[0])
            m = re.search(r"struct\s+(?:__align__\(\d+\)\s*)?(\w+)|(\w+)\s*\(", head)
            out.setdefault(m.group(1) or m.group(2), []).append(text)
            chunk = []
        elif line.endswith(";") and line[0] not in " \t":    # a declaration
            chunk = []
    return out


def test_items_of_the_persistent_kernel_take_coherent_loads():
    defs = _definitions("sph_device.cuh")
    kernel = _definitions("sph_batch.cu")["k_batch"][0]
    assert "ReadOnly" not in kernel
    assert re.findall(r"__ldg\([^)]*\)", kernel) == ["__ldg(src + w)"]      # the scenes' constants, never written
    calls = re.findall(r"\b(\w+_item)(<[^;(]*>)?\(", kernel)
    assert {n for n, _ in calls} >= {"hash_item", "scan_lookback_item", "scatter_item", "rank_gather_item", "search_item",
                                     "boundary_volume_item", "density_item", "force_item", "wrench_item"}
    for name, args in calls:
        if any("class LD" in text for text in defs[name]):
            assert args.rstrip(">").split(",")[-1].strip(" <") == "Coherent", name
        # what the item runs, without the code of the cooperating lanes (templates on their
        # number), which only single-scene kernels take
        seen, todo = set(), [name]
        while todo:
            used = todo.pop()
            if used in seen or used == "ReadOnly":
                continue
            seen.add(used)
            for text in defs[used]:
                if re.match(r"template <[^\n]*int G", text):
                    continue
                assert "__ldg(" not in text, f"{name} -> {used} loads through the read-only path"
                todo += [d for d in defs if re.search(r"\b%s\b" % d, text)]

"""What ptxas says of the attention kernels (a CPU compile, no GPU): nothing
spills, and the 128-token kernels are launched with the registers that their
warpgroups share out by setmaxnreg (with fewer, the raise would wait forever)."""
import os
import re
import subprocess

from paper_2608_05780_gb300.build import ARCH, CSRC, FLAGS, nvcc


def test_attention_registers(tmp_path):
    src = os.path.join(CSRC, "probe_attn.cu")
    log = subprocess.run([nvcc(), *ARCH, *FLAGS, "-Xptxas", "-v", "-c", src, "-o", str(tmp_path / "o.o")],
                         capture_output=True, text=True, check=True).stderr
    text = open(src).read()
    low, high = (int(re.search(rf"setmaxnreg_{way}<(\d+)>", text).group(1)) for way in ("dec", "inc"))
    kernels = re.findall(r"Function properties for (\S*probe_attn_kernel\S*)\n\s*(\d+) bytes stack frame, "
                         r"(\d+) bytes spill stores, (\d+) bytes spill loads\n.*?Used (\d+) registers", log)
    assert len(kernels) == 30
    for name, _, stores, loads, regs in kernels:
        assert int(stores) == int(loads) == 0, (name, stores, loads)
        if "ILi128E" in name.split("probe_attn_kernel")[1][:8]:
            assert 384 * int(regs) == 256 * high + 128 * low, (name, regs)

"""Rules that the kernel sources keep: replicas on several GPUs load this library, so no bulk
copy in it is multicast to the CTAs of a cluster."""
import pathlib
import re

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2410_13839_gb300" / "csrc"


def multicast_copies(text):
    """Bulk-copy instructions with a multicast modifier; adjacent string literals are one instruction."""
    joined = re.sub(r'"\s*"', "", text)
    return re.findall(r"cp\.async\.bulk[\w.:]*\.multicast::cluster", joined)


def test_no_bulk_copy_is_multicast():
    assert multicast_copies('asm("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"\n'
                            '    ".multicast::cluster [%0]"') != []  # the check sees one, split or not
    for path in sorted(CSRC.glob("*.cu*")):
        assert multicast_copies(path.read_text()) == [], path.name

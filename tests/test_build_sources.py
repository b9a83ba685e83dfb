"""The library is rebuilt when any file it is compiled from is newer."""
import os

from paper_1909_01092_gb300 import build


def test_every_source_file_is_watched():
    watched = set(build._sources())
    for folder in (build.CSRC, build.INCLUDE):
        files = {os.path.join(folder, f) for f in os.listdir(folder)}
        assert files and files <= watched, files - watched

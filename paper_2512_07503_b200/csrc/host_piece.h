// Whether the device can read a host array where it lies.  Free of CUDA calls: the query is the caller's.
#pragma once

#include <cstddef>
#include <cstdint>

namespace sjd {

struct HostPiece {
  char* device;  // the device's address of the asked byte
  char* start;   // and of the piece (one allocation, or one registration) it lies in
  size_t size;
};

// The device's address of `bytes` bytes from `p` on when ONE page-locked and mapped piece holds them all, else null.  (Two
// pieces with a gap between them can have both ends of an array; the gap is memory that the device must not touch.)
// piece_of(address, &piece): false where the byte is not page-locked and mapped, or nothing can be found out about it.
template <typename PieceOf>
void* device_address_of(const void* p, size_t bytes, PieceOf piece_of) {
  HostPiece piece{nullptr, nullptr, 0};
  if (!piece_of(p, &piece) || !piece.device || !piece.start) return nullptr;
  const uintptr_t at = reinterpret_cast<uintptr_t>(piece.device), from = reinterpret_cast<uintptr_t>(piece.start);
  if (at < from || at - from > piece.size || piece.size - (at - from) < bytes) return nullptr;
  return piece.device;
}

}  // namespace sjd

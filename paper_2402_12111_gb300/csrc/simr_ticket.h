// simr_ticket.h -- the block of counters and the status word that a context, and the
// scratch of simr_price_noalloc, keep on the device: all zero between launches.
#pragma once

#include "simr_internal.h"

namespace simr {

constexpr size_t kTicketBytes = 256;
constexpr size_t kTicketsAt = 0;     // words 0 .. kRowGroups: tickets of the sum over blocks (sum_block_rows)
constexpr size_t kStatusAt = 64;     // status bits that simr_sync reports
constexpr size_t kQueueAt = 128;     // the batched book's item counter
constexpr size_t kLsmTicketAt = 192;  // Longstaff-Schwartz: its ticket, and 16 bytes on its sweep's barrier counter
// a ticket past its bytes would count arrivals in the status word, and clear it
static_assert(kTicketsAt + (1 + kRowGroups) * sizeof(unsigned int) <= kStatusAt, "tickets run into the status word");
static_assert(kLsmTicketAt + 16 + sizeof(unsigned int) <= kTicketBytes, "the block is too small");

}  // namespace simr
